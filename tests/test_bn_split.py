"""How the batch-norm backward divides a tensor, for devices that hold more and fewer of its CTAs at once (host only)."""
import itertools

import pytest

from paper_2502_12499_b200 import binding as ck

SEPARATE, CLUSTERS, COOPERATIVE = 0, 1, 2
B200 = (7, 15, 33, 148)


@pytest.mark.parametrize("held", [B200, (0, 15, 33, 148), (0, 0, 33, 148), (0, 0, 0, 148), (1, 2, 4, 18), (0, 0, 0, 18), (0, 0, 0, 0)])
def test_no_more_ctas_than_the_device_holds(held):
    """Every cluster, or every CTA of the co-operative grid, has its place; a tensor for which there is none goes to the
    separate kernels."""
    sizes = dict(zip((16, 8, 4), held))
    seen = set()
    for dtype, rows, c, masked in itertools.product((ck.DTYPE_F32, ck.DTYPE_BF16), (1, 60, 777, 3003, 8192, 50176, 400000),
                                                    (3, 8, 24, 64, 72, 256, 1000, 2048, 8192), (0, 1)):
        form, groups, parts = ck.selftest_bn_split(dtype, rows, c, masked, held)
        seen.add(form)
        if form == CLUSTERS:
            size = min(s for s in (4, 8, 16) if parts <= s and sizes[s] >= groups)
            assert 1 <= parts <= size
        elif form == COOPERATIVE:
            assert 1 <= parts <= rows and groups * parts <= held[3]
        if c % 4:
            assert form == SEPARATE
    assert seen == ({SEPARATE} if held[3] == 0 else {SEPARATE, COOPERATIVE} if not any(held[:3]) else {SEPARATE, CLUSTERS, COOPERATIVE})


def test_forms_on_b200():
    split = lambda rows, c, held=B200: ck.selftest_bn_split(ck.DTYPE_BF16, rows, c, 0, held)
    assert split(3003, 256) == (CLUSTERS, 4, 16) and split(882, 2048) == (CLUSTERS, 16, 4)
    assert split(25088, 256) == (COOPERATIVE, 4, 37)
    assert split(3003, 256, (0, 15, 33, 148))[0] == CLUSTERS                # eight CTAs hold it too
    assert split(3003, 256, (3, 3, 3, 148)) == (COOPERATIVE, 4, 37)         # clusters for three groups of four
    assert split(3003, 256, (0, 0, 0, 3)) == (SEPARATE, 4, 0)
