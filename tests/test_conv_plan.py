"""Tiles of the role-swapped convolution kernel against the shared memory they need (host only)."""
import itertools

import pytest

from paper_2502_12499_b200 import binding as ck

SMEM_PER_BLOCK = 227 * 1024


def plans(epilogue):
    for c_red, c_out, k, hw, n in itertools.product((64, 192, 512, 1024, 1416, 1536, 2048, 4096, 8192), (64, 136, 512, 2048, 8192), (1, 3),
                                                    ((7, 7), (14, 14), (13, 11), (56, 56)), (1, 3, 6, 8, 13, 64)):
        if k == 3 and epilogue == 1:
            continue                                   # only 1x1 filters join
        try:
            yield (c_red, c_out, k, hw, n), ck.selftest_conv_plan(ck.ConvShape(n, hw[0], hw[1], c_red, c_out, k, 1, k // 2), epilogue)
        except ck.CkptError as e:
            assert e.code == -11, e                    # another kernel's shape


@pytest.mark.parametrize("epilogue", [0, 1, 2])
def test_tiles_fit_shared_memory(epilogue):
    """Every tile leaves at least two operand stages beside the epilogue's slabs, and the accumulators that the CTAs of a
    shared reduction exchange lie within the stages, whatever the epilogue."""
    wide = 0
    for shape, p in plans(epilogue):
        assert p["pixels"] % 32 == 0 and 64 <= p["pixels"] <= 256, (shape, p)
        assert p["smem"] <= SMEM_PER_BLOCK and 2 <= p["stages"] <= 8, (shape, p)
        assert p["exchange_bytes"] == (p["pixels"] * 128 * 4 if p["split"] > 1 else 0), (shape, p)
        assert p["exchange_bytes"] <= p["stage_bytes"], (shape, p)
        wide += p["split"] > 1 and p["pixels"] >= 160
    assert wide > 0                                    # the grid holds tiles whose accumulators outgrow two stages
