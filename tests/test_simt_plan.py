"""Plans of the CUDA-core convolution (host only)."""
import itertools

import pytest

from paper_2502_12499_b200 import binding as ck

SHAPES = [ck.ConvShape(n, h, w, cin, cout, k, s, k // 2) for (n, h, w), (cin, cout), k, s in itertools.product(
    ((1, 5, 5), (4, 32, 32), (9, 37, 11), (32, 16, 16), (16, 112, 112)), ((3, 64), (16, 16), (64, 64), (96, 300), (512, 512)), (1, 3, 7), (1, 2))]


@pytest.mark.parametrize("dtype,mode,aligned", list(itertools.product((ck.DTYPE_F32, ck.DTYPE_BF16), (0, 1, 2), (0, 1))))
def test_plan_covers_the_reduction(dtype, mode, aligned):
    for s in SHAPES:
        p = ck.selftest_simt_plan(s, dtype, mode, aligned)
        ho, wo = (s.h + 2 * s.pad - s.k) // s.stride + 1, (s.w + 2 * s.pad - s.k) // s.stride + 1
        reduction = (s.k ** 2 * s.c_in, (-(-s.k // s.stride)) ** 2 * s.c_out, s.n * ho * wo)[mode]
        parts = p["cluster"] * p["slices"]
        assert p["cluster"] in (1, 2, 4, 8) and (mode == 2 or p["slices"] == 1), p
        assert p["length"] % 32 == 0 or parts == 1, p
        assert parts * p["length"] >= reduction, (p, reduction)
        assert (p["slices"] - 1) * p["cluster"] * p["length"] < reduction, (p, reduction)
        if mode == 2 and p["slices"] > 1:
            assert p["slices"] * s.c_out * s.k ** 2 * s.c_in * 4 <= ck.conv2d_scratch_bytes(s, dtype)
        assert p["fetch"] == 3 or min(p["rows"], p["columns"]) <= 64


@pytest.mark.parametrize("k,cin,cout,forward,dgrad,wgrad", [(16, 64, 64, 3, 3, 3), (17, 64, 64, 7, 7, 3), (31, 16, 24, 7, 7, 3), (21, 64, 6, 7, 2, 2), (21, 6, 64, 0, 5, 1)])
def test_wide_filters_are_fetched_in_chunks(k, cin, cout, forward, dgrad, wgrad):
    for dtype in (ck.DTYPE_F32, ck.DTYPE_BF16):
        shape = ck.ConvShape(3, 40, 33, cin, cout, k, 1, k // 2)
        assert [ck.selftest_simt_plan(shape, dtype, m, 1)["fetch"] for m in (0, 1, 2)] == [forward, dgrad, wgrad]
        assert [ck.selftest_simt_plan(shape, dtype, m, 0)["fetch"] for m in (0, 1, 2)] == [0, 0, 0]
        if k > 16:
            assert all(ck.selftest_simt_plan(shape, dtype, m, 1)["rows"] == 64 for m in (0, 1) if (forward, dgrad)[m] & 4)


def test_plan_counts_on_what_the_kernels_are_compiled_for():
    """A 64 x 64 tile of float32 takes 128 registers a thread and is held four times, of bfloat16 168 and three times; of 128 x 16 tiles
    five would outgrow shared memory where the reduction is contiguous."""
    held = {}
    for s, dtype, mode in itertools.product(SHAPES, (ck.DTYPE_F32, ck.DTYPE_BF16), (0, 1, 2)):
        p = ck.selftest_simt_plan(s, dtype, mode, 1)
        held.setdefault((dtype, mode, p["rows"], p["columns"]), set()).add(p["held"])
    assert all(len(v) == 1 for v in held.values()), held
    for mode in (0, 1, 2):
        assert held.get((ck.DTYPE_F32, mode, 64, 64), {4}) == {4} and held.get((ck.DTYPE_BF16, mode, 64, 64), {3}) == {3}, held
        assert held.get((ck.DTYPE_F32, mode, 128, 16), {4}) == {4}
    assert (ck.DTYPE_F32, 0, 64, 64) in held and (ck.DTYPE_BF16, 0, 64, 64) in held, held
