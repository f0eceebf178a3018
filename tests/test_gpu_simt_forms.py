"""Forms of the CUDA-core convolution against float64: filters of more than 16 rows in 16-byte chunks - stride, padding on all sides and none,
operands that cannot be fetched in chunks beside ones that can, reductions shared by a cluster - and reductions of one chain at most,
value by value.  Sums in chains of 64 products are within 1e-6 of their norm; storing bfloat16 adds half a unit in the last
place, 2^-9."""
import pytest

from paper_2502_12499_b200 import binding as ck
from tests.gpu_util import torch_dtype

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [ck.DTYPE_F32, ck.DTYPE_BF16])
@pytest.mark.parametrize("n,h,w,cin,cout,k,stride,pad", [(2, 23, 19, 16, 24, 17, 1, 8), (1, 40, 33, 8, 8, 21, 1, 0), (3, 30, 37, 16, 32, 17, 2, 8), (2, 19, 20, 6, 64, 18, 1, 9),
                                                         (1, 9, 70, 64, 16, 31, 3, 15), (2, 24, 24, 16, 16, 16, 1, 8)])
def test_wide_filter(n, h, w, cin, cout, k, stride, pad, dtype):
    against_float64(n, h, w, cin, cout, k, stride, pad, dtype)


@pytest.mark.parametrize("dtype", [ck.DTYPE_F32, ck.DTYPE_BF16])
@pytest.mark.parametrize("n,h,w,cin,cout,k,stride,pad,one", [(3, 17, 19, 7, 33, 3, 1, 1, True), (2, 9, 11, 63, 20, 1, 1, 0, True), (2, 9, 11, 65, 20, 1, 1, 0, True), (24, 40, 40, 70, 20, 1, 1, 0, False),
                                                             (1, 7, 7, 1, 18, 8, 1, 3, True), (4, 13, 9, 3, 70, 1, 2, 0, True), (1, 3, 2, 3, 5, 3, 1, 1, True)])
def test_one_chain(n, h, w, cin, cout, k, stride, pad, one, dtype):
    plan = ck.selftest_simt_plan(ck.ConvShape(n, h, w, cin, cout, k, stride, pad), dtype, 0, 1)
    assert plan["fetch"] == 0 and (plan["length"] <= 64) == one, plan
    against_float64(n, h, w, cin, cout, k, stride, pad, dtype, impl=1)


def against_float64(n, h, w, cin, cout, k, stride, pad, dtype, impl=0):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    td, ho, wo = torch_dtype(dtype), (h + 2 * pad - k) // stride + 1, (w + 2 * pad - k) // stride + 1
    shape = ck.ConvShape(n, h, w, cin, cout, k, stride, pad)
    x, g = (torch.randn(s, generator=gen, device="cuda").to(td) for s in ((n, h, w, cin), (n, ho, wo, cout)))
    wt = (torch.randn((cout, k, k, cin), generator=gen, device="cuda") * (2.0 / (k * k * cin)) ** 0.5).to(td)
    z, dx, dw = torch.full_like(g, float("nan")), torch.full_like(x, float("nan")), torch.full((cout, k, k, cin), float("nan"), device="cuda")
    scratch = torch.empty(ck.conv2d_scratch_bytes(shape, dtype) + 256, dtype=torch.uint8, device="cuda")
    ck.conv2d_forward(shape, dtype, impl, x, wt, z, scratch)
    ck.conv2d_dgrad(shape, dtype, impl, g, wt, dx, scratch)
    ck.conv2d_wgrad(shape, dtype, impl, g, x, dw, scratch)
    x64, w64 = x.double().permute(0, 3, 1, 2).requires_grad_(), wt.double().permute(0, 3, 1, 2).requires_grad_()
    z64 = torch.nn.functional.conv2d(x64, w64, stride=stride, padding=pad)
    z64.backward(g.double().permute(0, 3, 1, 2))
    stored = 1e-6 if dtype == ck.DTYPE_F32 else 2.0 ** -9
    for got, want, tol in ((z, z64.detach(), stored), (dx, x64.grad, stored), (dw, w64.grad, 1e-6)):
        want = want.permute(0, 2, 3, 1)
        assert ((got.double() - want).norm() / want.norm()).item() <= tol
