"""Weight gradients of reductions below 4096 pixels (accumulation chains of 256 pixels, few slices) against float64.  A chain is sixteen
MMAs, each of which cuts at most 2^-23 of the running sum: 16 * 2^-23 = 1.9e-6 of the norm; what float32 additions of the
chains' sums add to that is smaller by the root of their number."""
import pytest

from paper_2502_12499_b200 import binding as ck

pytestmark = pytest.mark.gpu


def weight_gradient_error(n, h, w, cin, cout, k, stride):
    """Error against float64 in the norm, and the kernels that ran."""
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    pad = k // 2
    ho, wo = (h + 2 * pad - k) // stride + 1, (w + 2 * pad - k) // stride + 1
    shape = ck.ConvShape(n, h, w, cin, cout, k, stride, pad)
    x = torch.randn((n, h, w, cin), generator=gen, device="cuda").bfloat16()
    g = torch.randn((n, ho, wo, cout), generator=gen, device="cuda").bfloat16()
    dw = torch.full((cout, k, k, cin), float("nan"), device="cuda")
    scratch = torch.empty(ck.conv2d_scratch_bytes(shape, ck.DTYPE_BF16) + 256, dtype=torch.uint8, device="cuda")
    ck.launch_log(True)
    ck.conv2d_wgrad(shape, ck.DTYPE_BF16, 0, g, x, dw, scratch)
    ck.op_status()
    kernels = ck.launch_log_read()
    ck.launch_log(False)
    weight = torch.zeros((cout, cin, k, k), dtype=torch.double, device="cuda", requires_grad=True)
    torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), weight, stride=stride, padding=pad).backward(g.double().permute(0, 3, 1, 2))
    want = weight.grad.permute(0, 2, 3, 1)
    return ((dw.double() - want).norm() / want.norm()).item(), kernels


@pytest.mark.parametrize("n,h,w,cin,cout,k,stride", [
    (1, 1, 257, 64, 64, 1, 1), (5, 9, 7, 64, 128, 1, 1), (21, 13, 11, 1024, 256, 1, 1), (9, 7, 6, 512, 512, 3, 1), (128, 4, 4, 256, 512, 3, 1),
    (17, 15, 15, 128, 320, 3, 2), (7, 24, 24, 192, 64, 1, 2), (63, 5, 13, 64, 2048, 1, 1), (65, 7, 9, 128, 192, 1, 1), (3, 9, 11, 96, 136, 3, 2)])
def test_short_reduction(n, h, w, cin, cout, k, stride):
    error, _ = weight_gradient_error(n, h, w, cin, cout, k, stride)
    assert error <= 2e-6


# bound: half-way between what these chains measure and what longer ones do (in 1e-7: whole blocks of channels, one chain per slice
# of 256 pixels and more 3.3, 3.4, 3.9, 3.8, 4.7 against 1.9, 1.5, 2.0, 2.2, 2.1; ragged ones, all chains of 64 pixels in one
# slice 0.73, 0.91, 1.01 against 0.66, 0.87, 0.95)
@pytest.mark.parametrize("n,h,w,cin,cout,k,stride,bound,sliced", [
    (21, 13, 11, 1024, 256, 1, 1, 2.6e-7, True), (9, 7, 6, 512, 512, 3, 1, 2.4e-7, False), (128, 4, 4, 256, 512, 3, 1, 2.9e-7, False),
    (32, 7, 7, 2048, 512, 1, 1, 3.0e-7, False), (63, 5, 13, 64, 2048, 1, 1, 3.3e-7, True),
    (3, 10, 10, 96, 48, 3, 1, 7.0e-8, True), (12, 13, 13, 96, 96, 3, 1, 8.9e-8, True), (39, 10, 10, 72, 136, 3, 1, 9.8e-8, True),
    (11, 12, 12, 96, 136, 3, 2, 7.2e-8, True)])
def test_chains_are_short(n, h, w, cin, cout, k, stride, bound, sliced):
    error, kernels = weight_gradient_error(n, h, w, cin, cout, k, stride)
    assert "tc_conv_wgrad_kernel" in kernels and ("slice_sum_kernel" in kernels) == sliced, kernels
    assert error <= bound
