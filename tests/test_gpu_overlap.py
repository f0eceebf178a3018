"""Kernels that start under the tail of the one before them: operations queued back to back, each on what the one before
wrote, leave the bits that they leave with the device idle between them."""
import pytest

from paper_2502_12499_b200 import binding as ck
from tests.gpu_util import torch_dtype

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n,h,w,c", [(ck.DTYPE_BF16, 3, 5, 7, 64), (ck.DTYPE_BF16, 16, 14, 14, 128), (ck.DTYPE_BF16, 2, 9, 9, 24),
                                           (ck.DTYPE_F32, 4, 16, 16, 16), (ck.DTYPE_F32, 2, 7, 5, 3)])
def test_queued_operations_see_one_another(dtype, n, h, w, c):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    td, rows = torch_dtype(dtype), n * h * w
    shape = ck.ConvShape(n, h, w, c, c, 3, 1, 1)
    x0 = torch.randn((n, h, w, c), generator=gen, device="cuda").to(td)
    wt = (torch.randn((c, 3, 3, c), generator=gen, device="cuda") * (2.0 / (9 * c)) ** 0.5).to(td)
    gamma, beta = torch.rand(c, generator=gen, device="cuda") + 0.5, 0.2 * torch.randn(c, generator=gen, device="cuda")
    scratch = torch.empty(max(ck.conv2d_scratch_bytes(shape, dtype), ck.bn_scratch_bytes(rows, c)) + 256, dtype=torch.uint8, device="cuda")

    def walk(idle):
        x, z, y, g, dz = x0.clone(), *(torch.zeros_like(x0) for _ in range(4))
        stats, dgamma, dbeta, dw = torch.zeros(4, c, device="cuda"), torch.zeros(c, device="cuda"), torch.zeros(c, device="cuda"), torch.zeros(c, 3, 3, c, device="cuda")
        torch.cuda.synchronize()
        for _ in range(4):
            # the buffers take turns: every operation reads what the last one wrote and writes what it read
            for op in (lambda: ck.conv2d_forward(shape, dtype, 0, x, wt, z, scratch),
                       lambda: ck.bn_relu_forward(dtype, rows, c, z, gamma, beta, 1, y, stats, scratch),
                       lambda: ck.conv2d_forward(shape, dtype, 0, y, wt, g, scratch),
                       lambda: ck.bn_relu_backward(dtype, rows, c, g, z, gamma, stats, 1, dz, dgamma, dbeta, scratch),
                       lambda: ck.conv2d_wgrad(shape, dtype, 0, dz, y, dw, scratch),
                       lambda: ck.conv2d_dgrad(shape, dtype, 0, dz, wt, x, scratch),
                       lambda: ck.bn_relu_forward(dtype, rows, c, x, gamma, beta, 0, x, stats, scratch)):
                op()
                if idle:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return x, z, y, g, dz, stats, dgamma, dbeta, dw

    want = walk(True)
    for _ in range(3):
        for a, b in zip(walk(False), want):
            assert torch.equal(a, b)
    ck.op_status()
