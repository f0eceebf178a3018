"""Kernels that start under the tail of the one before them: operations queued back to back, each on what the one before
wrote, leave the bits that they leave with the device idle between them."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2502_12499_b200 import binding as ck
from paper_2502_12499_b200 import workloads as wl
from tests.conftest import ROOT
from tests.gpu_util import to_dev, torch_dtype

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


# a layer 3 -> cin in front of weight gradients of every form (the names are those of the launch log)
WGRADS = [(3, 16, 16, 64, 64, 3, 1, "tc_wgrad_c64_kernel"), (1, 16, 15, 64, 128, 3, 1, "tc_wgrad_c64_kernel"), (2, 16, 32, 64, 64, 3, 1, "tc_wgrad_rows_kernel (pixel pairs)"),
          (2, 14, 14, 128, 128, 3, 1, "tc_wgrad_rows_kernel"), (2, 20, 18, 48, 48, 3, 1, "tc_wgrad_rows_kernel"), (9, 7, 7, 256, 256, 3, 1, "tc_conv_wgrad_kernel"),
          (11, 12, 12, 96, 136, 3, 2, "tc_conv_wgrad_kernel"), (2, 12, 12, 64, 320, 1, 1, "tc_conv_wgrad_kernel")]


@pytest.mark.parametrize("n,h,w,cin,cout,k,stride,kernel", WGRADS)
def test_kernels_with_tensor_memory_follow_one_another(n, h, w, cin, cout, k, stride, kernel):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(6)
    dtype = ck.DTYPE_BF16

    def rand(*dims, scale=1.0):
        return (torch.randn(dims, generator=gen, device="cuda") * scale).bfloat16()

    pad = k // 2
    ho, wo = (h + 2 * pad - k) // stride + 1, (w + 2 * pad - k) // stride + 1
    first, stem = ck.ConvShape(n, h, w, 3, cin, 3, 1, 1), ck.ConvShape(n, 2 * h, 2 * w, 3, cin, 7, 2, 3)
    layer = ck.ConvShape(n, h, w, cin, cout, k, stride, pad)
    small, large, dz = rand(n, h, w, 3), rand(n, 2 * h, 2 * w, 3), rand(n, ho, wo, cout)
    w3, w7 = rand(cin, 3, 3, 3, scale=0.2), rand(cin, 7, 7, 3, scale=0.1)
    scratch = torch.empty(max(ck.conv2d_scratch_bytes(s, dtype) for s in (first, stem, layer)) + 256, dtype=torch.uint8, device="cuda")

    def walk(idle):
        x = torch.zeros((n, h, w, cin), dtype=torch.bfloat16, device="cuda")
        dw, dw3, dw7 = torch.zeros(cout, k, k, cin, device="cuda"), torch.zeros(cin, 3, 3, 3, device="cuda"), torch.zeros(cin, 7, 7, 3, device="cuda")
        out = []
        torch.cuda.synchronize()
        for _ in range(3):
            # every layer's output is what the weight gradient behind it reads, and what the next one overwrites
            for op in (lambda: ck.conv2d_forward(first, dtype, 0, small, w3, x, scratch), lambda: ck.conv2d_wgrad(layer, dtype, 0, dz, x, dw, scratch),
                       lambda: out.append(dw.clone()),
                       lambda: ck.conv2d_forward(stem, dtype, 0, large, w7, x, scratch), lambda: ck.conv2d_wgrad(layer, dtype, 0, dz, x, dw, scratch),
                       lambda: ck.conv2d_wgrad(stem, dtype, 0, x, large, dw7, scratch), lambda: ck.conv2d_wgrad(layer, dtype, 0, dz, x, dw, scratch),
                       lambda: ck.conv2d_wgrad(first, dtype, 0, x, small, dw3, scratch)):
                op()
                if idle:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return out + [x, dw, dw3, dw7]

    ck.launch_log(True)
    want = walk(True)
    kernels = ck.launch_log_read()
    ck.launch_log(False)
    for name in (kernel, "tc_conv_first_kernel", "tc_conv_stem_kernel", "tc_wgrad_stem_kernel"):
        assert name in kernels, (name, kernels)
    for _ in range(3):
        for a, b in zip(walk(False), want):
            assert torch.equal(a, b)
    ck.op_status()


def small_chains():
    """First layer, stem, both poolings, fully connected units, residual blocks with and without a stride, units of finer granularity and
    convolutions on the CUDA cores."""
    conv = {"kind": "conv", "cin": 64, "cout": 64, "k": 3, "stride": 1, "pad": 1}
    plain = [dict(conv, cin=3), conv, conv, {"kind": "avgpool"}, {"kind": "fc", "cin": 64, "cout": 10, "relu": False}]
    return [wl.vgg16_chain(4, hw=(32, 32), dtype="bf16", widths=(64, 64, 128, 128, 128), fc_width=64, classes=10, name="vgg"),
            wl.split_units(wl.vgg16_chain(2, hw=(32, 64), dtype="bf16", widths=(48, 48, 72, 64, 64), fc_width=72, classes=10, name="vgg_fine"))[0],
            wl.resnet_chain([1, 2, 1, 1], 3, hw=(72, 64), dtype="bf16", base=64, classes=10, name="resnet"),
            wl.vgg16_chain(2, hw=(32, 32), dtype="f32", widths=(8, 16, 24, 32, 32), fc_width=24, classes=10, name="vgg_f32"),
            dict(units=plain, input_hwc=(16, 16, 3), batch=4, dtype="bf16", loss="softmax_ce", name="plain_bf16")]


def gradients_of_steps(recorded):
    """Losses and gradients of each chain's planned step with early free: {chain: [arrays]}."""
    import torch
    out = {}
    for spec in small_chains():
        chain = ck.Chain(spec)
        chain.set_graph(recorded)
        d = chain.sizes()
        mask, peak = ck.plan(ck.ALGO_DYNAMIC_N, d)
        params, grads, _ = ck.upload_params(chain, wl.make_params(spec, seed=41, bn_affine="random"))
        x, labels = wl.make_batch(spec, seed=42)
        x, labels = to_dev(x, chain.dtype), torch.from_numpy(labels).cuda()
        arena, workspace = (torch.empty(n, dtype=torch.uint8, device="cuda") for n in (peak, chain.workspace_bytes()))
        for _ in range(4 if recorded else 2):
            for g in grads:
                g.fill_(float("nan"))
            arena.fill_(0xFF)
            report = ck.train_step(chain, mask, ck.POLICY_DYNAMIC, x, labels, params, grads, arena, workspace)
        assert bool(report["replayed"]) == recorded
        out[spec["name"]] = [np.float64(report["loss"])] + [g.cpu().numpy() for g in grads]
    return out


def test_recorded_and_queued_steps_against_one_launch_at_a_time(tmp_path):
    """The same steps in a process whose launches are waited for one by one, queued here, and replayed from a recording: the same bits."""
    program = "import sys; sys.path.insert(0, %r)\nfrom tests import test_gpu_overlap as t\nimport numpy as np\n" % ROOT
    program += "np.savez(%r, **{'%%s %%d' %% (n, i): a for n, arrays in t.gradients_of_steps(False).items() for i, a in enumerate(arrays)})" % str(tmp_path / "one.npz")
    subprocess.run([sys.executable, "-c", program], check=True, timeout=300, cwd=ROOT, env=dict(os.environ, CUDA_LAUNCH_BLOCKING="1"))
    want = np.load(tmp_path / "one.npz")
    for recorded in (False, True):
        for name, arrays in gradients_of_steps(recorded).items():
            for i, a in enumerate(arrays):
                assert np.isfinite(a).all() and np.array_equal(a, want["%s %d" % (name, i)]), (name, i, recorded)
