"""Batch-norm sums in the epilogue of the CUDA-core convolution: channel counts below, at and between tile widths, last tiles of a
few pixels, reductions shared by a cluster and not, 16-byte operands and value by value.  Tolerance: that of float32 steps (1e-3);
bfloat16 storage 3e-2."""
import numpy as np
import pytest

from oracle import numeric_oracle as no
from paper_2502_12499_b200 import binding as ck
from paper_2502_12499_b200 import workloads as wl
from tests.gpu_util import StepRunner, max_rel_err

pytestmark = pytest.mark.gpu

SHAPES = [("f32", 16, 16, 4, 32, 32), ("f32", 3, 5, 2, 7, 9), ("f32", 8, 20, 3, 11, 13), ("f32", 64, 33, 1, 5, 5), ("f32", 128, 128, 2, 8, 8),
          ("f32", 12, 300, 1, 9, 3), ("f32", 256, 64, 1, 4, 4), ("f32", 32, 64, 4, 21, 17), ("bf16", 5, 12, 3, 9, 7), ("bf16", 20, 36, 2, 6, 10)]


@pytest.mark.parametrize("dtype,cin,c,batch,h,w", SHAPES)
def test_statistics_of_convolution(dtype, cin, c, batch, h, w):
    spec = dict(units=[wl.conv_unit(cin, c), {"kind": "avgpool"}, {"kind": "fc", "cin": c, "cout": 10, "relu": False}],
                input_hwc=(h, w, cin), batch=batch, dtype=dtype, loss="softmax_ce", name="sums_%s_%d" % (dtype, c))
    params = wl.make_params(spec, seed=21, bn_affine="random")
    x, labels = wl.make_batch(spec, seed=22)
    runner = StepRunner(spec, params)
    ck.launch_log(True)
    rep, grads = runner.run(ck.POLICY_STORE_ALL, None, x, labels)
    kernels = ck.launch_log_read()
    ck.launch_log(False)
    assert "batch-norm statistics" not in kernels, kernels
    ref = no.chain_forward_backward(spec, [{k: v.astype(np.float64) for k, v in p.items()} for p in params], x.astype(np.float64), labels,
                                    storage="bf16" if dtype == "bf16" else "exact")
    tol = 3e-2 if dtype == "bf16" else 1e-3
    assert abs(rep["loss"] - ref["loss"]) <= tol * abs(ref["loss"])
    for (ui, name, _), g in zip(runner.flat, grads):
        want = ref["grads"][ui][name]
        assert max_rel_err(g.reshape(want.shape), want) <= tol, (ui, name)


MAX_PARTIAL_ROWS = 148 * 8


@pytest.mark.parametrize("dtype,cin,c,batch,h,w,shared,separate", [
    ("f32", 16, 16, 4, 32, 32, False, False), ("f32", 3, 5, 2, 7, 9, False, False), ("f32", 128, 128, 2, 8, 8, True, False), ("f32", 64, 33, 1, 5, 5, True, False),
    ("f32", 64, 64, 3, 150, 150, False, False), ("f32", 3, 64, 2, 200, 200, False, True), ("bf16", 20, 36, 2, 6, 10, True, False)])
def test_statistics_against_float64(dtype, cin, c, batch, h, w, shared, separate):
    """Mean and inverse deviation that a step saves against float64 ones of the z it stores: reductions shared by a cluster or not, and
    more partial rows than the scratch region holds, which take a pass of their own.  In the root mean square over channels: an inverse
    rounded to float32 is off by 2.5e-8 of itself, a mean of up to half a deviation by 1.2e-8 of the deviation; two thirds of that again are
    left for the sums.  A tree of float32 additions of N values is off by 2^-24 * 0.58 * sqrt(levels * N) deviations, a dozen levels at most:
    1.2e-7 / sqrt(N) of the deviation in the mean, which counts where N is small.  (Measured on 4,000 values and more: 2.5e-8 and 0.7e-8;
    one float32 chain over 67,500 values would be off by 4e-8 of the deviation.)"""
    import torch
    shape = ck.ConvShape(batch, h, w, cin, c, 3, 1, 1)
    code, store = (ck.DTYPE_BF16, torch.bfloat16) if dtype == "bf16" else (ck.DTYPE_F32, torch.float32)
    plan = ck.selftest_simt_plan(shape, code, 0, 1)
    assert (plan["cluster"] > 1) == shared, plan
    assert (-(-batch * h * w // plan["rows"]) * plan["cluster"] > MAX_PARTIAL_ROWS) == separate, plan
    spec = dict(units=[wl.conv_unit(cin, c), {"kind": "avgpool"}], input_hwc=(h, w, cin), batch=batch, dtype=dtype, loss="sum", name="stats")
    params = wl.make_params(spec, seed=31, bn_affine="random")
    x, _ = wl.make_batch(spec, seed=32)
    runner = StepRunner(spec, params)
    ck.launch_log(True)
    runner.run(ck.POLICY_STORE_ALL, None, x + np.float32(0.25) if dtype == "f32" else x, None)
    kernels = ck.launch_log_read()
    ck.launch_log(False)
    assert ("batch-norm statistics" in kernels) == separate, kernels
    z = torch.empty((batch, h, w, c), dtype=store, device="cuda")
    xd = torch.from_numpy(x + np.float32(0.25) if dtype == "f32" else x).cuda().to(store)
    ck.conv2d_forward(shape, code, 0, xd, torch.from_numpy(params[0]["w"]).cuda().to(store), z)        # as the step stores it
    mean = z.double().mean((0, 1, 2))
    inv = (z.double().var((0, 1, 2), unbiased=False) + 1e-5).rsqrt()
    # the saved rows [mean | inverse deviation | ...] lie in the workspace: where all of the means and inverses come close
    words = runner.workspace[:runner.workspace.numel() // 4 * 4].view(torch.float32)
    want = torch.cat((mean, inv)).float()
    found = [i for i in torch.nonzero((words[:-2 * c] - want[0]).abs() < 1e-4 * (1 / inv[0]).float()).flatten().tolist()
             if bool(((words[i:i + 2 * c] - want).abs() <= 1e-4 * torch.cat((1 / inv, inv)).float()).all())]
    assert len(found) == 1, found
    got = words[found[0]:found[0] + 2 * c].double()
    assert ((got[:c] - mean) * inv).square().mean().sqrt() <= 2e-8 + 1.2e-7 / (batch * h * w) ** 0.5
    assert (got[c:] / inv - 1).square().mean().sqrt() <= 4e-8 + 1.2e-7 / (batch * h * w) ** 0.5
