"""2x2 pooling behind a convolution with batch norm: forward through the pending normalisation, backward through pooling and batch
norm together, where channel groups do not divide a block, fill it exactly or are a single one, and where the last block has
a window or two.  Tolerances: those of the step's gradients (1e-3 in float32, 3e-2 with bfloat16 storage)."""
import numpy as np
import pytest

from oracle import numeric_oracle as no
from paper_2502_12499_b200 import binding as ck
from paper_2502_12499_b200 import workloads as wl
from tests.gpu_util import StepRunner, max_rel_err

pytestmark = pytest.mark.gpu

SHAPES = [("f32", 4, 3, 6, 10), ("f32", 12, 2, 2, 2), ("f32", 100, 2, 4, 6), ("f32", 1024, 1, 2, 4), ("f32", 1028, 1, 2, 4), ("f32", 64, 5, 14, 18),
          ("bf16", 8, 3, 6, 10), ("bf16", 48, 3, 10, 6), ("bf16", 72, 5, 2, 2), ("bf16", 256, 2, 4, 6), ("bf16", 2048, 1, 2, 4), ("bf16", 2056, 1, 2, 4)]


@pytest.mark.parametrize("dtype,c,batch,h,w", SHAPES)
def test_pool_behind_batch_norm(dtype, c, batch, h, w):
    spec = dict(units=[wl.conv_unit(8, c), {"kind": "maxpool", "k": 2, "stride": 2, "pad": 0}, {"kind": "avgpool"},
                       {"kind": "fc", "cin": c, "cout": 10, "relu": False}],
                input_hwc=(h, w, 8), batch=batch, dtype=dtype, loss="softmax_ce", name="pool_%s_%d" % (dtype, c))
    params = wl.make_params(spec, seed=11, bn_affine="random")
    x, labels = wl.make_batch(spec, seed=12)
    runner = StepRunner(spec, params)
    rep, grads = runner.run(ck.POLICY_STORE_ALL, None, x, labels)
    ref = no.chain_forward_backward(spec, [{k: v.astype(np.float64) for k, v in p.items()} for p in params], x.astype(np.float64), labels,
                                    storage="bf16" if dtype == "bf16" else "exact")
    tol = 3e-2 if dtype == "bf16" else 1e-3
    assert abs(rep["loss"] - ref["loss"]) <= tol * abs(ref["loss"])
    for (ui, name, _), g in zip(runner.flat, grads):
        want = ref["grads"][ui][name]
        assert max_rel_err(g.reshape(want.shape), want) <= tol, (ui, name)


@pytest.mark.parametrize("batch,h,w,c", [(64, 56, 56, 256), (128, 32, 32, 64), (64, 14, 14, 512)])
def test_sums_behind_pooling_against_float64(batch, h, w, c):
    """dgamma and dbeta of the convolution in front of a pooling against float64 sums of the same stored z, statistics and gradient.
    A float32 result is off by 2.5e-8 of its norm from its own rounding (2^-24 of the last place's value at most, 0.58 of that in the root
    mean square, over mantissas between 1 and 2); a quarter more is left for the sums in front of it.  Plain float32 chains: 3.0e-8 to
    5.4e-8 for dgamma."""
    import torch
    spec = dict(units=[wl.conv_unit(64, c, 1, 1, 0), {"kind": "maxpool", "k": 2, "stride": 2, "pad": 0},
                       {"kind": "fc", "cin": (h // 2) * (w // 2) * c, "cout": 16, "relu": False}],
                input_hwc=(h, w, 64), batch=batch, dtype="bf16", loss="softmax_ce", name="pool_sums")
    chain = ck.Chain(spec)
    d = [int(v) for v in chain.sizes()]

    def empty(n):
        return torch.empty(n, dtype=torch.uint8, device="cuda")

    arena, workspace, tap = empty(sum(d)), empty(chain.workspace_bytes()), empty(sum(d[1:]))
    chain.set_gradient_tap(tap)
    shape = ck.ConvShape(batch, h, w, 64, c, 1, 1, 0)
    scratch = empty(max(ck.conv2d_scratch_bytes(shape, ck.DTYPE_BF16), ck.bn_scratch_bytes(batch * h * w, c)) + 256)
    labels = torch.arange(batch, device="cuda", dtype=torch.int32) % 16
    errors = []
    for seed in range(8):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)

        def rand(*dims, scale=1.0):
            return torch.randn(dims, generator=gen, device="cuda") * scale

        x = rand(batch, h, w, 64).bfloat16()
        params = [rand(c, 1, 1, 64, scale=0.2).bfloat16(), torch.rand(c, generator=gen, device="cuda") + 0.5, rand(c, scale=0.2),
                  rand(16, (h // 2) * (w // 2) * c, scale=1e-3).bfloat16(), rand(16, scale=0.1)]
        grads = [torch.zeros(p.shape, device="cuda") for p in params]
        ck.train_step(chain, None, ck.POLICY_STORE_ALL, x, labels, params, grads, arena, workspace)
        z, stats = torch.empty((batch, h, w, c), dtype=torch.bfloat16, device="cuda"), torch.empty((4, c), device="cuda")
        ck.conv2d_bn_statistics(shape, ck.DTYPE_BF16, x, params[0], z, params[1], params[2], stats, scratch)       # as the step has them
        dy = tap[d[1]:].view(torch.bfloat16)[:batch * (h // 2) * (w // 2) * c].view(batch, h // 2, w // 2, c)
        mean, inv, scale, shift = stats.double()
        sum_g = torch.zeros(c, dtype=torch.double, device="cuda")
        sum_gz = torch.zeros_like(sum_g)
        for i in range(0, batch, 8):
            windows = z[i:i + 8].double().view(-1, h // 2, 2, w // 2, 2, c).permute(0, 1, 3, 5, 2, 4).flatten(-2)          # row-major in a window
            seen = torch.relu((windows * scale[:, None] + shift[:, None]).float()).bfloat16()
            top = seen.amax(-1, keepdim=True)
            first = (seen == top).float().argmax(-1, keepdim=True)
            g = torch.where(top[..., 0] > 0, dy[i:i + 8].double(), 0.0)
            sum_g += g.sum((0, 1, 2))
            sum_gz += (g * windows.gather(-1, first)[..., 0]).sum((0, 1, 2))
        dgamma = inv * (sum_gz - mean * sum_g)
        errors.append([((grads[1].double() - dgamma).norm() / dgamma.norm()).item(), ((grads[2].double() - sum_g).norm() / sum_g.norm()).item()])
    chain.set_gradient_tap(None)
    of_dgamma, of_dbeta = np.mean(errors, axis=0)
    assert of_dgamma <= 1.25 * 2.5e-8 and of_dbeta <= 1.25 * 2.5e-8, (of_dgamma, of_dbeta)
