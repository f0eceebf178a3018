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
