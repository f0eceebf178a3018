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
