"""Whole training steps of the benchmark configurations against the oracle, in bfloat16, at the configurations' own
layer shapes (reduced batch where the float64 oracle needs it) and on the tensor-core dispatch.

Two comparisons per chain, both on a store-all step (Algorithm 1; every checkpointed schedule is bit-identical to it,
see test_gpu_step.py / test_gpu_fullsize.py):

1. Unit by unit (tests/parity_util.py): the oracle's definition of each unit is given the tensors the executor's unit
   was given - its stored input d_{i-1} and its incoming gradient r_i (Eqs. (2)-(3)) - and must reproduce the unit's
   stored output d_i, its weight gradients g_i (Eq. (5)) and its outgoing gradient r_{i-1}, each element-wise within
   3e-2 of the tensor's largest magnitude.  Both sides take every ReLU and arg-max decision on the same stored
   bfloat16 codes, so nothing amplifies: observed errors are 6e-3 and below.  Inside a bottleneck block the three
   interior activations are re-derived by each side from the block's input, so a handful of interior ReLU decisions
   can differ (a few per million elements); an element of a weight gradient summed over few pixels, or of the
   outgoing gradient, that meets such a decision moves by a whole term.  For the quantities downstream of interior
   decisions (w1, g1, b1, w2, g2, b2 and r_{i-1} of a block) the bound is therefore: relative L2 distance <= 3e-2 and
   at most 2 % of the elements further than 3e-2 from the reference; everything else in a block is element-wise.
   The same holds, far more rarely, for a max-pool that reads a conv unit's output through its pending
   normalisation: the executor normalises in float32, the oracle in float64, and in a few windows per ten million
   the two largest values end up in the other order (equal or adjacent bfloat16 codes), so the gradient lands on the
   neighbouring element - both are valid arg-max choices.  For the gradient leaving such a pool at most 1e-5 of the
   elements may differ, with the relative L2 distance still <= 3e-2.

2. End to end: every weight gradient against the oracle's own whole step with the same storage rounding.  Measured
   at these shapes, the two runs take different ReLU decisions on a fraction f_i of the elements of layer i that
   grows with depth (1e-7 after one layer, 1 % after 16 - one rounding that falls the other way flips decisions
   downstream), and at random initialisation a weight gradient is a sum of products without a dominant term, so
   changing a fraction f of its terms moves it by about sqrt(f) in relative L2 norm: 10-50 % on the early layers of
   these chains, for any two independent implementations (the oracle's own two storage modes included).  The
   element-wise bound of 3e-2 is asserted where no decision differs upstream; elsewhere the deviation has to stay
   within 3e-2 + 4 sqrt(sum of the measured flip fractions), and the loss within 2 %.
"""
import numpy as np
import pytest

from oracle import numeric_oracle as no
from paper_2502_12499_b200 import binding as ck
from paper_2502_12499_b200 import workloads as wl
from tests import parity_util as pu
from tests.gpu_util import StepRunner

pytestmark = pytest.mark.gpu
TOL = 3e-2
FLIP_SENSITIVE = {"dw1", "dg1", "db1", "dw2", "dg2", "db2"}


def run_case(spec, seed=0):
    params = wl.make_params(spec, seed=seed, bn_affine="random")
    x, labels = wl.make_batch(spec, seed=seed + 1)
    if spec["loss"] != "softmax_ce":
        labels = None
    runner = StepRunner(spec, params)
    step = pu.StoredStep(runner, x, labels)
    assert step.report["device_status"] == 0 and np.isfinite(step.report["loss"])
    return params, x, labels, step


def assert_tensor_core_dispatch(step, expected):
    cuda_core = [k for k in step.kernels if "CUDA cores" in k]
    assert not cuda_core, cuda_core
    for name in expected:
        assert step.kernels.get(name, 0) > 0, (name, sorted(step.kernels))


def assert_units_match_locally(step, params, labels):
    rows = pu.check_units_locally(step, params, labels, "bf16")
    kinds = [u["kind"] for u in step.spec["units"]]
    bad = []
    for where, what, err, l2, outliers in rows:
        in_block = 1 <= where <= len(kinds) and kinds[where - 1] == "bottleneck"
        # r_i leaves the backward of unit i+1: flip-sensitive when that unit is a block
        from_block = what == "r_i" and where < len(kinds) and kinds[where] == "bottleneck"
        # r_i leaves a max-pool that read a conv unit's output through its pending normalisation
        from_pool = what == "r_i" and where < len(kinds) and kinds[where] == "maxpool" and kinds[where - 1] == "conv_bn_relu"
        if (in_block and what in FLIP_SENSITIVE) or from_block:
            ok = l2 <= TOL and outliers <= 2e-2
        elif from_pool:
            ok = err <= TOL or (l2 <= TOL and outliers <= 1e-5)
        else:
            ok = err <= TOL
        if not ok:
            bad.append((where, what, err, l2, outliers))
    assert not bad, bad
    return rows


def assert_whole_step_explained(step, params, x, labels):
    p64 = [{k: v.astype(np.float64) for k, v in p.items()} for p in params]
    ref = no.chain_forward_backward(step.spec, p64, x.astype(np.float64), labels, storage="bf16")
    assert abs(step.report["loss"] - ref["loss"]) <= 2e-2 * abs(ref["loss"])
    flips = pu.decision_flips(step, params, ref)
    total = sum(f for _, f in flips)
    bound = TOL + 4.0 * np.sqrt(total)
    table = pu.whole_step_errors(step, ref)
    n = len(step.spec["units"])
    for unit, name, err, l2 in table:
        # decisions upstream of unit's gradient: every layer for the backward signal, so only a chain without any
        # differing decision gets the element-wise bound; the last unit's parameters see the forward flips only
        upstream = total if unit < n else sum(f for i, f in flips if i < n)
        if upstream == 0.0:
            assert err <= TOL, (unit, name, err, flips)
        assert l2 <= bound, (unit, name, err, l2, bound, flips)
    return table, flips


def test_config2_vgg16_chain():
    """The VGG-16 chain unchanged (224 x 224, full widths) at batch 13: every 3x3 layer from 224 x 224 down to 28 x 28
    takes the halo-patch role-swapped kernel as at batch 64, the 14 x 14 layers the role-swapped kernel."""
    spec = dict(wl.config(2), batch=13)
    params, x, labels, step = run_case(spec)
    assert_tensor_core_dispatch(step, ["tc_conv_first_kernel", "tc_conv_tp_kernel", "tc_conv_t_kernel", "tc_wgrad_rows_kernel",
                                       "tc_wgrad_rows_kernel (pixel pairs)", "tc_fc_fwd_kernel", "tc_conv_wgrad_kernel",
                                       "max-pool 2x2 backward with batch-norm sums"])
    assert step.kernels["tc_conv_tp_kernel"] >= 16          # forward and dgrad of conv1_2 .. conv4_3
    assert_units_match_locally(step, params, labels)
    assert_whole_step_explained(step, params, x, labels)


def test_config3_resnet50_chain():
    """The ResNet-50 chain unchanged at batch 16: stem on its own gather kernels, 3x3 stride-2 max-pool, all 16
    bottleneck blocks (projection, stride 2, identity), average pool, classifier."""
    spec = dict(wl.config(3), batch=16)
    params, x, labels, step = run_case(spec)
    assert_tensor_core_dispatch(step, ["tc_conv_stem_kernel", "tc_wgrad_stem_kernel", "tc_conv_t_kernel", "tc_conv_fwd_kernel", "tc_conv_c64_kernel",
                                       "tc_conv_wgrad_kernel", "tc_wgrad_rows_kernel", "residual join", "gradient join",
                                       "max-pool backward from arg-max"])
    assert_units_match_locally(step, params, labels)
    assert_whole_step_explained(step, params, x, labels)


def test_config4_resnet152_chain_unit_by_unit():
    """All 54 units of the ResNet-152 chain at batch 4, unit by unit."""
    spec = dict(wl.config(4), batch=4)
    params, x, labels, step = run_case(spec)
    assert_tensor_core_dispatch(step, ["tc_conv_t_kernel", "tc_conv_wgrad_kernel"])
    assert_units_match_locally(step, params, labels)


def test_config5_first_units_at_full_tensor_size():
    """The first 16 units of the 1000-unit chain on its real tensors (32 x 56 x 56 x 64): pixel-pair form of the
    halo-patch kernel forward and dgrad, pixel-pair wgrad, as in the full configuration."""
    spec = wl.config(5)
    spec = dict(spec, units=spec["units"][:16])
    params, x, labels, step = run_case(spec)
    assert_tensor_core_dispatch(step, ["tc_conv_tp_kernel", "tc_wgrad_rows_kernel (pixel pairs)", "pairview_fold_kernel"])
    assert step.kernels["tc_conv_tp_kernel"] == 31
    assert_units_match_locally(step, params, labels)
    assert_whole_step_explained(step, params, x, labels)


def resnet_stage_blocks(stage, batch):
    """The first two blocks of a ResNet-50 stage (projection block, identity block) on that stage's input."""
    mid = 64 * 2 ** stage
    cin = 64 if stage == 0 else 2 * mid
    hw = 56 if stage == 0 else 56 // 2 ** (stage - 1)
    units = [{"kind": "bottleneck", "cin": cin, "mid": mid, "cout": 4 * mid, "stride": 1 if stage == 0 else 2, "project": True},
             {"kind": "bottleneck", "cin": 4 * mid, "mid": mid, "cout": 4 * mid, "stride": 1, "project": False}]
    return dict(units=units, input_hwc=(hw, hw, cin), batch=batch, dtype="bf16", loss="sum", name="stage%d_blocks" % stage)


@pytest.mark.parametrize("stage,batch,expected", [
    (0, 64, ["tc_conv_tp_kernel", "tc_wgrad_rows_kernel (pixel pairs)", "tc_conv_t_kernel"]),
    (1, 64, ["tc_conv_tp_kernel", "tc_wgrad_rows_kernel", "tc_conv_t_kernel"]),
])
def test_resnet_blocks_at_benchmark_dispatch(stage, batch, expected):
    """Bottleneck blocks at a batch large enough for the kernels the full-batch configurations run: the pixel-pair
    halo-patch form for the 64-channel 3x3 layer, the halo-patch form for the 128-channel one, strided boxes for the
    stride-2 layers."""
    spec = resnet_stage_blocks(stage, batch)
    params, x, labels, step = run_case(spec, seed=5)
    assert_tensor_core_dispatch(step, expected)
    assert_units_match_locally(step, params, labels)


@pytest.mark.parametrize("batch", [6, 13])
def test_wide_blocks_share_long_reductions(batch):
    """Residual blocks of 2048 channels on few pixels: the joined input gradient and the residual join of a recomputed
    output share one tile's 2048-channel reduction among the CTAs of a cluster, in tiles of 160 pixels.  The store-all
    step against the oracle, and the checkpointed step (which recomputes the first block) bit for bit against it."""
    plan = ck.selftest_conv_plan(ck.ConvShape(batch, 7, 7, 2048, 2048, 1, 1, 0), 1)
    assert plan["split"] > 1 and plan["pixels"] >= 160, plan
    block = {"kind": "bottleneck", "cin": 2048, "mid": 2048, "cout": 2048, "stride": 1, "project": False}
    spec = dict(units=[block, dict(block)], input_hwc=(7, 7, 2048), batch=batch, dtype="bf16", loss="sum", name="wide_blocks")
    params, x, labels, step = run_case(spec, seed=9)
    assert_tensor_core_dispatch(step, ["tc_conv_t_kernel"])
    assert_units_match_locally(step, params, labels)
    _, kept = step.runner.run(ck.POLICY_STORE_ALL, None, x, labels)
    report, grads = step.runner.run(ck.POLICY_DYNAMIC, ck.mask_from_set(2, [0, 2]), x, labels)
    assert report["device_status"] == 0 and report["recomputed_units"] > 0
    for a, b in zip(kept, grads):
        assert np.array_equal(a, b)
