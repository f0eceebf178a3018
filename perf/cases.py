"""Performance cases of the framework: what a user has it do, through its public entry points.

A case is one of

* a training step (``binding.train_step``) of a convolutional chain - VGG-shaped, bottleneck-residual or plain - under
  one of the schedules (planned checkpoints with early free, planned checkpoints freed per batch, store all), launched
  kernel by kernel or replayed from its recording, on a batch in device memory or one staged from pinned host memory;
  with a classifier's loss the step updates the parameters, under the sum loss it leaves the gradients;
* one layer's single operations (``kind == "layer"``), each on tensors of its own: convolution, batch norm + ReLU and 2x2
  pooling, forward and backward.

Parameters: He-normal matrices, batch-norm scales in [0.5, 1.5] and shifts of 0.2 standard deviations as trained
networks have them; images N(0, 1), uniform labels.
"""
import math

import torch

from paper_2502_12499_b200 import binding as ck
from paper_2502_12499_b200 import workloads as wl

POLICIES = {"plan": ck.POLICY_DYNAMIC, "batch_free": ck.POLICY_STATIC, "store_all": ck.POLICY_STORE_ALL,
            "keep_interiors": ck.POLICY_STORE_ALL}
LEARNING_RATE = 1e-4       # the first steps of a warm-up


def _step(kind, dtype="bf16", policy="plan", graph=True, staged=False, **sizes):
    return dict(kind=kind, dtype=dtype, policy=policy, graph=graph, staged=staged, **sizes)


def listed():
    return [
        # the smallest call: eight 16-channel float32 layers on four 32 x 32 images, launched kernel by kernel (the
        # repository's first configuration); launches and host work are all there is
        dict(_step("plain", "f32", graph=False, units=8, channels=16, in_channels=3, classes=0, h=32, w=32, batch=4), name="plain8_f32"),
        # classification of 32 x 32 images: many small kernels, replayed from the recording
        dict(_step("vgg", base=64, fc=512, classes=10, h=32, w=32, batch=128), name="vgg16_32px_b128"),
        # the headline configuration: VGG-16 at 224 x 224, batch 64, least recomputation at Algorithm 6's peak
        dict(_step("vgg", base=64, fc=4096, classes=1000, h=224, w=224, batch=64), name="vgg16_b64"),
        # finer granularity (convolution, normalisation, ReLU as units of their own), an odd batch of ragged images, the
        # batch-free schedule on Algorithm 3's plan, launched kernel by kernel
        dict(_step("vgg", policy="batch_free", graph=False, split=True, base=64, fc=1024, classes=100, h=160, w=96, batch=13), name="vgg16_split_b13"),
        # channel counts that are no multiple of 64 (a slimmed network)
        dict(_step("vgg", base=48, fc=1000, classes=100, h=96, w=96, batch=16), name="vgg16_slim48_b16"),
        # full-precision training of a small network
        dict(_step("vgg", "f32", base=32, fc=256, classes=10, h=32, w=32, batch=32), name="vgg16_f32_32px_b32"),
        # residual network at the size it is trained at (third configuration)
        dict(_step("resnet", b1=3, b2=4, b3=6, b4=3, base=64, classes=1000, h=224, w=224, batch=128), name="resnet50_b128"),
        # enough memory to keep everything, odd image sizes and an odd batch
        dict(_step("resnet", policy="keep_interiors", b1=3, b2=4, b3=6, b4=3, base=64, classes=1000, h=200, w=168, batch=21), name="resnet50_keep_b21"),
        # training loop end to end: every step's batch from pinned host memory, the next one's copy under this step
        dict(_step("resnet", staged=True, b1=3, b2=4, b3=6, b4=3, base=64, classes=1000, h=224, w=224, batch=32), name="resnet50_staged_b32"),
        # the largest configuration (the fourth)
        dict(_step("resnet", b1=3, b2=8, b3=36, b4=3, base=64, classes=1000, h=224, w=224, batch=256), name="resnet152_b256"),
        # deep chain of small kernels: the fifth configuration's unit under a classifier, as many of them as keep the
        # update of the first below a few per cent (a chain's gradients grow by 1.18 per unit)
        dict(_step("plain", units=32, channels=64, in_channels=64, classes=100, h=56, w=56, batch=32), name="plain32_b32"),
        # one layer by the single operations
        dict(kind="layer", dtype="bf16", cin=128, cout=256, k=3, stride=1, h=56, w=56, batch=32, name="layer_128_256_56px"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above; its arithmetic is held below that of the largest listed case."""
    while True:
        kind = rng.choice(["vgg", "vgg", "resnet", "resnet", "plain", "plain", "layer"])
        dtype = "f32" if rng.random() < 0.2 else "bf16"
        policy = rng.choice(["plan", "plan", "batch_free", "store_all"])
        graph = rng.random() < 0.6
        staged = rng.random() < 0.2
        if kind == "vgg":
            c = _step("vgg", dtype, policy, graph, staged, split=rng.random() < 0.2, base=rng.choice([32, 48, 64, 64, 64, 96]), fc=8 * _log(rng, 32, 512),
                      classes=rng.randint(10, 1000), h=32 * rng.randint(1, 7), w=32 * rng.randint(1, 7), batch=_log(rng, 8, 64))
        elif kind == "resnet":
            policy = rng.choice([policy, "keep_interiors"])
            c = _step("resnet", dtype, policy, graph, staged, b1=rng.randint(1, 3), b2=rng.randint(1, 8), b3=rng.randint(1, 36), b4=rng.randint(1, 3),
                      base=rng.choice([32, 64, 64, 64]), classes=rng.randint(10, 1000), h=rng.randint(64, 224), w=rng.randint(64, 224),
                      batch=_log(rng, 8, 256))
        elif kind == "plain":
            channels = rng.choice([16, 24, 32, 48, 64, 64, 64, 96, 128, 128, 256])
            c = _step("plain", dtype, policy, graph, staged, units=_log(rng, 4, 32), channels=channels, in_channels=rng.choice([3, channels]),
                      classes=rng.randint(10, 1000), h=_log(rng, 14, 112), w=_log(rng, 14, 112), batch=_log(rng, 4, 64))
        else:
            c = dict(kind="layer", dtype=dtype, cin=rng.choice([3, 32, 64, 64, 96, 128, 256, 512]), cout=rng.choice([32, 64, 64, 96, 128, 256, 512]),
                     k=rng.choice([1, 3, 3]), stride=rng.choice([1, 1, 1, 2]), h=_log(rng, 7, 112), w=_log(rng, 7, 112), batch=_log(rng, 4, 64))
        w = work(c)
        odd = c.get("base", c.get("channels", 64)) % 64 or c["dtype"] == "f32"
        if w["flops"] < (5e11 if odd else 2e13) and w["bytes"] < 1.2e11:
            return c


# ------------------------------------------------------------------------------------------------
# chains
# ------------------------------------------------------------------------------------------------

def _spec(case):
    hw = (case["h"], case["w"])
    if case["kind"] == "vgg":
        b = case["base"]
        spec = wl.vgg16_chain(case["batch"], hw=hw, dtype=case["dtype"], widths=(b, 2 * b, 4 * b, 8 * b, 8 * b), fc_width=case["fc"],
                              classes=case["classes"])
        return wl.split_units(spec)[0] if case.get("split") else spec
    if case["kind"] == "resnet":
        return wl.resnet_chain([case["b%d" % s] for s in (1, 2, 3, 4)], case["batch"], hw=hw, dtype=case["dtype"], base=case["base"],
                               classes=case["classes"])
    spec = wl.plain_chain(case["units"], case["channels"], case["in_channels"], hw, case["batch"], case["dtype"],
                          "softmax_ce" if case["classes"] else "sum")
    if case["classes"]:
        spec["units"] += [{"kind": "avgpool"}, {"kind": "fc", "cin": case["channels"], "cout": case["classes"], "relu": False}]
    return spec


def _mask(case, chain):
    """The checkpoint set of the case's schedule, as a user plans it."""
    d = chain.sizes()
    if POLICIES[case["policy"]] == ck.POLICY_STORE_ALL:
        return None
    if case["policy"] == "batch_free":
        return ck.plan(ck.ALGO_STATIC_N3, d)[0]
    return ck.plan_min_recompute(d, chain.unit_costs())[0]


def _peak(case, chain, mask):
    model = {"plan": ck.MODEL_DYNAMIC, "batch_free": ck.MODEL_STATIC}.get(case["policy"], ck.MODEL_STORE_ALL)
    return ck.eval(model, chain.sizes(), mask)


def _convs(unit, shape_in, shape_out):
    """(output positions, filter size^2 * input channels, output channels) of every contraction of one unit."""
    px_in, px_out = shape_in[0] * shape_in[1], shape_out[0] * shape_out[1]
    if unit["kind"] in ("conv_bn_relu", "conv"):
        return [(px_out, unit["k"] ** 2 * unit["cin"], unit["cout"])]
    if unit["kind"] == "fc":
        return [(1, unit["cin"], unit["cout"])]
    if unit["kind"] == "bottleneck":
        out = [(px_in, unit["cin"], unit["mid"]), (px_out, 9 * unit["mid"], unit["mid"]), (px_out, unit["mid"], unit["cout"])]
        return out + ([(px_out, unit["cin"], unit["cout"])] if unit["project"] else [])
    return []


class _Tensors:
    """One tensor per parameter, as views of a few buffers (a buffer holds one kind of parameter of neighbouring
    units), the way a training program keeps them for its optimiser."""
    BINS = 20

    def __init__(self, spec, dtype_of):
        self.items, used = [], {}
        n = len(spec["units"])
        for ui, unit in enumerate(spec["units"]):
            for name, shape in wl.param_shapes(unit).items():
                key = "%s%02d" % (name[0], ui * self.BINS // max(n, self.BINS))
                self.items.append((unit, name, shape, key, used.get(key, 0)))
                used[key] = used.get(key, 0) + -(-math.prod(shape) // 64) * 64
        self.buffers = {key: torch.zeros(size, dtype=dtype_of(key[0]), device="cuda") for key, size in used.items()}
        self.views = [self.buffers[key][at:at + math.prod(shape)].view(shape) for _, _, shape, key, at in self.items]


def _fill_params(tensors, gen):
    for (unit, name, shape, _, _), t in zip(tensors.items, tensors.views):
        if name[0] == "w":
            t.copy_(torch.randn(shape, generator=gen, device="cuda") * math.sqrt(2.0 / math.prod(shape[1:])))
        elif name[0] == "g":
            t.copy_(torch.rand(shape, generator=gen, device="cuda") + 0.5)
        else:
            t.copy_(torch.randn(shape, generator=gen, device="cuda") * (0.1 if unit["kind"] == "fc" else 0.2))


def _storage(dtype):
    return torch.bfloat16 if dtype == "bf16" else torch.float32


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] == "layer":
        return _prepare_layer(case, gen)
    spec = _spec(case)
    chain = ck.Chain(spec)
    if case["graph"]:
        chain.set_graph(True)
    if case["classes"]:
        chain.set_sgd(LEARNING_RATE)
    if case["policy"] == "keep_interiors":
        chain.set_keep_interiors(True)
    mask, policy = _mask(case, chain), POLICIES[case["policy"]]
    store = _storage(case["dtype"])
    params = _Tensors(spec, lambda kind: store if kind == "w" else torch.float32)
    _fill_params(params, gen)
    grads = _Tensors(spec, lambda kind: torch.float32)
    h, w, c = spec["input_hwc"]
    x = torch.randn((spec["batch"], h, w, c), generator=gen, device="cuda").to(store)
    labels = None
    if spec["loss"] == "softmax_ce":
        labels = torch.randint(0, case["classes"], (spec["batch"],), generator=gen, device="cuda", dtype=torch.int32)
    state = dict(case=case, chain=chain, mask=mask, policy=policy, params=params, grads=grads,
                 arena=torch.empty(_peak(case, chain, mask), dtype=torch.uint8, device="cuda"),
                 workspace=torch.empty(chain.workspace_bytes_for(policy), dtype=torch.uint8, device="cuda"))
    if case["staged"]:
        state["host"] = (x.cpu().pin_memory(), None if labels is None else labels.cpu().pin_memory())
        state["staging"] = torch.empty(chain.staging_bytes(), dtype=torch.uint8, device="cuda")
        state["slot"] = 0
        state["next"] = chain.stage_batch(0, *state["host"], state["staging"])
    else:
        state["batch"] = (x, labels)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "layer":
        return _run_layer(state)
    batch = state.get("batch")
    if batch is None:
        batch = state["next"]
        state["slot"] ^= 1
        state["next"] = state["chain"].stage_batch(state["slot"], *state["host"], state["staging"])
    report = ck.train_step(state["chain"], state["mask"], state["policy"], batch[0], batch[1], state["params"].views, state["grads"].views,
                           state["arena"], state["workspace"])
    # with the update the step's result is the new parameters; without it the gradients
    return {"loss": report["loss"], "state": (state["params"] if case["classes"] else state["grads"]).buffers}


# ------------------------------------------------------------------------------------------------
# one layer by the single operations
# ------------------------------------------------------------------------------------------------

def _layer_shape(case):
    pad = case["k"] // 2
    ho, wo = ((v + 2 * pad - case["k"]) // case["stride"] + 1 for v in (case["h"], case["w"]))
    return ck.ConvShape(case["batch"], case["h"], case["w"], case["cin"], case["cout"], case["k"], case["stride"], pad), ho, wo


def _prepare_layer(case, gen):
    shape, ho, wo = _layer_shape(case)
    dtype = ck.DTYPE_BF16 if case["dtype"] == "bf16" else ck.DTYPE_F32
    n, c, store = case["batch"], case["cout"], _storage(case["dtype"])

    def rand(*dims):
        return torch.randn(dims, generator=gen, device="cuda")

    s = dict(case=case, shape=shape, dtype=dtype, rows=n * ho * wo, out=(ho, wo), x=rand(n, case["h"], case["w"], case["cin"]).to(store),
             w=(rand(c, case["k"], case["k"], case["cin"]) * math.sqrt(2.0 / (case["k"] ** 2 * case["cin"]))).to(store),
             gamma=torch.rand(c, generator=gen, device="cuda") + 0.5, beta=0.2 * rand(c), z_in=(1.4 * rand(n, ho, wo, c) + 0.3 * rand(c)).to(store),
             g_in=rand(n, ho, wo, c).to(store), g_pool=rand(n, ho // 2, wo // 2, c).to(store))
    mean, var = s["z_in"].double().mean((0, 1, 2)), s["z_in"].double().var((0, 1, 2), unbiased=False)
    inv = (var + 1e-5).rsqrt()
    s["saved"] = torch.stack((mean, inv, s["gamma"] * inv, s["beta"] - mean * s["gamma"] * inv)).float()      # of the forward pass
    s["y_in"] = torch.relu(s["z_in"] * s["saved"][2] + s["saved"][3]).to(store)
    for name, dims in (("z", (n, ho, wo, c)), ("y", (n, ho, wo, c)), ("pool", (n, ho // 2, wo // 2, c)), ("dy", (n, ho, wo, c)),
                       ("dz", (n, ho, wo, c)), ("dx", (n, case["h"], case["w"], case["cin"]))):
        s[name] = torch.empty(dims, dtype=store, device="cuda")
    for name, dims in (("stats", (4, c)), ("dgamma", (c,)), ("dbeta", (c,)), ("dw", tuple(s["w"].shape))):
        s[name] = torch.empty(dims, dtype=torch.float32, device="cuda")
    sizes = (ck.conv2d_scratch_bytes(shape, dtype), ck.bn_scratch_bytes(s["rows"], c), ck.maxpool_backward_scratch_bytes(dtype, n, ho, wo, c, 2, 2, 0))
    s["scratch"] = torch.empty(max(sizes + (256,)), dtype=torch.uint8, device="cuda")
    return s


def _run_layer(s):
    shape, dt, rows, c, scratch = s["shape"], s["dtype"], s["rows"], s["case"]["cout"], s["scratch"]
    pool = (dt, s["case"]["batch"], s["out"][0], s["out"][1], c, 2, 2, 0)
    ck.conv2d_forward(shape, dt, 0, s["x"], s["w"], s["z"], scratch)
    ck.bn_relu_forward(dt, rows, c, s["z_in"], s["gamma"], s["beta"], 1, s["y"], s["stats"], scratch)
    ck.maxpool_forward(*pool, s["y_in"], s["pool"])
    ck.maxpool_backward(*pool, s["y_in"], s["g_pool"], s["dy"], scratch)
    ck.bn_relu_backward(dt, rows, c, s["g_in"], s["z_in"], s["gamma"], s["saved"], 1, s["dz"], s["dgamma"], s["dbeta"], scratch)
    ck.conv2d_dgrad(shape, dt, 0, s["g_in"], s["w"], s["dx"], scratch)
    ck.conv2d_wgrad(shape, dt, 0, s["g_in"], s["x"], s["dw"], scratch)
    return {name: s[name] for name in ("z", "y", "stats", "pool", "dy", "dz", "dgamma", "dbeta", "dx", "dw")}


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct passes may lie apart
# ------------------------------------------------------------------------------------------------

def work(case):
    """Arithmetic: every contraction forward, once more for a unit that the schedule recomputes (a residual block whose
    interior tensors are not kept counts as one more forward), and twice backward (the first unit has no input
    gradient).  Bytes: every unit's input and output once per forward, its input, its incoming and its outgoing gradient
    once in the backward, the parameters once per phase and the gradients once; batch normalisation has to see a whole
    tensor before it can apply itself, so the tensors between units cannot stay on the chip."""
    es = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "layer":
        shape, ho, wo = _layer_shape(case)
        n, c, px_in, px = case["batch"], case["cout"], case["h"] * case["w"], ho * wo
        weights = c * case["k"] ** 2 * case["cin"]
        tensors = 2 * n * px_in * case["cin"] + n * px * c * 9 + 2 * n * (ho // 2) * (wo // 2) * c
        return {"bytes": es * (tensors + 2 * weights) + 4 * weights, "flops": 6.0 * n * px * weights}
    spec = _spec(case)
    chain = ck.Chain(spec)
    d, shapes, mask = chain.sizes(), chain.shapes(), _mask(case, chain)
    n_bytes = flops = 0.0
    for i, unit in enumerate(spec["units"], start=1):
        convs = _convs(unit, shapes[i - 1], shapes[i])
        forward = sum(2.0 * spec["batch"] * px * k * c for px, k, c in convs)
        weights = sum(k * c for _, k, c in convs)
        passes = 1 + (mask is not None and not mask[i])
        again = unit["kind"] == "bottleneck" and case["policy"] != "keep_interiors"
        flops += forward * (passes + again + (2 if i > 1 else 1))
        n_bytes += passes * float(d[i - 1] + d[i]) + float(d[i - 1] + d[i] + (d[i - 1] if i > 1 else 0)) + weights * (es * (passes + 1) + 4)
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    """Measured between this path and a copy of it that takes the batch-norm sums (forward and backward) and the float32
    convolution sums in another order, about four times what was seen.

    Single operations differ by the order of float32 sums, and by single roundings of stored bfloat16 values (one unit
    in the last place is at most 2^-7 of a value; 3e-6..5e-5 in norm).  In a whole network a last bit of a batch-norm sum
    flips ReLU decisions further on, and at random initialisation a gradient is a sum of products without a dominant
    term: a share f of flipped terms moves it by sqrt(f).  After four layers in bfloat16 every implementation rounds
    independently and the early gradients lie 30-50 % apart, in float32 a few flips in 1e7 remain (3e-3).  The updated
    parameters carry that difference times the learning rate: up to 1e-2 in the deepest networks' first layers."""
    if case["kind"] == "layer":
        return {"rel": 2e-3, "max": 0.03} if case["dtype"] == "bf16" else {"rel": 2e-5, "max": 1e-3}
    if not case["classes"]:
        return {"rel": 0.015, "max": 0.15}
    if case["dtype"] == "f32" and case["kind"] != "resnet":
        return {"rel": 1e-3, "max": 0.03}           # (seen: 1e-5; fifty layers of a residual network: 6e-3)
    return {"rel": 0.02, "max": 0.3}
