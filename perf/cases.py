"""The work a user of the library has it do, as cases that can be timed and compared.

Four kinds of case:

  train     a closed-loop training step of a Fixup ResNet (``chain.ChainedStep``): image quantizer, all convolution
            units forward, float head, backward with error joins and weight gradients, 8-bit update.  The program
            captured the step once and replays it; every pass is the next step of the run.
  layers    convolution units called one by one on tensors the program has at hand: forward only, backward only
            (error head, error back-propagation, weight gradient) or all of it with the weight update.  One unit is
            called directly; the units of a bottleneck block are captured once and replayed.
  quantize  the standalone quantizers on an fp32 tensor.
  update    the 8-bit update of all weight tensors of a network in one call.
"""
import math

import torch

from paper_2105_13890_b200 import chain, eoq, workloads

DEV = "cuda:0"
ROUND = {"nearest": eoq.EOQ_ROUND_RNE, "stochastic": eoq.EOQ_ROUND_STOCHASTIC}
QMODE = {"Q": eoq.EOQ_Q, "CQ": eoq.EOQ_CQ, "SQ": eoq.EOQ_SQ}
MOST_MACS = 512 * 56 * 56 * 64 * 64 * 9     # of one drawn layer: those of the largest listed one
MOST_PIXELS = 64 * 224 * 224                # images of a drawn training step: those of the largest listed one


def listed():
    return [
        # online training, one image at a time: launches and dependencies count, not arithmetic
        _train("online step ResNet-18 b1", "resnet18", 1, 224, "stochastic"),
        # the same on a CIFAR-shaped stream, a few images at a time
        _train("small batch ResNet-20 b2", "resnet20", 2, 32, "stochastic"),
        # the CIFAR-shaped network at its usual batch
        _train("step ResNet-20 b128", "resnet20", 128, 32, "nearest"),
        # a batch and an image size that divide nothing: 89, 45, 23, 12 and 6 pixel rows
        _train("ragged step ResNet-18 b13", "resnet18", 13, 178, "nearest"),
        # the benchmark's workload
        _train("step ResNet-18 b64", "resnet18", 64, 224, "nearest"),
        # 1x1 filters, a strided 3x3 and a projection: the block that opens a stage of ResNet-50
        {"name": "bottleneck ResNet-50 b32", "kind": "layers", "net": "resnet50", "block": "layer3.0", "batch": 32, "passes": "all",
         "graph": True},
        # the single 3x3 layer, called directly: host time and launch latency
        _layer("single layer", 8, 32, 32, 16, 16, 3, 1, "all", False),
        # forward of a large layer with its shortcut: tensors beyond the L2 cache
        _layer("forward 64ch 56x56 b512", 512, 56, 56, 64, 64, 3, 1, "forward", True),
        # backward of a strided layer whose sizes are odd and whose channels are no powers of two
        _layer("ragged strided backward", 5, 37, 29, 48, 80, 3, 2, "backward", False),
        # backward of the widest layers: long reductions over small images
        _layer("backward 512ch 7x7 b64", 64, 7, 7, 512, 512, 3, 1, "backward", True),
        # scale quantizer on a tensor of activation size, one element over
        {"name": "SQ of 12.8 M floats", "kind": "quantize", "mode": "SQ", "n": 64 * 56 * 56 * 64 + 1},
        # weight update of a whole network
        {"name": "update ResNet-34", "kind": "update", "net": "resnet34", "rounding": "stochastic"},
    ]


def _train(name, net, batch, image, rounding):
    return {"name": name, "kind": "train", "net": net, "batch": batch, "image": image, "rounding": rounding}


def _layer(name, n, h, w, c_in, c_out, k, stride, passes, residual):
    return {"name": name, "kind": "layers", "n": n, "h": h, "w": w, "c_in": c_in, "c_out": c_out, "k": k, "stride": stride,
            "passes": passes, "residual": residual, "graph": False}


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choices(["train", "block", "layers", "quantize", "update"], [5, 1, 4, 1, 1])[0]
    rounding = rng.choice(["nearest", "stochastic"])
    if kind == "train":
        if rng.random() < 0.4:
            c = _train("", "resnet20", log_int(1, 128), rng.randint(24, 32), rounding)
        else:
            image = 2 * rng.randint(48, 112)   # a 7x7 first layer on 8 channels takes even widths
            c = _train("", "resnet18", log_int(1, min(64, MOST_PIXELS // image ** 2)), image, rounding)
    elif kind == "block":
        stage = rng.randint(1, 4)
        c = {"kind": "layers", "net": "resnet50", "block": "layer%d.%d" % (stage, rng.randint(0, 2)), "batch": log_int(1, 32),
             "passes": "all", "graph": True}
    elif kind == "layers":
        while True:
            h = log_int(5, 64)
            c = _layer("", log_int(1, 512), h, max(5, h + rng.randint(-h // 4, h // 4)), 16 * log_int(1, 32), 16 * log_int(1, 32),
                       rng.choice([1, 3, 3, 3]), rng.choice([1, 1, 1, 2]), rng.choice(["forward", "backward", "all"]), rng.random() < 0.5)
            l, = _geometry(c)
            if l.macs <= MOST_MACS and l.n * l.h * l.w * max(l.c_in, l.c_out) <= 512 * 56 * 56 * 64:
                break
    elif kind == "quantize":
        c = {"kind": "quantize", "mode": rng.choice(["Q", "CQ", "SQ"]), "n": log_int(2304, 64 * 56 * 56 * 64)}
    else:
        c = {"kind": "update", "net": rng.choice(["resnet20", "resnet18", "resnet34"]), "rounding": rounding}
    c.pop("name", None)
    return c


def _workload(case):
    return {"resnet18": workloads.resnet18, "resnet20": workloads.resnet20, "resnet34": workloads.resnet34,
            "resnet50": workloads.resnet50}[case["net"]](case.get("batch", 1), case.get("image", 32 if case["net"] == "resnet20" else 224))


def _geometry(case):
    """The layers of a ``layers`` case."""
    if "block" in case:
        return [l for l in _workload(case).layers if l.name.startswith(case["block"] + ".")]
    c, k = case, case["k"]
    return [workloads.Layer("layer", c["n"], c["h"], c["w"], c["c_in"], c["c_out"], k, c["stride"], k // 2, c["c_in"],
                            shortcut=c["residual"], gamma_trainable=c["residual"])]


# ---------------------------------------------------------------------------------------------- states

def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    return {"train": _prepare_train, "layers": _prepare_layers, "quantize": _prepare_quantize, "update": _prepare_update}[case["kind"]](
        case, int(seed), gen)


def run(state):
    return state["run"](state)


def _prepare_train(case, seed, gen):
    wl = _workload(case)
    small = case["net"] == "resnet20"
    stochastic = case["rounding"] == "stochastic"
    step = chain.ChainedStep(wl, eoq.eoq_create(0), DEV, seed=seed, lr_mant=1 if stochastic else 3, lr_exp=-8 if stochastic else -4,
                             classes=10 if small else 1000, pool=None if small else (3, 2, 1), round_mode=ROUND[case["rounding"]])
    step.image.copy_(torch.randn(step.image.shape, generator=gen, device=DEV))
    step.labels.copy_(torch.randint(0, step.classes, step.labels.shape, generator=gen, device=DEV, dtype=torch.int32))
    step.capture()
    outputs = {"weights": [u.w for u in step.units], "scalars": [u.scal for u in step.units], "head": [step.W, step.bias],
               "logits": step.logits, "loss": step.loss}
    return {"run": _run_train, "step": step, "outputs": outputs}


def _run_train(s):
    s["step"].replay()
    return s["outputs"]


class _Unit:
    """Tensors of one convolution unit: post-ReLU codes as input, rounded-normal error codes, Kaiming weights."""

    def __init__(self, l, gen):
        def codes(shape, std, relu=False):
            v = torch.randn(shape, generator=gen, device=DEV) * std
            return (v.clamp_(min=0) if relu else v).round_().clamp_(-127, 127).to(torch.int8)

        def ints(*v):
            return torch.tensor(v, dtype=torch.int32, device=DEV)

        def empty(shape, dtype=torch.int8):
            return torch.zeros(shape, dtype=dtype, device=DEV)

        self.l = l
        self.desc = eoq.conv_desc(l.n, l.h, l.w, l.c_in, l.c_out, l.k, l.k, l.stride, l.pad)
        out = (l.n, l.ho, l.wo, l.c_out)
        self.n_out = math.prod(out)
        self.x = codes((l.n, l.h, l.w, l.c_in), 48.0, relu=True)
        self.w = codes((l.c_out, l.k, l.k, l.c_in), 128.0 * math.sqrt(2.0 / (l.c_in * l.k * l.k)))
        self.scal = ints(-2, 118 if l.gamma_trainable else 128, 3 if l.relu else 0)   # b1, gamma, b2
        self.b1, self.gamma = self.scal[0:1], self.scal[1:2]
        self.shortcut = codes(out, 48.0, relu=True) if l.shortcut else None
        self.e0, self.e0_exp = codes(out, 32.0), ints(-12)
        self.x5, self.e3, self.e4 = empty(out), empty(out), empty((l.n, l.h, l.w, l.c_in))
        self.x2 = empty(out, torch.int16) if l.gamma_trainable else None
        self.mask = empty((self.n_out + 7) // 8, torch.uint8) if l.relu else None
        self.e3_exp, self.e4_exp, self.g_exp = ints(0), ints(0), ints(0)
        self.sum_e1, self.sum_e1x2, self.sum_e4 = (empty(1, torch.int64) for _ in range(3))
        self.g = empty(self.w.shape)
        self.prep = empty(max(256, eoq.eoq_weight_prep_size(self.desc)), torch.uint8)


def _prepare_layers(case, seed, gen):
    h = eoq.eoq_create(0)
    units = [_Unit(l, gen) for l in _geometry(case)]
    need = max(eoq.eoq_workspace_size(u.desc, p) for u in units for p in (eoq.EOQ_PASS_FWD, eoq.EOQ_PASS_DGRAD, eoq.EOQ_PASS_WGRAD))
    s = {"run": _run_layers, "h": h, "units": units, "passes": case["passes"], "ws": torch.empty(need + 256, dtype=torch.uint8, device=DEV),
         "step": torch.zeros(1, dtype=torch.int64, device=DEV)}
    eoq.eoq_weight_prep(h, [u.desc for u in units], [u.w for u in units], [u.prep for u in units])
    _forward(s)   # what a backward pass finds: the mask and x2 of its forward
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _calls(s)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"], stream=side):
            _calls(s)
    out = {}
    for i, u in enumerate(units):
        if case["passes"] != "backward":
            out["fwd%d" % i] = [u.x5, u.x2, u.mask]
        if case["passes"] != "forward":
            out["bwd%d" % i] = [u.e3, u.e3_exp, u.sum_e1, u.sum_e1x2, u.e4, u.e4_exp, u.sum_e4, u.g, u.g_exp]
        if case["passes"] == "all":
            out["w%d" % i] = u.w
    s["outputs"] = out
    return s


def _forward(s):
    for u in s["units"]:
        eoq.eoq_conv_fwd_dev(s["h"], u.desc, u.x, None, u.scal, u.w, u.prep, u.shortcut, u.l.relu, u.x5, u.x2, u.mask)


def _backward(s):
    for u in reversed(s["units"]):
        eoq.eoq_err_prescale_dev(s["h"], u.e0, u.e0_exp, u.mask, u.x2, u.n_out, u.gamma, u.e3, u.e3_exp, u.sum_e1,
                                 u.sum_e1x2 if u.x2 is not None else None)
        eoq.eoq_conv_dgrad(s["h"], u.desc, u.e3, u.e3_exp, u.w, u.e4, u.e4_exp, u.sum_e4, None, s["ws"])
        eoq.eoq_conv_wgrad_dev(s["h"], u.desc, u.e3, u.e3_exp, u.x, u.b1, u.g, u.g_exp, s["ws"])


def _calls(s):
    if s["passes"] != "backward":
        _forward(s)
    if s["passes"] != "forward":
        _backward(s)
    if s["passes"] == "all":
        us = s["units"]
        eoq.eoq_update_dev(s["h"], [u.w for u in us], [u.g for u in us], [u.g_exp for u in us], 1, -6, eoq.EOQ_ROUND_RNE, 1, s["step"])
        eoq.eoq_weight_prep(s["h"], [u.desc for u in us], [u.w for u in us], [u.prep for u in us])


def _run_layers(s):
    if "graph" in s:
        s["graph"].replay()
    else:
        _calls(s)
    return s["outputs"]


def _prepare_quantize(case, seed, gen):
    n = case["n"]
    src = torch.randn(n, generator=gen, device=DEV) * (0.05 if case["mode"] == "CQ" else 1.0)   # weights, or activations
    return {"run": _run_quantize, "h": eoq.eoq_create(0), "mode": QMODE[case["mode"]], "src": src, "n": n,
            "dst": torch.zeros(n, dtype=torch.int16 if case["mode"] == "Q" else torch.int8, device=DEV),
            "exp": torch.zeros(1, dtype=torch.int32, device=DEV)}


def _run_quantize(s):
    eoq.eoq_quantize(s["h"], s["mode"], s["src"], True, None, s["n"], s["dst"], s["exp"])
    return [s["dst"], s["exp"]]


def _prepare_update(case, seed, gen):
    sizes = [l.weight_elems for l in _workload(case).layers]

    def codes(n, std):
        return (torch.randn(n, generator=gen, device=DEV) * std).round_().clamp_(-127, 127).to(torch.int8)

    return {"run": _run_update, "h": eoq.eoq_create(0), "w": [codes(n, 3.0) for n in sizes], "g": [codes(n, 24.0) for n in sizes],
            "g_exp": [torch.tensor([-8 - i % 3], dtype=torch.int32, device=DEV) for i in range(len(sizes))], "seed": seed,
            "round": ROUND[case["rounding"]], "step": torch.zeros(1, dtype=torch.int64, device=DEV)}


def _run_update(s):
    eoq.eoq_update_dev(s["h"], s["w"], s["g"], s["g_exp"], 1, -6, s["round"], s["seed"], s["step"])
    return [s["w"], s["step"]]


# ---------------------------------------------------------------------------------------------- work and tolerance

def work(case):
    """Inputs read once and outputs written once; a training step also keeps every unit's output from forward to backward."""
    if case["kind"] == "quantize":
        return {"bytes": case["n"] * (4 + (2 if case["mode"] == "Q" else 1)), "flops": 0}
    if case["kind"] == "update":
        return {"bytes": 3 * sum(l.weight_elems for l in _workload(case).layers), "flops": 0}
    if case["kind"] == "train":
        wl = _workload(case)
        first, last = wl.layers[0], wl.layers[-1]
        head = (10 if case["net"] == "resnet20" else 1000) * last.c_out * 4
        kept = sum(2 * l.n * l.ho * l.wo * l.c_out for l in wl.layers)
        return {"bytes": first.n * first.h * first.w * 12 + 2 * sum(l.weight_elems for l in wl.layers) + 2 * head + kept,
                "flops": wl.total_ops}
    total = {"bytes": 0, "flops": 0}
    for l in _geometry(case):
        n_in, n_out, w = l.n * l.h * l.w * l.c_in, l.n * l.ho * l.wo * l.c_out, l.weight_elems
        mask, x2 = (n_out // 8 if l.relu else 0), (2 * n_out if l.gamma_trainable else 0)
        if case["passes"] != "backward":
            total["bytes"] += n_in + w + n_out + (n_out if l.shortcut else 0) + mask + x2
            total["flops"] += 2 * l.macs
        if case["passes"] != "forward":
            # e0, mask, x2 -> e3; e3, w -> e4; e3, x -> g
            total["bytes"] += n_out + mask + x2 + n_out + w + n_in + n_in + w
            total["flops"] += 4 * l.macs
        if case["passes"] == "all":
            total["bytes"] += w
    return total


def tolerance(case):
    # codes, exponents and sums are whole numbers; the float head is defined operation by operation and reproducible bit for bit
    return "exact"
