"""The work that programs have this library do, as measured cases over the real range of its public entry points.

Five kinds of case:
  block      one training step of one Conv-BN-SiLU block (CbsBlock.step: forward, data gradient, weight gradient),
  eval       the evaluation-mode forward of every layer of the detector (nb_conv_bn_silu_infer),
  train      one training iteration minus the loss of the chained detector: GraphRunner.forward, .backward with the weight
             gradients on a second stream, and the fused clip + SGD-Nesterov update of every parameter,
  optimizer  the optimiser step alone, with the dynamic loss scaler and 16-bit working copies,
  host       one training step of a block whose tensors live in pinned host memory (nb_conv_bn_silu_step_host).

Layer shapes are those of the benchmark configurations and of the random-shape tests; inputs follow
workloads.make_inputs (images U[0,1), activations and gradients N(0,1), Kaiming-uniform filters), drawn on the device.
"""
import math
import random

import torch

from paper_2609_10632_b200 import binding as nb
from paper_2609_10632_b200 import workloads as wl
from paper_2609_10632_b200.block import CbsBlock
from paper_2609_10632_b200.detector import GraphRunner

MODES = {"bf16": nb.NB_MODE_BF16_TC, "f16": nb.NB_MODE_F16_TC, "f32": nb.NB_MODE_F32_REF}
DTYPES = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}
HYPER = dict(lr=[1e-4, 1e-4, 1e-4], weight_decay=[3.75e-4, 0.0, 0.0], momentum=0.937, max_norm=10.0)


# ------------------------------------------------------------------------------------------------ cases
def _block(name, n, h, w, c_in, c_out, k, stride, mode, kind="block"):
    return {"name": name, "kind": kind, "n": n, "h": h, "w": w, "c_in": c_in, "c_out": c_out, "k": k, "stride": stride, "mode": mode}


def listed():
    return [
        # benchmark configuration 1, in fp32: the smallest call, what a gradient check or a first experiment runs
        _block("block tiny f32", 2, 32, 32, 16, 32, 3, 1, "f32"),
        # an ordinary layer in the fp32 mode that 16-bit runs are checked against
        _block("block 40x40 f32", 2, 40, 40, 64, 64, 3, 1, "f32"),
        # benchmark configuration 2: the first layer on a batch of images
        _block("block first layer", 16, 640, 640, 3, 48, 3, 2, "bf16"),
        # benchmark configuration 3: a bottleneck at high resolution, tensors larger than L2
        _block("block 160x160", 16, 160, 160, 96, 96, 3, 1, "bf16"),
        # benchmark configuration 4: a pointwise layer at low resolution (here in the fp16 mode) and a downsampling layer
        _block("block 1x1 f16", 16, 40, 40, 384, 384, 1, 1, "f16"),
        _block("block down", 16, 80, 80, 192, 384, 3, 2, "bf16"),
        # a narrower network on images that are not square: odd extents, channel counts that are multiples of 8 only
        _block("block ragged", 3, 53, 75, 72, 136, 3, 1, "bf16"),
        # serving one image
        {"name": "eval one image", "kind": "eval", "batch": 1, "image": 640, "mode": "bf16"},
        # a training iteration at the recipe's batch size, and a small one (debugging, fine-tuning on small images)
        {"name": "train batch 16", "kind": "train", "batch": 16, "image": 640},
        {"name": "train small", "kind": "train", "batch": 2, "image": 320},
        # the optimiser step over the detector's 243 tensors with fp16 working copies and loss scaling
        {"name": "optimizer detector", "kind": "optimizer", "tensors": 243, "numel": 0, "layout": 0, "copy": "f16"},
        # a caller whose data lives in host memory
        _block("host 1x1", 16, 40, 40, 384, 384, 1, 1, "bf16", kind="host"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_block(rng, kind, most):
    """A block with at most `most` multiply-add operations x 2 in its three convolutions."""
    while True:
        mode = rng.choice(["bf16", "bf16", "bf16", "f16", "f32"]) if kind == "block" else rng.choice(["bf16", "f16"])
        if rng.random() < 0.1:  # a first layer
            n, c_in, c_out, k, stride = _log(rng, 1, 16), 3, 16 * rng.randint(1, 5), 3, 2
            h, w = 2 * _log(rng, 32, 320), 2 * _log(rng, 32, 320)
        else:
            k, stride = rng.choice([(1, 1), (3, 1), (3, 1), (3, 2)])
            n, h, w = _log(rng, 1, 16), _log(rng, 7, 160), _log(rng, 7, 160)
            c_in, c_out = 8 * _log(rng, 2, 72), 8 * _log(rng, 2, 72)
        c = {"kind": kind, "n": n, "h": h, "w": w, "c_in": c_in, "c_out": c_out, "k": k, "stride": stride, "mode": mode}
        s = _shape(c)
        limit = most / 8 if mode == "f32" else most
        if s.m >= 256 and 3 * s.gemm_flops <= limit and n * h * w * c_in <= 1 << 26 and s.m * c_out <= 1 << 26:
            return c


def draw(rng):
    kind = rng.choices(["block", "eval", "train", "optimizer", "host"], [6, 1, 1, 1, 1])[0]
    if kind == "block":
        return _draw_block(rng, kind, 3e11)
    if kind == "host":
        return _draw_block(rng, kind, 1e11)
    if kind == "eval":
        return {"kind": kind, "batch": _log(rng, 1, 16), "image": 32 * _log(rng, 5, 20), "mode": rng.choice(["bf16", "f16"])}
    if kind == "train":
        return {"kind": kind, "batch": _log(rng, 1, 12), "image": 32 * _log(rng, 5, 20)}
    return {"kind": kind, "tensors": _log(rng, 10, 400), "numel": _log(rng, 10_000, 30_000_000), "layout": rng.randrange(1 << 20),
            "copy": rng.choice(["bf16", "f16"])}


def _shape(c):
    return wl.ConvShape("layer", c["n"], c["h"], c["w"], c["c_in"], c["c_out"], c["k"], c["stride"], c["c_in"] == 3)


def _optimizer_tensors(c):
    """[(numel, group, has a working copy)]: the detector's list, or a network's with `numel` elements in `tensors` tensors."""
    if c["numel"] == 0:
        return [(n, group, group == 0) for _, n, group in wl.detector_parameter_tensors()]
    rng = random.Random(c["layout"])
    share = [math.exp(rng.uniform(0.0, 7.0)) for _ in range(c["tensors"])]
    out = []
    for i, f in enumerate(share):
        group = rng.choice([0, 1, 2])
        out.append((max(1, int(f / sum(share) * c["numel"])), group, group == 0))
    return out


# ------------------------------------------------------------------------------------------------ inputs
def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return gen


def _flat(sizes, dtype):
    """One zeroed buffer and a view of it per size, each on a 16-byte boundary."""
    at, total = [], 0
    for n in sizes:
        at.append(total)
        total += -(-n // 8) * 8
    buf = torch.zeros(total, dtype=dtype, device="cuda")
    return buf, [buf[o:o + n] for o, n in zip(at, sizes)]


def _fill_block(blk, gen):
    s = blk.shape
    rand = lambda t: torch.rand(t.shape, generator=gen, device="cuda")
    randn = lambda t: torch.randn(t.shape, generator=gen, device="cuda")
    blk.x.copy_(rand(blk.x) if s.image_input else randn(blk.x))
    blk.w.copy_((2 * rand(blk.w) - 1) / math.sqrt(s.c_in * s.k * s.k))
    blk.gamma.copy_(0.5 + rand(blk.gamma))
    blk.beta.copy_(0.1 * randn(blk.beta))
    blk.g.copy_(randn(blk.g))


def _prepare_block(c, seed):
    blk = CbsBlock(_shape(c), mode=MODES[c["mode"]], running_stats=True)
    _fill_block(blk, _generator(seed))
    return {"block": blk}


def _prepare_host(c, seed):
    src = CbsBlock(_shape(c), mode=MODES[c["mode"]])
    _fill_block(src, _generator(seed))
    pinned = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    inputs = {k: pinned(getattr(src, k)).copy_(getattr(src, k)) for k in ("x", "w", "gamma", "beta", "g")}
    outputs = {k: pinned(getattr(src, k)) for k in ("a", "dx", "dw", "dgamma", "dbeta")}
    scratch = torch.empty(src.plan.step_host_scratch_bytes(), dtype=torch.uint8, device="cuda")
    return {"plan": src.plan, "in": inputs, "out": outputs, "scratch": scratch}


def _prepare_eval(c, seed):
    gen, dtype = _generator(seed), DTYPES[c["mode"]]
    layers = wl.detector_layers(c["batch"], c["image"])
    rand = lambda *sz: torch.rand(sz, generator=gen, device="cuda")
    randn = lambda *sz: torch.randn(sz, generator=gen, device="cuda")
    flat, outs = _flat([s.m * s.c_out for s in layers], dtype)
    plans = {}
    items = []
    for s, a in zip(layers, outs):
        if s.key not in plans:
            plans[s.key] = nb.Plan.for_shape(s, mode=MODES[c["mode"]])
        size = (s.n, s.h, s.w, s.c_in)
        x = (rand(*size) if s.image_input else randn(*size)).to(dtype)
        w = ((2 * rand(s.c_out, s.k, s.k, s.c_in) - 1) / math.sqrt(s.c_in * s.k * s.k)).to(dtype)
        items.append((plans[s.key], x, w, 0.5 + rand(s.c_out), 0.1 * randn(s.c_out), 0.2 * randn(s.c_out), 0.25 + 0.5 * rand(s.c_out), a))
    ws = torch.empty(max(max(p.infer_bytes for p in plans.values()), 256), dtype=torch.uint8, device="cuda")
    return {"items": items, "ws": ws, "out": flat}


def _prepare_train(c, seed):
    gen = _generator(seed)
    ops, layers, outs, plain = wl.detector_graph(c["batch"], c["image"], plain_head=True)
    runner = GraphRunner(ops, layers, outs, plain_layers=plain)
    runner.fill_parameters(seed=seed)
    for pl in runner.plain:
        pl["w"].normal_(0.0, 0.05, generator=gen)
        pl["bias"].normal_(0.0, 0.5, generator=gen)
    runner.buf["img"].uniform_(0.0, 1.0, generator=gen)
    for name in outs:
        runner.grad[name].normal_(generator=gen)
    # all gradients in one buffer, all fp32 filters in another, as data-parallel programs keep them
    wide = [(b.w, b.dw) for b in runner.blocks] + [(pl["w"], pl["dw"]) for pl in runner.plain]
    small = [t for b in runner.blocks for t in (b.dgamma, b.dbeta)] + [pl["dbias"] for pl in runner.plain]
    grads, views = _flat([dw.numel() for _, dw in wide] + [t.numel() for t in small], torch.float32)
    masters, master_views = _flat([w.numel() for w, _ in wide], torch.float32)
    momentum, momentum_views = _flat([v.numel() for v in views], torch.float32)
    v = iter(views)
    for b in runner.blocks:
        b.dw = next(v).view(b.dw.shape)
    for pl in runner.plain:
        pl["dw"] = next(v).view(pl["dw"].shape)
    for b in runner.blocks:
        b.dgamma, b.dbeta = next(v), next(v)
    for pl in runner.plain:
        pl["dbias"] = next(v)
    items = []
    for (w, _), g, p, m in zip(wide, views, master_views, momentum_views):
        p.copy_(w.reshape(-1))
        items.append((g, p, m, w, 0))
    params = [(t, group) for b in runner.blocks for t, group in ((b.gamma, 1), (b.beta, 2))] + [(pl["bias"], 2) for pl in runner.plain]
    for (p, group), g, m in zip(params, views[len(wide):], momentum_views[len(wide):]):
        items.append((g, p, m, None, group))
    sgd = nb.SgdPlan(items)
    sgd_ws = torch.empty(sgd.workspace_bytes, dtype=torch.uint8, device="cuda")
    sgd.upload(sgd_ws)
    side_ws = torch.empty(max(b.plan.bwd_bytes for b in runner.blocks), dtype=torch.uint8, device="cuda")
    return {"runner": runner, "heads": outs, "sgd": sgd, "sgd_ws": sgd_ws, "side": torch.cuda.Stream(), "side_ws": side_ws,
            "grads": grads, "masters": masters, "momentum": momentum, "keep": items}


def _prepare_optimizer(c, seed):
    gen, tensors = _generator(seed), _optimizer_tensors(c)
    grads, gv = _flat([n for n, _, _ in tensors], torch.float32)
    params, pv = _flat([n for n, _, _ in tensors], torch.float32)
    momentum, mv = _flat([n for n, _, _ in tensors], torch.float32)
    copies, cv = _flat([n for n, _, low in tensors if low], DTYPES[c["copy"]])
    scale = 65536.0
    grads.normal_(0.0, 0.02 * scale, generator=gen)
    params.normal_(0.0, 0.05, generator=gen)
    momentum.normal_(0.0, 0.01, generator=gen)
    low = iter(cv)
    plan = nb.SgdPlan([(g, p, m, next(low) if has else None, group) for g, p, m, (_, group, has) in zip(gv, pv, mv, tensors)])
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    plan.upload(ws)
    scaler = torch.zeros(4, dtype=torch.float32, device="cuda")  # nb_loss_scaler: the scale, then three integers at zero
    scaler[0] = scale
    return {"plan": plan, "ws": ws, "scaler": scaler, "norm": torch.zeros(4, device="cuda"), "grads": grads, "params": params,
            "momentum": momentum, "copies": copies}


def prepare(case, seed):
    return {"kind": case["kind"], **globals()["_prepare_" + case["kind"]](case, seed)}


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    kind = state["kind"]
    if kind == "block":
        b = state["block"]
        b.step()
        return {k: getattr(b, k) for k in ("a", "y", "mean", "invstd", "running_mean", "running_var", "dy", "dx", "dw", "dgamma", "dbeta")}
    if kind == "host":
        i, o = state["in"], state["out"]
        nb.nb_conv_bn_silu_step_host(state["plan"], i["x"], i["w"], i["gamma"], i["beta"], i["g"], o["a"], o["dx"], o["dw"], o["dgamma"],
                                     o["dbeta"], state["scratch"])
        return o
    if kind == "eval":
        for plan, x, w, gamma, beta, mean, var, a in state["items"]:
            nb.nb_conv_bn_silu_infer(plan, x, w, gamma, beta, mean, var, a, state["ws"])
        return state["out"]
    if kind == "train":
        runner, side, main = state["runner"], state["side"], torch.cuda.current_stream()
        runner.forward()
        side.wait_stream(main)
        runner.backward(wgrad_stream=side, wgrad_workspace=state["side_ws"])
        main.wait_stream(side)
        state["sgd"].step(state["sgd_ws"], first_step=False, **HYPER)
        return {"heads": [runner.buf[name] for name in state["heads"]], "image gradient": runner.grad["img"], "gradients": state["grads"],
                "filters": state["masters"], "momentum": state["momentum"]}
    state["plan"].step_scaled(state["ws"], state["scaler"], first_step=False, floor_scale=1.0, total_norm=state["norm"], **HYPER)
    return {k: state[k] for k in ("params", "momentum", "copies", "norm", "scaler")}


# ------------------------------------------------------------------------------------------------ what a pass needs
def _block_bytes(s, size):
    """x, w and g read; y, a, dy, dx (16-bit or fp32) and dw (fp32) written."""
    filters = s.c_out * s.kdim
    return size * (2 * s.n * s.h * s.w * s.c_in + filters + 4 * s.m * s.c_out) + 4 * filters


def work(case):
    kind = case["kind"]
    if kind in ("block", "host"):
        s, size = _shape(case), 4 if case["mode"] == "f32" else 2
        saved = 2 * s.m * s.c_out if kind == "host" else 0  # y and dy stay on the device: not among the call's outputs
        return {"bytes": _block_bytes(s, size) - size * saved, "flops": 3 * s.gemm_flops}
    if kind == "eval":
        layers = wl.detector_layers(case["batch"], case["image"])
        return {"bytes": sum(2 * (s.n * s.h * s.w * s.c_in + s.c_out * s.kdim + s.m * s.c_out) for s in layers), "flops": sum(s.gemm_flops for s in layers)}
    if kind == "train":
        _, layers, _, plain = wl.detector_graph(case["batch"], case["image"], plain_head=True)
        every = layers + plain
        update = 22 * sum(n for _, n, _ in wl.detector_parameter_tensors())
        return {"bytes": sum(_block_bytes(s, 2) for s in every) + update, "flops": 3 * sum(s.gemm_flops for s in every)}
    # gradient read, parameter and momentum read and written, working copy written
    return {"bytes": sum(n * (22 if low else 20) for n, _, low in _optimizer_tensors(case)), "flops": 0}


def tolerance(case):
    """A single block: the tolerances of the parity tests.  The chain is 83 layers deep with batch statistics over random
    data, in which one rounding of a 16-bit tensor grows from layer to layer (a model of 16-bit storage in exact arithmetic
    is 0.2 away from exact arithmetic at the heads), so that only results that round almost everywhere alike stay within
    a few percent.  Optimiser: fp32 sums; a working copy may round the other way."""
    if case["kind"] == "train":
        return {"rel": 3e-2, "max": 0.9}
    if case["kind"] == "optimizer":
        return {"rel": 1e-5, "max": 1e-2}
    return {"rel": 1e-5} if case["mode"] == "f32" else {"rel": 5e-3, "max": 5e-2}
