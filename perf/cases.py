"""Performance cases of the online extrapolation stage, through its public entry points.

One pass of a case is what a sampler's loop does at one step (or, for the
whole-schedule case, at every step): write a full step's branch outputs into
the history, add them to the hidden states, or predict them on a skipped step.

Fields of a case
  path      "skip"      predictions (``preds``) and/or hidden states (``hidden``) of a skipped step
            "push"      a new sample's first full step: reset, cache write
            "push_add"  the same with the hidden-state update fused
            "schedule"  a whole sampling run: every full step pushes, every skipped step predicts
  entry     how a skipped step is called: "step" (cb_extrapolate, or cb_extrapolate_gated with
            gates), "noalloc" (a caller's own history buffer) or "taylor" (caller-chosen weights)
  layout    "blocks": ``blocks`` blocks of ``branches`` tensors [batch, tokens, hidden];
            "streams": ``blocks`` double-stream blocks (two branches of ``tokens`` image and of
            ``text`` text tokens) and ``single`` blocks over both
  K         history size;  cache / feat / io / gate: storage types of the history, the pushed
            features, the outputs and hidden states, and the gates ("" = no gates)
"""
import math

import numpy as np
import torch

from paper_2608_23429_gb300 import chebboost as cb

DEV = "cuda"
TORCH = {"bf16": torch.bfloat16, "fp32": torch.float32}
CODE = {"bf16": cb.CB_BF16, "fp32": cb.CB_FP32}
SIZE = {"bf16": 2, "fp32": 4}
T_MIN, T_MAX = 0.0, 999.0
STEPS, REFRESH = 50, 4  # the DDIM-50 run with a full step every fourth


def _case(name, path, **kw):
    c = dict(name=name, path=path, entry="step", layout="blocks", blocks=28, branches=2, single=0, batch=1, tokens=256,
             text=0, hidden=1152, K=4, cache="bf16", feat="bf16", io="bf16", gate="", preds=True, hidden_states=False)
    c.update(kw)
    return c


def listed():
    return [
        # a program that hooks single blocks calls once per block: the smallest call, all latency
        _case("one_block", "skip", blocks=1, K=3),
        # the repository's tiny configuration: two fp32 blocks, small enough to stay in L2
        _case("tiny_fp32", "skip", blocks=2, cache="fp32", feat="fp32", io="fp32"),
        # an operator inside an inference engine (own history buffer) on a text stream of 77
        # tokens: short tensors whose last tile is ragged
        _case("engine_text", "skip", entry="noalloc", blocks=12, tokens=77, hidden=768, hidden_states=True),
        # odd sizes throughout: no tensor in the stacked buffers but the first is 16-byte aligned
        _case("odd_gated", "skip", blocks=8, branches=3, batch=3, tokens=333, hidden=577, K=5, gate="bf16",
              hidden_states=True),
        # a whole DDIM-50 run of a class-conditional model, one image
        _case("dit_schedule", "schedule"),
        # DiT-XL/2 256^2 as the bench states it: predictions and hidden states of a skipped step
        _case("dit256_skip", "skip", batch=8, hidden_states=True),
        # the same model's full step, un-gated branches: cache write and gated hidden states in one pass
        _case("dit256_full_gated", "push_add", batch=8, gate="bf16", hidden_states=True),
        # DiT-XL/2 512^2 with the residual stream and the gates in fp32 (mixed-precision inference),
        # where only the hidden states are wanted
        _case("dit512_fp32_stream", "skip", batch=4, tokens=1024, io="fp32", gate="fp32", preds=False,
              hidden_states=True),
        # the longest history, predictions in fp32 for a solver that works in fp32, Taylor weights
        _case("dit512_taylor_fp32", "skip", entry="taylor", batch=4, tokens=1024, K=8, io="fp32"),
        # PixArt-Sigma 1024^2: fp32 features (no autocast) into a bf16 history
        _case("pixart_push_fp32", "push", branches=3, batch=2, tokens=4096, feat="fp32"),
        # FLUX.1-dev 1024^2, the largest: predictions of a skipped step ...
        _case("flux_skip", "skip", layout="streams", blocks=19, single=38, tokens=4096, text=512, hidden=3072, K=5),
        # ... and a full step with its residual adds
        _case("flux_full", "push_add", layout="streams", blocks=19, single=38, tokens=4096, text=512, hidden=3072, K=5,
              hidden_states=True),
    ]


def draw(rng):
    """A case of the listed ranges: any path, type and K, sizes spread over their logarithm."""
    path = rng.choice(["skip"] * 6 + ["push", "push_add", "push_add", "schedule"])
    cache = rng.choice(["bf16", "bf16", "bf16", "fp32"])
    feat = rng.choice(["bf16", "bf16", "fp32"]) if cache == "bf16" else "fp32"
    io = rng.choice(["bf16", "bf16", "fp32"]) if cache == "bf16" else rng.choice(["bf16", "fp32"])
    c = _case("", path, cache=cache, feat=feat, io=io)
    c["K"] = rng.randint(1, 8) if path != "schedule" else rng.randint(2, 5)
    c["hidden"] = int(round(math.exp(rng.uniform(math.log(256), math.log(4096)))))
    if rng.random() < 0.75:
        c["hidden"] = max(8, c["hidden"] // 8 * 8)
    c["batch"] = rng.randint(1, 8)
    if rng.random() < 0.2:
        c["layout"] = "streams"
        c["blocks"], c["single"] = rng.randint(1, 19), rng.randint(0, 38)
        c["branches"], c["text"] = 2, rng.randint(20, 512)
    else:
        c["blocks"], c["branches"] = rng.randint(1, 40), rng.randint(1, 4)
    if path == "skip":
        c["entry"] = rng.choice(["step", "step", "noalloc", "taylor"])
        c["preds"] = rng.random() < 0.7
        c["hidden_states"] = not c["preds"] or rng.random() < 0.5
        if c["hidden_states"] and c["entry"] == "step" and rng.random() < 0.5:
            c["gate"] = rng.choice(["bf16", "fp32"])
    elif path == "push_add":
        c["hidden_states"] = True
        if rng.random() < 0.5:
            c["gate"] = rng.choice(["bf16", "fp32"])
    elements = math.exp(rng.uniform(math.log(6e5), math.log(3e7 if path == "schedule" else 4e8)))
    rows = c["batch"] * c["hidden"] * (2 * c["blocks"] + c["single"] if c["layout"] == "streams"
                                       else c["blocks"] * c["branches"])
    c["tokens"] = max(1, min(8192, int(elements / rows)))
    while work(c)["bytes"] > 8e9 and max(c["tokens"], c["text"]) > 1:
        c["tokens"], c["text"] = -(-c["tokens"] // 2), -(-c["text"] // 2)
    del c["name"]
    return c


# ---- shapes

def _tensors(c):
    """(layer, branch, shape, group) of every cached tensor."""
    out, g = [], 0
    for layer in range(c["blocks"]):
        if c["layout"] == "blocks":
            out += [(layer, b, (c["batch"], c["tokens"], c["hidden"]), g) for b in range(c["branches"])]
            g += 1
            continue
        for s, tokens in enumerate((c["tokens"], c["text"])):
            out += [(layer, 2 * s + b, (c["batch"], tokens, c["hidden"]), g) for b in range(2)]
            g += 1
    for k in range(c["single"]):
        out.append((c["blocks"] + k, 0, (c["batch"], c["tokens"] + c["text"], c["hidden"]), g))
        g += 1
    return out


def _group_shapes(c):
    shapes = {}
    for _, _, shape, g in _tensors(c):
        shapes[g] = shape
    return [shapes[g] for g in range(len(shapes))]


def _slot_elems(c):
    """Element offset of every tensor in a slot, and the slot's elements (each tensor on a 256-byte boundary)."""
    per, off, o = 256 // SIZE[c["cache"]], [], 0
    for _, _, shape, _ in _tensors(c):
        off.append(o)
        o += -(-math.prod(shape) // per) * per
    return off, o


def _stacks(shapes, dtype):
    """One buffer per distinct shape, and a view of it for every entry, as a program stacks what it keeps."""
    count = {}
    for s in shapes:
        count[s] = count.get(s, 0) + 1
    bufs = {s: torch.empty((n, *s), dtype=dtype, device=DEV) for s, n in count.items()}
    used, views = dict.fromkeys(count, 0), []
    for s in shapes:
        views.append(bufs[s][used[s]])
        used[s] += 1
    return list(bufs.values()), views


# ---- times and inputs

def _times(c):
    """Times of the full steps that are pushed, and of the skipped step that is timed."""
    step = (T_MAX - T_MIN) / (STEPS - 1)
    nodes = [T_MAX - step * REFRESH * j for j in range(c["K"])]
    return nodes, nodes[-1] - 2 * step


def _run_times(c):
    """The whole run's steps as (time, index of the full step, or None where it is skipped)."""
    out, full = [], 0
    for s in range(STEPS):
        t = T_MAX * (1.0 - s / (STEPS - 1))
        if s % REFRESH == 0 or full < c["K"]:
            out.append((t, full))
            full += 1
        else:
            out.append((t, None))
    return out, full


def _generator(seed, *at):
    g = torch.Generator(device=DEV)
    h = int(seed) + 1
    for p in at:
        h = (h * 1000003 + p + 7) % (1 << 62)
    g.manual_seed(h)
    return g


def _features(c, seed, i, shape, times):
    """Branch output i at each time: a smooth trajectory in t with noise, in the pushed type."""
    g = _generator(seed, 1, i)
    c0, c1, c2 = (torch.randn(shape, generator=g, device=DEV) for _ in range(3))
    got = []
    for t in times:
        x = 2.0 * (t - T_MIN) / (T_MAX - T_MIN) - 1.0
        f = torch.randn(shape, generator=g, device=DEV).mul_(0.1)
        f.add_(c0).add_(c1, alpha=x / 4).add_(c2, alpha=(2 * x * x - 1) / 9)
        got.append(f.to(TORCH[c["feat"]]))
    return got


def _hidden_values(c, seed, k, shape):
    return torch.randn(shape, generator=_generator(seed, 2, k), device=DEV).to(TORCH[c["io"]])


def _gate_values(c, seed, i, shape):
    g = torch.randn((shape[0], shape[2]), generator=_generator(seed, 3, i), device=DEV).mul_(0.5)
    return g.to(TORCH[c["gate"]])


def prepare(case, seed):
    c = dict(case)
    tensors = _tensors(c)
    shapes = [t[2] for t in tensors]
    nodes, target = _times(c)
    s = {"c": c, "nodes": nodes, "target": target}
    if c["path"] == "schedule":
        steps, n_full = _run_times(c)
        s["steps"] = steps
        times = [t for t, k in steps if k is not None]
    else:
        times = nodes if c["path"] == "skip" else nodes[:1]
    plan_nodes = times if c["path"] == "schedule" else nodes
    plan = cb.cb_plan_create(plan_nodes, c["K"], [(la, b, math.prod(sh), g) for la, b, sh, g in tensors],
                             CODE[c["cache"]], T_MIN, T_MAX)
    s["plan"] = plan
    cb.cb_plan_set_shapes(plan, shapes)
    s["arena"] = torch.zeros(cb.cb_plan_cache_bytes(plan), dtype=torch.uint8, device=DEV)
    cb.cb_plan_bind_cache(plan, s["arena"], s["arena"].numel())
    feats = [[] for _ in times]
    for i, sh in enumerate(shapes):
        for j, f in enumerate(_features(c, seed, i, sh, times)):
            feats[j].append(f)
    if c["path"] == "skip":
        for t, f in zip(nodes, feats):
            cb.cb_cache_push(plan, f, CODE[c["feat"]], t)
        if c["entry"] == "noalloc":
            s["slot_t"] = np.array(nodes)
            s["hist_bytes"] = s["arena"].numel() - cb.CB_STATUS_BYTES
            s["status"] = torch.zeros(1, dtype=torch.int32).pin_memory()
    else:
        s["feats"] = feats
    # buffers that outlive a step: their pointer arrays are built once
    if c["path"] in ("skip", "schedule") and c["preds"]:
        s["preds"], views = _stacks(shapes, TORCH[c["io"]])
        s["preds_at"] = cb.ptr_array(views)
    if c["hidden_states"]:
        s["x"], views = _stacks(_group_shapes(c), TORCH[c["io"]])
        for k, v in enumerate(views):
            v.copy_(_hidden_values(c, seed, k, v.shape))
        s["x_at"] = cb.ptr_array(views)
    if c["gate"]:
        s["gates"], views = _stacks([(sh[0], sh[2]) for sh in shapes], TORCH[c["gate"]])
        for i, v in enumerate(views):
            v.copy_(_gate_values(c, seed, i, shapes[i]))
        s["gates_at"] = cb.ptr_array(views)
    return s


def _slots(s, n):
    """The first n slots of the history, in its type."""
    _, elems = _slot_elems(s["c"])
    raw = s["arena"][: n * elems * SIZE[s["c"]["cache"]]]
    return raw.view(TORCH[s["c"]["cache"]]).view(n, elems)


def run(state):
    s = state
    c, plan = s["c"], s["plan"]
    preds, x = s.get("preds_at"), s.get("x_at")
    io, feat = CODE[c["io"]], CODE[c["feat"]]
    if c["path"] == "skip":
        if c["gate"]:
            cb.cb_extrapolate_gated(plan, s["target"], preds, io, x, io, s["gates_at"], CODE[c["gate"]])
        elif c["entry"] == "noalloc":
            cb.cb_extrapolate_noalloc(plan, s["arena"], s["hist_bytes"], s["slot_t"], 0, s["target"], preds, io, x, io,
                                      status=s["status"])
        elif c["entry"] == "taylor":
            w = cb.cb_taylor_weights(s["nodes"], s["target"])
            cb.cb_extrapolate_weights(plan, w, preds, io, x, io)
        else:
            cb.cb_extrapolate(plan, s["target"], preds, io, x, io)
        return {k: s[k] for k in ("preds", "x") if k in s}
    cb.cb_plan_reset(plan)
    if c["path"] == "push":
        cb.cb_cache_push(plan, s["feats"][0], feat, s["nodes"][0])
        return {"slot": _slots(s, 1)}
    if c["path"] == "push_add":
        gates = s.get("gates_at")
        cb.cb_cache_push_residual(plan, s["feats"][0], feat, s["nodes"][0], x, io, gates,
                                  CODE[c["gate"]] if c["gate"] else cb.CB_BF16)
        return {"slot": _slots(s, 1), "x": s["x"]}
    for t, k in s["steps"]:
        if k is not None:
            cb.cb_cache_push(plan, s["feats"][k], feat, t)
        else:
            cb.cb_extrapolate(plan, t, preds, io)
    return {"slots": _slots(s, c["K"]), "preds": s["preds"]}


def work(case):
    c = case
    n = sum(math.prod(t[2]) for t in _tensors(c))
    cache, feat, io = SIZE[c["cache"]], SIZE[c["feat"]], SIZE[c["io"]]
    x = 2 * io * sum(math.prod(sh) for sh in _group_shapes(c)) if c["hidden_states"] else 0
    gates = SIZE[c["gate"]] * sum(t[2][0] * t[2][2] for t in _tensors(c)) if c["gate"] else 0
    if c["path"] == "skip":
        return {"bytes": n * (c["K"] * cache + (io if c["preds"] else 0)) + x + gates, "flops": 2 * c["K"] * n}
    if c["path"] == "push":
        return {"bytes": n * (feat + cache), "flops": 0}
    if c["path"] == "push_add":
        return {"bytes": n * (feat + cache) + x + gates, "flops": 2 * n}
    steps, full = _run_times(c)
    skipped = len(steps) - full
    return {"bytes": n * (full * (feat + cache) + skipped * (c["K"] * cache + io)), "flops": 2 * c["K"] * n * skipped}


def tolerance(case):
    c = case
    if c["path"] == "push":
        return "exact"  # a copy or one rounding to nearest
    if c["io"] == "fp32" and (c["cache"] == "fp32" or c["path"] == "skip"):
        return {"rel": 2e-7, "max": 2e-6}  # one rounding of a compensated sum: 3e-8 seen against 64 bits
    return {"rel": 7e-3, "max": 3e-2}  # one rounding to bf16: 1.7e-3 seen against 64 bits


# ---- the same in 64 bits

def _lagrange(nodes, t):
    w = []
    for j, a in enumerate(nodes):
        p = 1.0
        for k, b in enumerate(nodes):
            if k != j:
                p *= (t - b) / (a - b)
        w.append(p)
    return w


def _taylor(nodes, t):
    """sum_i theta^i / i! nabla^i on equispaced nodes, oldest first."""
    n = len(nodes)
    theta = (t - nodes[-1]) / (nodes[-1] - nodes[-2]) if n > 1 else 0.0
    w = [0.0] * n
    for i in range(n):
        for k in range(i + 1):
            w[n - 1 - k] += theta ** i / math.factorial(i) * math.comb(i, k) * (-1) ** k
    return w


def exact(case, seed):
    c = dict(case)
    tensors = _tensors(c)
    shapes = [t[2] for t in tensors]
    kept = TORCH[c["cache"]]
    nodes, target = _times(c)
    off, elems = _slot_elems(c)
    got = {}

    def stacked(shs):
        return _stacks(shs, torch.float64)

    if c["path"] == "schedule":
        steps, full = _run_times(c)
        times = [t for t, k in steps if k is not None]
        last = max(i for i, (_, k) in enumerate(steps) if k is None)
        held = [k for _, k in steps[:last] if k is not None][-c["K"]:]
        w = _lagrange([times[k] for k in held], steps[last][0])
        got["slots"] = torch.zeros((c["K"], elems), dtype=torch.float64, device=DEV)
        got["preds"], views = stacked(shapes)
        for i, sh in enumerate(shapes):
            f = _features(c, seed, i, sh, times)
            views[i].copy_(sum(wj * f[k].to(kept).double() for wj, k in zip(w, held)))
            for k in range(full):
                got["slots"][k % c["K"], off[i]: off[i] + math.prod(sh)] = f[k].double().reshape(-1)
        return got
    if c["path"] in ("push", "push_add"):
        got["slot"] = torch.zeros((1, elems), dtype=torch.float64, device=DEV)
    w = None
    if c["path"] == "skip":
        w = _taylor(nodes, target) if c["entry"] == "taylor" else _lagrange(nodes, target)
    out = x = None
    if c["path"] == "skip" and c["preds"]:
        got["preds"], out = stacked(shapes)
    if c["hidden_states"]:
        got["x"], x = stacked(_group_shapes(c))
        for k, v in enumerate(x):
            v.copy_(_hidden_values(c, seed, k, v.shape))
    for i, (_, _, sh, g) in enumerate(tensors):
        f = _features(c, seed, i, sh, nodes if c["path"] == "skip" else nodes[:1])
        if w is None:
            p = f[0].double()
            got["slot"][0, off[i]: off[i] + math.prod(sh)] = p.reshape(-1)
        else:
            p = torch.zeros(sh, dtype=torch.float64, device=DEV)
            for wj, fj in zip(w, f):
                p.add_(fj.to(kept).double(), alpha=wj)
        if out is not None:
            out[i].copy_(p)
        if x is not None:
            x[g].add_(p * _gate_values(c, seed, i, sh).double()[:, None, :] if c["gate"] else p)
    return got
