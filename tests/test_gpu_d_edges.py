"""Tiles and items at the edges of the bulk kernel's paths (GPU): ragged last
tiles around every tile size, outputs, hidden states and gates off the 16-byte
grid (alone and beside aligned items), and compensated sums at the ends of the
number range."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2608_23429_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cb():
    from paper_2608_23429_gb300 import chebboost
    return chebboost


@pytest.fixture(scope="module")
def H():
    import gpu_harness
    return gpu_harness


def _workload(K, cache):
    """Lone tensors of one element around the tile sizes 2048, 2816, 4096 and
    4864, and groups of odd and even channel counts."""
    T = workloads.TensorSpec
    tensors = [T(0, b, (2, 37, 77), 0) for b in range(3)] + [T(1, b, (3, 41, 136), 1) for b in range(2)]
    tensors += [T(2, 0, (1, 1, 1), 2), T(3, 0, (2, 2816, 1), 3)]
    tensors += [T(4 + i, 0, (1, 1, n), -1)
                for i, n in enumerate([7, 2047, 2049, 2815, 2816, 4095, 4097, 4863, 4864, 9733])]
    return workloads.Workload(name="edges", tensors=tensors, K=K, cache_dtype=cache, T=0, r=0, t_min=0.0, t_max=999.0,
                              timesteps=[], degree=6, noise=0.1, seed=77)


def _shifted(shape, dtype, off):
    """A view `off` elements into its buffer, and the buffer (filled with ones)."""
    n = int(np.prod(shape))
    buf = torch.ones(n + off + 9, dtype=dtype, device="cuda")
    return buf[off:off + n].view(shape), buf


@pytest.mark.parametrize("shift", ["none", "some", "all"])
@pytest.mark.parametrize("K,cache,io", [(1, "bf16", "fp32"), (2, "bf16", "bf16"), (2, "fp32", "fp32"),
                                        (3, "bf16", "fp32"), (4, "fp32", "bf16"), (5, "bf16", "bf16"),
                                        (8, "bf16", "fp32"), (8, "fp32", "fp32")])
def test_ragged_tiles_and_off_grid_items(cb, H, K, cache, io, shift):
    w = _workload(K, cache)
    nodes = [990.0 - 37.0 * k for k in range(K)]
    walk = H.Walk(w, node_t=nodes)
    cb.cb_plan_set_shapes(walk.plan, [s.shape for s in w.tensors])
    for k, t in enumerate(nodes):
        walk.push(t, k)
    dt, target = H.TORCH[io], nodes[-1] - 20.0
    gen = torch.Generator(device="cuda").manual_seed(5)
    gates = [(0.5 * torch.randn(s.shape[0], s.shape[2], generator=gen, device="cuda")).to(dt) if i % 3 != 1 else None
             for i, s in enumerate(w.tensors)]
    for gated in (False, True):
        off = [0 if shift == "none" or (shift == "some" and i % 2) else 1 + i % 7 for i in range(len(w.tensors))]
        outs, bufs = zip(*[_shifted(s.shape, dt, o) for s, o in zip(w.tensors, off)])
        resid, rbufs, rh = [], [], []
        for g in range(walk.n_groups):
            x, b = _shifted(w.group_shape(g), dt, off[g])
            x.copy_(workloads.hidden_state(w, g, "cuda", dt, salt=9))
            resid.append(x)
            rbufs.append(b)
            rh.append(H.host(x))
        if gated:
            cb.cb_extrapolate_gated(walk.plan, target, outs, H.CB[io], resid, H.CB[io], gates, H.CB[io])
        else:
            cb.cb_extrapolate(walk.plan, target, outs, H.CB[io], resid, H.CB[io])
        torch.cuda.synchronize()
        assert cb.cb_plan_device_status(walk.plan) == 0
        G = [None if g is None else H.expand_gate(g, s.shape) for g, s in zip(gates, w.tensors)] if gated else None
        so, sr, _ = walk.expected_and_compare(target, outs, resid, rh, out_dtype=io, resid_dtype=io, G=G)
        assert so["bad"] == 0 and sr["bad"] == 0, (gated, so, sr)
        for buf, o, s in list(zip(bufs, off, w.tensors)) + [(b, off[g], next(t for t in w.tensors if t.group == g))
                                                           for g, b in enumerate(rbufs)]:
            assert torch.all(buf[:o] == 1) and torch.all(buf[o + s.numel:] == 1)  # nothing beside the tensor
    walk.close()


@pytest.mark.parametrize("kernel", ["bulk", "direct"])
@pytest.mark.parametrize("cache", ["bf16", "fp32"])
@pytest.mark.parametrize("n", [9728, 1234])
def test_compensated_sums_at_the_ends_of_the_range(cb, H, cache, kernel, n):
    """Features up to the largest finite value, where the sum's anchor would
    overflow, and infinities and NaN: the newest entry alone (weights 0, 0, 1)
    comes back exactly, and only elements that hold no number give none."""
    w = workloads.Workload(name="range", tensors=[workloads.TensorSpec(0, 0, (1, 1, n), 0)], K=3, cache_dtype=cache, T=0,
                           r=0, t_min=0.0, t_max=999.0, timesteps=[], degree=3, noise=0.1, seed=3)
    walk = H.Walk(w, node_t=[900.0, 800.0, 700.0], kernel=kernel)
    dt = H.TORCH[cache]
    feats = [workloads.trajectory(w, 0, t, k, "cuda", out_dtype=dt) for k, t in enumerate(walk.node_t)]
    big, flat = float(torch.finfo(dt).max), feats[2].reshape(-1)
    for i, v in enumerate([big, -big, big / 8, float(torch.finfo(dt).tiny), 0.0, -0.0]):
        flat[100 * i + 3] = v
    flat[901], flat[902], flat[n - 1] = float("inf"), float("nan"), -big
    for t, f in zip(walk.node_t, feats):
        cb.cb_cache_push(walk.plan, [f], H.CB[cache], t)
    out = torch.empty(n, dtype=torch.float32, device="cuda")
    x = torch.zeros(n, dtype=torch.float32, device="cuda")
    cb.cb_extrapolate_weights(walk.plan, np.array([0.0, 0.0, 1.0]), [out], cb.CB_FP32, [x], cb.CB_FP32)
    torch.cuda.synchronize()
    want = flat.float()
    fine = torch.isfinite(want)
    assert torch.equal(out[fine], want[fine]) and torch.equal(x[fine], want[fine])
    assert not torch.isfinite(out[~fine]).any() and not torch.isfinite(x[~fine]).any()
    walk.close()


@pytest.mark.parametrize("src", ["bf16", "fp32"])
@pytest.mark.parametrize("io", ["bf16", "fp32"])
def test_full_step_beside_off_grid_hidden_states(cb, H, src, io):
    """A full step whose hidden states lie partly off the 16-byte grid writes
    the cache write's bytes and the oracle's hidden states."""
    w = _workload(3, "bf16")
    nodes = [900.0, 800.0, 700.0]
    a, b = H.Walk(w, node_t=nodes), H.Walk(w, node_t=nodes)
    dt = H.TORCH[io]
    offs, slot = H.slot_layout([s.numel for s in w.tensors], 2)
    for k, t in enumerate(nodes):
        feats = [workloads.trajectory(w, i, t, k, "cuda", out_dtype=H.TORCH[src]) for i in range(len(w.tensors))]
        resid = []
        for g in range(a.n_groups):
            x, _ = _shifted(w.group_shape(g), dt, (g + k) % 2)
            x.copy_(workloads.hidden_state(w, g, "cuda", dt, salt=k))
            resid.append(x)
        rh = [H.host(x) for x in resid]
        cb.cb_cache_push_residual(a.plan, feats, H.CB[src], t, resid, H.CB[io])
        cb.cb_cache_push(b.plan, feats, H.CB[src], t)
        torch.cuda.synchronize()
        assert cb.cb_plan_device_status(a.plan) == 0
        for i, s in enumerate(w.tensors):
            lo = k * slot + offs[i]
            assert torch.equal(a.cache[lo:lo + 2 * s.numel], b.cache[lo:lo + 2 * s.numel]), (k, i)
        for g in range(a.n_groups):
            F = [[H.host(feats[i])] for i, s in enumerate(w.tensors) if s.group == g]
            _, r64 = orc.extrapolate(F, [1.0], H.ORC[src], None, X=rh[g], x_dtype=H.ORC[io], resid_dtype=orc.FP64)
            f64 = [H.bf16_to_f64(f[0]) if src == "bf16" else f[0].astype(np.float64) for f in F]
            x64 = H.bf16_to_f64(rh[g]) if io == "bf16" else rh[g].astype(np.float64)
            if io == "bf16":
                st = H.compare_bf16(H.host(resid[g]), orc.convert(r64, orc.FP64, orc.BF16), r64,
                                    np.abs(np.array(f64)).sum(0) + np.abs(x64))
            else:
                st = H.compare_fp32(H.host(resid[g]), r64, float(np.max(np.abs(f64))))
            assert st["bad"] == 0, (k, g, st)
    a.close()
    b.close()


@pytest.mark.parametrize("steps", [1, 12])
def test_steps_in_a_row_match_the_direct_kernel(cb, H, steps):
    """Launches that overlap the end of the one before, each adding to the
    hidden states that it left, with a history a little larger than L2's share
    for it (71 MB, most of it copied in for eviction first): bit for bit what
    the direct-load kernel gives, which overlaps nothing."""
    tensors = [workloads.TensorSpec(g, b, (1, 256, 1152), g) for g in range(15) for b in range(2)]
    w = workloads.Workload(name="row", tensors=tensors, K=4, cache_dtype="bf16", T=0, r=0, t_min=0.0, t_max=999.0,
                           timesteps=[], degree=6, noise=0.1, seed=41)
    nodes = [900.0, 860.0, 820.0, 780.0]
    got = {}
    for kernel in ("auto", "direct"):
        walk = H.Walk(w, node_t=nodes, kernel=kernel)
        feats = [[workloads.trajectory(w, i, t, k, "cuda") for i in range(len(tensors))] for k, t in enumerate(nodes)]
        resid = [workloads.hidden_state(w, g, "cuda") for g in range(walk.n_groups)]
        outs = [torch.empty(s.shape, dtype=torch.bfloat16, device="cuda") for s in tensors]
        for t, f in zip(nodes, feats):
            cb.cb_cache_push(walk.plan, f, cb.CB_BF16, t)
        for k in range(steps):
            cb.cb_extrapolate(walk.plan, 770.0 - k, outs, cb.CB_BF16, resid, cb.CB_BF16)
        cb.cb_cache_push(walk.plan, outs, cb.CB_BF16, 700.0)  # the last predictions, as a full step's features
        torch.cuda.synchronize()
        assert cb.cb_plan_device_status(walk.plan) == 0
        got[kernel] = (outs, resid, walk.cache[: walk.cache.numel() - cb.CB_STATUS_BYTES])
        walk.close()
    for a, b in zip(got["auto"][0] + got["auto"][1], got["direct"][0] + got["direct"][1]):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    assert torch.equal(got["auto"][2], got["direct"][2])


@pytest.mark.parametrize("gated", [False, True])
@pytest.mark.parametrize("K,cache", [(6, "bf16"), (7, "bf16"), (6, "fp32")])
def test_groups_too_large_to_hold(cb, H, K, cache, gated):
    """Groups of four whose stages do not fit beside one another, whole tiles
    and a ragged one: predictions and hidden states in bf16, on either side of
    the rule that sends them to the compensated kernels."""
    tensors = [workloads.TensorSpec(g, b, (2, 53, 136), g) for g in range(2) for b in range(4)]
    w = workloads.Workload(name="deep", tensors=tensors, K=K, cache_dtype=cache, T=0, r=0, t_min=0.0, t_max=999.0,
                           timesteps=[], degree=6, noise=0.1, seed=23)
    nodes = [990.0 - 37.0 * k for k in range(K)]
    walk = H.Walk(w, node_t=nodes)
    cb.cb_plan_set_shapes(walk.plan, [s.shape for s in tensors])
    for k, t in enumerate(nodes):
        walk.push(t, k)
    outs = [torch.empty(s.shape, dtype=torch.bfloat16, device="cuda") for s in tensors]
    resid = [workloads.hidden_state(w, g, "cuda") for g in range(walk.n_groups)]
    rh = [H.host(x) for x in resid]
    gen = torch.Generator(device="cuda").manual_seed(6)
    gates = [torch.randn(s.shape[0], s.shape[2], generator=gen, device="cuda").bfloat16() for s in tensors]
    target = nodes[-1] - 20.0
    if gated:
        cb.cb_extrapolate_gated(walk.plan, target, outs, cb.CB_BF16, resid, cb.CB_BF16, gates, cb.CB_BF16)
    else:
        cb.cb_extrapolate(walk.plan, target, outs, cb.CB_BF16, resid, cb.CB_BF16)
    torch.cuda.synchronize()
    assert cb.cb_plan_device_status(walk.plan) == 0
    G = [H.expand_gate(g, s.shape) for g, s in zip(gates, tensors)] if gated else None
    so, sr, _ = walk.expected_and_compare(target, outs, resid, rh, G=G)
    assert so["bad"] == 0 and sr["bad"] == 0, (so, sr)
    walk.close()


@pytest.mark.parametrize("kernel", ["bulk", "direct"])
@pytest.mark.parametrize("K,cache,io", [(3, "bf16", "fp32"), (4, "bf16", "bf16"), (8, "bf16", "fp32"), (3, "fp32", "bf16"),
                                        (5, "fp32", "fp32"), (8, "fp32", "fp32")])
@pytest.mark.parametrize("weight", [0.0, 2.0 ** -24])
def test_a_large_feature_under_a_small_weight(cb, H, K, cache, io, kernel, weight):
    """One history entry 2^20 to 2^30 times the size of the others, with a weight
    of (nearly) nothing, and the others' terms cancelling to any depth: whole
    tiles, a ragged one, and buffers off the 16-byte grid. The error bound of the
    compensated sums is u |P| + 2^-40 sum_j |w_j F_j| for fp32 results (u = 2^-24,
    one rounding) and the bf16 gate's otherwise."""
    sizes = [9728, 6099, 4865]
    tensors = [workloads.TensorSpec(i, 0, (1, 1, n), i) for i, n in enumerate(sizes)]
    w = workloads.Workload(name="spread", tensors=tensors, K=K, cache_dtype=cache, T=0, r=0, t_min=0.0, t_max=999.0,
                           timesteps=[], degree=1, noise=0.0, seed=1)
    nodes = [900.0 - 50.0 * k for k in range(K)]
    walk = H.Walk(w, node_t=nodes, kernel=kernel)
    rng = np.random.default_rng(12 + K)
    wts = rng.standard_normal(K)
    wts[K // 2] = weight
    feats = [[None] * len(sizes) for _ in range(K)]
    for i, n in enumerate(sizes):
        f = rng.standard_normal((K, n))
        f[K // 2] *= 2.0 ** rng.uniform(20, 30, n)
        rest = sum(wts[j] * f[j] for j in range(1, K) if j != K // 2)
        f[0] = -rest / wts[0] * (1 + rng.standard_normal(n) * 2.0 ** -rng.uniform(0, 20, n))
        for j in range(K):
            feats[j][i] = torch.tensor(f[j], device="cuda").to(H.TORCH[cache])
    for j in range(K):
        cb.cb_cache_push(walk.plan, feats[j], H.CB[cache], nodes[j])
    dt = H.TORCH[io]
    outs, resid = [[_shifted((1, 1, n), dt, int(i == 2))[0] for i, n in enumerate(sizes)] for _ in range(2)]
    for x in resid:
        x.copy_(torch.tensor(rng.standard_normal(x.shape) * 2.0 ** -8))
    x64 = [x.double().cpu().numpy().reshape(-1) for x in resid]
    cb.cb_extrapolate_weights(walk.plan, wts, outs, H.CB[io], resid, H.CB[io])
    torch.cuda.synchronize()
    assert cb.cb_plan_device_status(walk.plan) == 0
    for i in range(len(sizes)):
        f64 = np.array([feats[j][i].double().cpu().numpy() for j in range(K)])
        p, bound = wts @ f64, np.abs(wts) @ np.abs(f64)
        for got, want, b in [(outs[i], p, bound), (resid[i], p + x64[i], bound + np.abs(x64[i]))]:
            if io == "bf16":
                st = H.compare_bf16(H.host(got), orc.convert(want, orc.FP64, orc.BF16), want, b)
                assert st["bad"] == 0, (i, st)
            else:
                err = np.abs(H.host(got).astype(np.float64) - want)
                assert np.all(err <= 2.0 ** -24 * np.abs(want) + H.FLOOR * b), (i, float((err / b).max()))
    walk.close()


@pytest.mark.parametrize("cache", ["bf16", "fp32"])
def test_slot_padding_does_not_matter(cb, H, cache):
    """Tensors of odd length, whose last pair ends in the slot's padding: the
    same bits whether that holds zeros or NaN, with terms that cancel so far that
    another way of summing would show."""
    K, sizes = 8, [2501 + 2 * i for i in range(40)]
    tensors = [workloads.TensorSpec(i, 0, (1, 1, n), -1) for i, n in enumerate(sizes)]
    w = workloads.Workload(name="padding", tensors=tensors, K=K, cache_dtype=cache, T=0, r=0, t_min=0.0, t_max=999.0,
                           timesteps=[], degree=1, noise=0.0, seed=1)
    nodes = [900.0 - 50.0 * k for k in range(K)]
    rng = np.random.default_rng(4)
    wts = rng.standard_normal(K)
    feats = [[None] * len(sizes) for _ in range(K)]
    for i, n in enumerate(sizes):
        f = rng.standard_normal((K, n))
        f[0] = -(wts[1:] @ f[1:]) / wts[0] * (1 + rng.standard_normal(n) * 2.0 ** -26)
        for j in range(K):
            feats[j][i] = torch.tensor(f[j], device="cuda").to(H.TORCH[cache])
    got = []
    for fill in (0x00, 0xFF):
        walk = H.Walk(w, node_t=nodes, kernel="bulk")
        walk.cache.fill_(fill)
        for j in range(K):
            cb.cb_cache_push(walk.plan, feats[j], H.CB[cache], nodes[j])
        outs = [torch.empty(n, dtype=torch.float32, device="cuda") for n in sizes]
        cb.cb_extrapolate_weights(walk.plan, wts, outs, cb.CB_FP32)
        torch.cuda.synchronize()
        assert cb.cb_plan_device_status(walk.plan) == 0
        got.append(outs)
        walk.close()
    assert all(torch.equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("K,cache,io,members,hidden", [(8, "fp32", "fp32", 1, 2048), (6, "bf16", "bf16", 2, 3072)])
def test_wide_gate_rows(cb, H, K, cache, io, members, hidden):
    """fp32 gate rows too wide to be staged beside the pipeline's stages, read from
    global memory by the same kernels: two batches, whole tiles and a ragged one."""
    tensors = [workloads.TensorSpec(g, b, (2, 13, hidden), g) for g in range(2) for b in range(members)]
    w = workloads.Workload(name="wide", tensors=tensors, K=K, cache_dtype=cache, T=0, r=0, t_min=0.0, t_max=999.0,
                           timesteps=[], degree=6, noise=0.1, seed=29)
    nodes = [990.0 - 37.0 * k for k in range(K)]
    walk = H.Walk(w, node_t=nodes)
    cb.cb_plan_set_shapes(walk.plan, [s.shape for s in tensors])
    for k, t in enumerate(nodes):
        walk.push(t, k)
    gen = torch.Generator(device="cuda").manual_seed(8)
    gates = [torch.randn(s.shape[0], s.shape[2], generator=gen, device="cuda") for s in tensors]
    resid = [workloads.hidden_state(w, g, "cuda", H.TORCH[io]) for g in range(walk.n_groups)]
    rh = [H.host(x) for x in resid]
    outs = [torch.empty(s.shape, dtype=H.TORCH[io], device="cuda") for s in tensors]
    target = nodes[-1] - 20.0
    cb.cb_extrapolate_gated(walk.plan, target, outs, H.CB[io], resid, H.CB[io], gates, cb.CB_FP32)
    torch.cuda.synchronize()
    assert cb.cb_plan_device_status(walk.plan) == 0
    G = [H.expand_gate(g, s.shape) for g, s in zip(gates, tensors)]
    so, sr, _ = walk.expected_and_compare(target, outs, resid, rh, out_dtype=io, resid_dtype=io, G=G)
    assert so["bad"] == 0 and sr["bad"] == 0, (so, sr)
    walk.close()


@pytest.mark.parametrize("entry", ["step", "noalloc"])
@pytest.mark.parametrize("small", [True, False])
def test_overlapping_launches_of_mixed_plans(cb, H, entry, small):
    """Steps in a row whose buffers lie partly off the 16-byte grid (two launches
    each) on hidden states that each leaves to the next, full steps with hidden
    states between them, and the status handover's own launch after each: bit for
    bit what the same calls give when every one is waited for."""
    shape = (1, 77, 136) if small else (2, 256, 1152)
    tensors = [workloads.TensorSpec(g, b, shape, g) for g in range(6) for b in range(2)]
    w = workloads.Workload(name="mixed", tensors=tensors, K=4, cache_dtype="bf16", T=0, r=0, t_min=0.0, t_max=999.0,
                           timesteps=[], degree=6, noise=0.1, seed=43)
    nodes = [900.0 - 40.0 * k for k in range(10)]
    got = {}
    for wait in (True, False):
        walk = H.Walk(w, node_t=nodes)
        feats = [[workloads.trajectory(w, i, t, k, "cuda") for i in range(len(tensors))] for k, t in enumerate(nodes)]
        resid = [_shifted(shape, torch.bfloat16, g % 2)[0] for g in range(6)]
        for g, x in enumerate(resid):
            x.copy_(workloads.hidden_state(w, g, "cuda"))
        outs = [_shifted(shape, torch.bfloat16, (i // 2) % 2)[0] for i in range(len(tensors))]
        status = torch.full((24,), -1, dtype=torch.int32).pin_memory()
        torch.cuda.synchronize()
        n = 0

        def done():
            if wait:
                torch.cuda.synchronize()

        for k in range(4):
            cb.cb_cache_push(walk.plan, feats[k], cb.CB_BF16, nodes[k])
            done()
        for k in range(4, 10):
            for i in range(4):
                t = nodes[k - 1] - 5.0 * (i + 1)
                if entry == "step":
                    cb.cb_extrapolate(walk.plan, t, outs, cb.CB_BF16, resid, cb.CB_BF16)
                    status[n] = 0
                else:
                    slot_t, head, _ = cb.cb_plan_history(walk.plan, 4)
                    cb.cb_extrapolate_noalloc(walk.plan, walk.cache, walk.cache.numel() - cb.CB_STATUS_BYTES, slot_t, head,
                                              t, outs, cb.CB_BF16, resid, cb.CB_BF16, status=status[n:])
                n += 1
                done()
            cb.cb_cache_push_residual(walk.plan, outs if k % 2 else feats[k], cb.CB_BF16, nodes[k], resid, cb.CB_BF16)
            done()
        torch.cuda.synchronize()
        assert cb.cb_plan_device_status(walk.plan) == 0 and not status.any()
        got[wait] = [x.view(torch.int16).clone() for x in outs + resid]
        got[wait].append(walk.cache[: walk.cache.numel() - cb.CB_STATUS_BYTES].clone())
        walk.close()
    assert all(torch.equal(a, b) for a, b in zip(got[True][:-1], got[False][:-1]))
    offs, slot = H.slot_layout([s.numel for s in tensors], 2)
    for j in range(4):  # the slots, but for their padding
        for i, s in enumerate(tensors):
            lo = j * slot + offs[i]
            assert torch.equal(got[True][-1][lo:lo + 2 * s.numel], got[False][-1][lo:lo + 2 * s.numel])


@pytest.mark.parametrize("shift", [0, 1])
def test_overlapping_launches_captured_across_streams(cb, H, shift):
    """A captured fork and join: launches whose graph node follows a kernel, a copy,
    another stream's kernel, or two streams' at once, each waiting for all of them.
    Replays on new inputs give what the same calls give outside of a graph."""
    tensors = [workloads.TensorSpec(g, b, (1, 200, 1152), g) for g in range(4) for b in range(2)]
    w = workloads.Workload(name="fork", tensors=tensors, K=3, cache_dtype="bf16", T=0, r=0, t_min=0.0, t_max=999.0,
                           timesteps=[], degree=6, noise=0.1, seed=47)
    nodes = [900.0, 860.0, 820.0]
    walks = [H.Walk(w, node_t=nodes) for _ in range(2)]
    bf = torch.bfloat16
    bufs = [[[_shifted(s.shape, bf, shift)[0] for s in tensors] for _ in range(2)] for _ in range(2)]  # outputs, inputs
    resid = [[_shifted((1, 200, 1152), bf, shift if g % 2 else 0)[0] for g in range(4)] for _ in range(2)]
    status = torch.full((2,), -1, dtype=torch.int32).pin_memory()
    side = torch.cuda.Stream()

    def fill(salt):
        for k, walk in enumerate(walks):
            cb.cb_plan_reset(walk.plan)
            for j, t in enumerate(nodes):
                cb.cb_cache_push(walk.plan, [workloads.trajectory(w, i, t, 10 * salt + 3 * k + j, "cuda") for i in range(8)],
                                 cb.CB_BF16, t)
            for g, x in enumerate(resid[k]):
                x.copy_(workloads.hidden_state(w, g, "cuda", salt=10 * salt + k))
            for x in bufs[0][k] + bufs[1][k]:
                x.zero_()

    def step():
        here = torch.cuda.current_stream()
        outs, ins = bufs
        cb.cb_extrapolate(walks[0].plan, 800.0, outs[0], cb.CB_BF16, resid[0], cb.CB_BF16, stream=here)
        side.wait_stream(here)
        # on the side: after another stream's kernel; then after a copy
        cb.cb_extrapolate(walks[1].plan, 800.0, outs[1], cb.CB_BF16, resid[0], cb.CB_BF16, stream=side)
        with torch.cuda.stream(side):
            for a, b in zip(ins[1], outs[1]):
                a.copy_(b)
        cb.cb_extrapolate(walks[1].plan, 790.0, ins[1], cb.CB_BF16, resid[1], cb.CB_BF16, stream=side)
        cb.cb_extrapolate(walks[0].plan, 790.0, ins[0], cb.CB_BF16, stream=here)
        here.wait_stream(side)
        # after both streams' kernels
        slot_t, head, _ = cb.cb_plan_history(walks[0].plan, 3)
        cb.cb_extrapolate_noalloc(walks[0].plan, walks[0].cache, walks[0].cache.numel() - cb.CB_STATUS_BYTES, slot_t, head,
                                  780.0, outs[0], cb.CB_BF16, resid[1], cb.CB_BF16, status=status, stream=here)
        for a, b in zip(outs[1], outs[0]):
            a.add_(b)

    def result():
        torch.cuda.synchronize()
        assert int(status[0]) == 0 and all(cb.cb_plan_device_status(x.plan) == 0 for x in walks)
        return [x.view(torch.int16).clone() for pair in bufs + [resid] for xs in pair for x in xs]

    main = torch.cuda.Stream()
    want = []
    for salt in (0, 1):
        fill(salt)
        torch.cuda.synchronize()
        with torch.cuda.stream(main):
            step()
        want.append(result())
    fill(0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        step()
    for salt in (0, 1, 0):
        fill(salt)
        status.fill_(-1)
        torch.cuda.synchronize()
        graph.replay()
        assert all(torch.equal(a, b) for a, b in zip(result(), want[salt])), salt
    for walk in walks:
        walk.close()
