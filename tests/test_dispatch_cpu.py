"""Which kernel a call runs, with what, and what stays behind when a launch fails:
the library's host side over stand-ins for the CUDA runtime and the launchers
(host_stub.cpp), on the CPU."""
import ctypes
import importlib.util
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NODES = [900.0 - 50.0 * k for k in range(8)]


@pytest.fixture(scope="module")
def cb(tmp_path_factory):
    """The binding over the stub, with `stub` for the stub's own functions."""
    from paper_2608_23429_gb300 import build
    build.build()
    so = str(tmp_path_factory.mktemp("stub") / "libstub.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    subprocess.run([shutil.which("g++"), "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", f"-I{cuda}", "-o", so,
                    os.path.join(ROOT, "tests", "host_stub.cpp"), os.path.join(build.CSRC, "plan.cpp")], check=True)
    spec = importlib.util.spec_from_file_location("chebboost_on_stub", os.path.join(build.HERE, "chebboost.py"))
    mod = importlib.util.module_from_spec(spec)
    cdll, ctypes.CDLL = ctypes.CDLL, lambda path, *a: cdll(so)
    try:
        spec.loader.exec_module(mod)
    finally:
        ctypes.CDLL = cdll
    mod.stub = cdll(so)
    mod.stub.stub_log.restype = ctypes.c_char_p
    return mod


def _log(cb):
    """(name, {field: value}) of every call noted since the last reset."""
    return [(line.split()[0], {k: int(v) for k, v in re.findall(r"(\w+)=(\d+)", line)})
            for line in cb.stub.stub_log().decode().splitlines()]


def _plan(cb, K, shapes, groups, cache, steps=None):
    plan = cb.cb_plan_create(NODES[:max(K, 1)], K, [(i, 0, b * t * h, g) for i, ((b, t, h), g) in enumerate(zip(shapes, groups))],
                             cache, 0.0, 999.0)
    cb.cb_plan_set_shapes(plan, shapes)
    cb.cb_plan_bind_cache(plan, 1 << 40, cb.cb_plan_cache_bytes(plan))
    cb.stub.stub_reset()
    for k in range(K if steps is None else steps):
        cb.cb_cache_push(plan, [(1 << 41) + (i << 32) for i in range(len(shapes))], cache, NODES[k])
    cb.stub.stub_reset()
    return plan


def _addresses(n, base, off=0):
    return [base + (i << 32) + off for i in range(n)]


def test_failed_launch_leaves_no_error_behind(cb):
    """A launch that fails reports CB_ERR_CUDA once: the runtime's last error is
    taken with it, so that the caller's next check finds none."""
    plan = _plan(cb, 3, [(1, 16, 64)], [-1], cb.CB_BF16, steps=1)
    cb.stub.stub_fail(b"launch")
    with pytest.raises(cb.CbError) as e:
        cb.cb_cache_push(plan, [1 << 41], cb.CB_BF16, NODES[1])
    assert e.value.status == cb.CB_ERR_CUDA
    assert cb.stub.stub_last_error() == 0
    cb.cb_cache_push(plan, [1 << 41], cb.CB_BF16, NODES[1])  # the failed step left the history as it was
    cb.cb_plan_destroy(plan)


def _noalloc(cb, plan, outs, status):
    n = cb.cb_plan_cache_bytes(plan) - cb.CB_STATUS_BYTES
    cb.cb_extrapolate_noalloc(plan, 1 << 42, n, NODES[:3], 0, 780.0, outs, cb.CB_BF16, status=status)


@pytest.mark.parametrize("fails", ["bulk", "bulk_strided", "take_status", "memcpy", "memset"])
def test_status_that_nobody_was_told_is_cleared(cb, fails):
    """A call that fails between its launch and the handover of the status word
    leaves that word to be cleared by the next call that asks, once, before its
    launch; a captured clearing runs later and does not count."""
    plan = _plan(cb, 3, [(1, 64, 64)] * 2, [-1, -1], cb.CB_BF16)
    outs = [(1 << 43) + 16, (1 << 44) + 2]  # an aligned one and one off the grid: two launches
    word = ctypes.c_int(-1)
    pinned = fails not in ("memcpy", "memset")
    cb.stub.stub_host_memory(pinned)
    cb.stub.stub_fail(fails.encode())
    with pytest.raises(cb.CbError):
        _noalloc(cb, plan, outs, ctypes.addressof(word))

    def calls(status):
        cb.stub.stub_reset()
        cb.stub.stub_host_memory(1)
        return_to = ctypes.addressof(word) if status else None
        _noalloc(cb, plan, outs, return_to)
        return [c[0] for c in _log(cb)]

    launches = ["bulk_strided", "bulk"]
    assert calls(False) == launches  # asks nothing, records nothing
    cb.stub.stub_reset()
    cb.stub.stub_host_memory(1)
    cb.stub.stub_capturing(1)
    _noalloc(cb, plan, outs, ctypes.addressof(word))
    assert [c[0] for c in _log(cb)] == ["memset"] + launches + ["take_status"]
    assert calls(True) == ["memset"] + launches + ["take_status"]
    assert calls(True) == launches + ["take_status"]
    cb.cb_plan_destroy(plan)


@pytest.mark.parametrize("offset", [0, 1, 2])
def test_status_off_the_word_grid_is_copied(cb, offset):
    """The device writes a pinned status itself only where an int may lie; any
    other address is copied to, as ordinary memory is."""
    plan = _plan(cb, 3, [(1, 64, 64)], [-1], cb.CB_BF16)
    buf = (ctypes.c_int * 2)()
    cb.stub.stub_host_memory(1)
    _noalloc(cb, plan, [1 << 43], ctypes.addressof(buf) + offset)
    assert [c[0] for c in _log(cb)] == ["bulk"] + (["take_status"] if offset == 0 else ["memcpy", "memset"])
    cb.cb_plan_destroy(plan)


@pytest.mark.parametrize("K,cache,io,gate,members,hidden,name,staged",
                         [(8, 1, 1, 1, 1, 1024, "bulk_precise", True), (8, 1, 1, 1, 1, 2048, "bulk_precise", False),
                          (8, 1, 1, 0, 2, 4096, "bulk_precise", False), (5, 0, 0, 1, 2, 3072, "bulk_gated", True),
                          (6, 0, 0, 1, 2, 3072, "bulk_gated", False), (2, 0, 1, 1, 2, 4096, "bulk_precise", True)])
def test_wide_gate_rows_stay_on_the_pipeline(cb, K, cache, io, gate, members, hidden, name, staged):
    """Gate rows that leave no room for the pipeline's stages are left in global
    memory; the launch keeps its kernel."""
    plan = _plan(cb, K, [(1, 64, hidden)] * members, [0] * members, cache)
    cb.cb_extrapolate_gated(plan, 100.0, None, io, [1 << 45], io, _addresses(members, 1 << 43), gate)
    (got, a), = _log(cb)
    assert got == name and (a["gates"] > 0) == staged and a["stages"] >= (2 if name == "bulk_precise" else members + 1), a
    assert a["smem"] <= 232448
    cb.cb_plan_destroy(plan)


@pytest.mark.parametrize("groups,batch,tokens,hidden,fewer", [(1, 1, 256, 1152, False), (28, 1, 256, 1152, False),
                                                              (4, 4, 1024, 1152, False), (28, 8, 256, 1152, True),
                                                              (28, 4, 1024, 2048, True), (19, 1, 4096, 3072, False)])
def test_gated_full_steps_take_every_processor_unless_large(cb, groups, batch, tokens, hidden, fewer):
    """Gated full steps of groups of two: a launch that leaves processors free
    cannot overlap the one before, which small steps live by."""
    plan = _plan(cb, 3, [(batch, tokens, hidden)] * (2 * groups), [i // 2 for i in range(2 * groups)], cb.CB_BF16, steps=0)
    cb.cb_cache_push_residual(plan, _addresses(2 * groups, 1 << 41), cb.CB_BF16, NODES[0], _addresses(groups, 1 << 42),
                              cb.CB_BF16, _addresses(2 * groups, 1 << 43), cb.CB_BF16)
    (name, a), = [c for c in _log(cb) if c[0] != "memset"]
    tiles = groups * batch * tokens * hidden // 4096
    assert name == "bulk_gated" and a["overlap"] == int(not fewer)
    assert a["grid"] == (288 if fewer else min(304, tiles))
    cb.cb_plan_destroy(plan)
