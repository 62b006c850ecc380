"""The host code of the library on a CPU, over a CUDA runtime in host memory
(tests/host/fake_cuda.cpp), where a buffer that a launch is given and that is
not live memory of the context's device, large enough, is counted: after an
allocation that failed (every one of a call in turn), a later call of any size
gets buffers that are there; a caller's memory is given to a kernel only where
that can read it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import paper_2007_09884_gb300 as G
from paper_2007_09884_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="session")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("host") / "libopmm_host.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    if not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        cuda = "/usr/local/cuda/include"
    src = [os.path.join(B.CSRC, f) for f in ("capi.cu", "surrogate.cu", "serve.cu")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-pthread", "-Wl,-Bsymbolic", "-I", cuda, "-I", B.CSRC, "-include",
                    os.path.join(HERE, "host", "device_names.h"), "-x", "c++", *src,
                    os.path.join(HERE, "host", "fake_cuda.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    for f in ("fake_allocs", "fake_bad", "fake_in_use"):
        getattr(lib, f).restype = ctypes.c_longlong
    lib.fake_scored_at.restype = ctypes.c_void_p
    lib.fake_move.argtypes = [ctypes.c_void_p, ctypes.c_int]
    for f in ("fake_fail_alloc", "fake_capacity"):
        getattr(lib, f).argtypes = [ctypes.c_longlong]
    lib.opmm_destroy.restype = lib.opmm_plan_destroy.restype = None
    return lib


@pytest.fixture
def ctx(lib):
    h = ctypes.c_void_p()
    assert lib.opmm_create(0, ctypes.byref(h)) == G.OPMM_OK
    assert lib.opmm_surrogate_init(h, ctypes.c_uint64(1)) == G.OPMM_OK
    yield h
    lib.fake_fail_alloc(-1)
    lib.opmm_destroy(h)


def _batch(n, L=60):
    y = np.zeros(L, np.float32)
    return G.make_batch([y] * n, [1000.0] * n, [10] * n, [0.0] * n, [10.0] * n, [43.0] * n)


def _predict(lib, ctx, n):
    descs, keep = _batch(n).descriptors()
    out = np.zeros((n, 18), np.float32)
    return lib.opmm_surrogate_predict(ctx, descs, n, G.OPMM_PULSE_CALIBRATED, out.ctypes.data_as(ctypes.c_void_p))


def _train(lib, ctx, batch):
    return lib.opmm_surrogate_train(ctx, 1, batch, ctypes.c_float(1e-3), ctypes.c_float(0.0), ctypes.c_uint64(1),
                                    ctypes.c_int64(0), None)


def _grad(lib, ctx, m):
    x, t = np.zeros((m, 512), np.float32), np.zeros((m, 18), np.float32)
    g, loss = np.zeros(4 * (512 * 512 + 512) + 18 * 513, np.float32), ctypes.c_float()
    return lib.opmm_surrogate_grad(ctx, *(v.ctypes.data_as(ctypes.c_void_p) for v in (x, t)), m, ctypes.byref(loss),
                                   g.ctypes.data_as(ctypes.c_void_p), None)


@pytest.mark.parametrize("call", [_predict, _train, _grad], ids=["predict", "train", "grad"])
def test_buffers_after_a_failed_allocation(lib, ctx, call):
    bad = lib.fake_bad()
    for nth in range(60):
        assert call(lib, ctx, 256 * (1 + 3 * nth)) == G.OPMM_OK     # what a first call leaves behind
        before = lib.fake_allocs()
        lib.fake_fail_alloc(nth)
        rc = call(lib, ctx, 256 * (3 + 3 * nth))                    # grows, and its nth allocation fails
        hit = lib.fake_allocs() - before > nth
        lib.fake_fail_alloc(-1)
        assert rc == (G.OPMM_ENOMEM if hit else G.OPMM_OK)
        assert call(lib, ctx, 256) == G.OPMM_OK                     # smaller than what was there
        assert lib.fake_bad() == bad, f"allocation {nth} failed: a later launch got a buffer that is not there"
        if not hit:
            break
    else:
        pytest.fail("the call allocates more often than this test fails it")


# where the caller keeps the trace: host memory, this device's, this device's off a float's boundary, another device's
@pytest.mark.parametrize("where,in_place", [("host", False), ("device", True), ("odd", False), ("other", False)])
def test_score_reads_a_trace_in_place_only_where_its_kernel_can(lib, ctx, where, in_place):
    L, m = 61, 5
    y = np.arange(L, dtype=np.float32)
    block = ctypes.c_void_p()
    assert lib.cudaMalloc(ctypes.byref(block), ctypes.c_size_t(4 * L + 4)) == 0
    at = block.value + (2 if where == "odd" else 0)
    ctypes.memmove(at, y.ctypes.data, 4 * L)
    if where == "other":
        lib.fake_move(block, 1)
    if where == "host":
        at = y.ctypes.data
    sac = G.opmm_saccade(at, L, 1000.0, 10, 0.0, 10.0, 43.0)
    opc, f = np.full((m, 18), 1.0, np.float32), np.zeros(m, np.float32)
    bad = lib.fake_bad()
    assert lib.opmm_score(ctx, opc.ctypes.data_as(ctypes.c_void_p), m, ctypes.byref(sac),
                          f.ctypes.data_as(ctypes.c_void_p)) == G.OPMM_OK
    assert lib.fake_bad() == bad
    assert (lib.fake_scored_at() == at) == in_place
    np.testing.assert_array_equal(np.frombuffer(ctypes.string_at(lib.fake_scored_at(), 4 * L), np.float32), y)
    assert lib.cudaFree(block) == 0


def _tuned_shapes(lib, ctx, n, simplices):
    descs, keep = _batch(n).descriptors()
    o, keep_o = G.fit_opts(candidates=22 * simplices, iterations=4)
    plan = ctypes.c_void_p()
    assert lib.opmm_plan_create(ctx, descs, n, ctypes.byref(o), ctypes.byref(plan)) == G.OPMM_OK
    variants, count = (ctypes.c_int32 * 16)(), ctypes.c_int32()
    assert lib.opmm_plan_tuning(plan, variants, None, None, None, None, 16, ctypes.byref(count)) == G.OPMM_OK
    lib.opmm_plan_destroy(plan)
    return variants[:count.value]


# 64 saccades of 64 simplices leave every unit at 32 simplices, so the larger shapes are not tried; 3,000 do not
@pytest.mark.parametrize("first,then", [(64, 3000), (3000, 64), (74, 1024)])
def test_tuning_does_not_depend_on_an_earlier_plan(lib, ctx, first, then):
    fresh = ctypes.c_void_p()
    assert lib.opmm_create(0, ctypes.byref(fresh)) == G.OPMM_OK
    want = _tuned_shapes(lib, fresh, then, 64)
    lib.opmm_destroy(fresh)
    assert _tuned_shapes(lib, ctx, first, 64) != want          # the two batches have different candidate shapes
    assert _tuned_shapes(lib, ctx, then, 64) == want
    assert _tuned_shapes(lib, ctx, then, 64) == want           # and again, from the cache


def _slots(lib, ctx):
    cfg = G.opmm_serve_opts(max_slots=1 << 30, max_queue=4, max_samples=400, round_iters=5, max_admit_per_round=4)
    o, keep = G.fit_opts(candidates=4096, iterations=4)
    stats = G.opmm_serve_stats()
    assert lib.opmm_serve_start(ctx, ctypes.byref(cfg), ctypes.byref(o)) == G.OPMM_OK
    assert lib.opmm_serve_stats_get(ctx, ctypes.byref(stats)) == G.OPMM_OK
    assert lib.opmm_serve_stop(ctx) == G.OPMM_OK
    return stats.slots


def test_kept_buffers_do_not_shrink_the_request_loop(lib, ctx):
    lib.fake_capacity(lib.fake_in_use() + (1 << 30))
    try:
        slots = _slots(lib, ctx)
        assert _predict(lib, ctx, 50000) == G.OPMM_OK     # leaves 150 MB of activations and 30 MB beside
        assert lib.fake_in_use() > (100 << 20)
        assert _slots(lib, ctx) == slots
    finally:
        lib.fake_capacity(1 << 40)


@pytest.mark.parametrize("call", [_train, _grad], ids=["train", "grad"])
def test_kept_buffers_are_given_back_when_memory_runs_out(lib, ctx, call):
    m = 128 * 200
    own = lib.fake_in_use()
    other = ctypes.c_void_p()
    assert lib.opmm_create(0, ctypes.byref(other)) == G.OPMM_OK
    assert lib.opmm_surrogate_init(other, ctypes.c_uint64(1)) == G.OPMM_OK
    base = lib.fake_in_use()
    assert call(lib, other, m) == G.OPMM_OK
    need = lib.fake_in_use() - base
    lib.opmm_destroy(other)
    assert _predict(lib, ctx, 50000) == G.OPMM_OK
    kept = lib.fake_in_use() - own
    assert kept > (100 << 20)
    lib.fake_capacity(own + need + (64 << 20))            # room for the call, but not beside what is kept
    try:
        assert call(lib, ctx, m) == G.OPMM_OK
    finally:
        lib.fake_capacity(1 << 40)
    assert _predict(lib, ctx, 300) == G.OPMM_OK           # and the next one-shot call allocates anew
    assert lib.fake_bad() == 0


def test_what_a_failed_call_leaves_is_bounded(lib, ctx):
    assert _predict(lib, ctx, 256) == G.OPMM_OK
    own = lib.fake_in_use()
    for nth in range(1, 3):                                # activations: X grows, then a layer's buffer fails
        lib.fake_fail_alloc(nth)
        assert _predict(lib, ctx, 1200000) == G.OPMM_ENOMEM
        lib.fake_fail_alloc(-1)
        assert lib.fake_in_use() <= own
    assert _predict(lib, ctx, 256) == G.OPMM_OK
