"""opmm_detect_saccades with the caller's own array: it holds the first
max_events of the kept events and nothing past them, *n_events counts all of
them, and malformed arguments are refused without touching either.  The events
are the ones of the view (tested against the reference definition elsewhere),
byte for byte."""
import ctypes

import numpy as np
import pytest

import paper_2007_09884_gb300 as G

pytestmark = pytest.mark.gpu

GUARD = 0x5A


@pytest.fixture(scope="module")
def stream():
    rng = np.random.default_rng(5)
    parts, pos = [np.zeros(30, np.float32)], 0.0
    for _ in range(40):
        step = rng.uniform(4.5, 12.0) * (1 if pos < 0 else -1)
        parts += [pos + step * np.arange(1, 13) / 12.0, np.full(70, pos + step)]
        pos += step
    return np.concatenate(parts).astype(np.float32)


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    h = G.opmm_create(0)
    yield h
    G.opmm_destroy(h)


def _opts(**kw):
    o = dict(threshold_dps=30.0, min_duration_ms=6.0, min_amplitude_deg=4.0, valid_min_deg=-90.0, valid_max_deg=90.0,
             pre_samples=10, post_samples=40)
    o.update(kw)
    return G.opmm_ivt_opts(**o)


def _call(ctx, x, opts, out, max_events, n_events):
    return G.load_library().opmm_detect_saccades(
        ctx, None if x is None else x.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(0 if x is None else x.size),
        ctypes.c_float(1000.0), None if opts is None else ctypes.byref(opts),
        None if out is None else out.ctypes.data_as(ctypes.c_void_p), max_events,
        None if n_events is None else ctypes.byref(n_events))


@pytest.mark.parametrize("cap", [0, 1, 39, 40, 41, 100])
def test_first_events_and_the_count_of_all(ctx, stream, cap):
    want = G.opmm_detect_saccades(ctx, stream, 1000.0)
    assert len(want) == 40
    size = G.IVT_EVENT_DTYPE.itemsize
    out = np.full((cap + 2) * size, GUARD, np.uint8)
    n = ctypes.c_int32(-1)
    assert _call(ctx, stream, _opts(), out if cap else None, cap, n) == G.OPMM_OK
    assert n.value == 40
    k = min(cap, 40)
    np.testing.assert_array_equal(out[:k * size], want[:k].view(np.uint8).reshape(-1))
    assert (out[k * size:] == GUARD).all()


def test_a_stream_without_events(ctx):
    out, n = np.full(64, GUARD, np.uint8), ctypes.c_int32(-1)
    assert _call(ctx, np.zeros(500, np.float32), _opts(), out, 1, n) == G.OPMM_OK
    assert n.value == 0 and (out == GUARD).all()


def test_malformed_arguments(ctx, stream):
    out, n = np.full(64, GUARD, np.uint8), ctypes.c_int32(-1)
    for args in [(None, _opts(), out, 1, n), (stream, None, out, 1, n), (stream, _opts(), out, 1, None),
                 (stream, _opts(), None, 1, n), (stream, _opts(), out, -1, n), (stream[:1], _opts(), out, 1, n),
                 (stream, _opts(threshold_dps=0.0), out, 1, n), (stream, _opts(pre_samples=-1), out, 1, n),
                 (stream, _opts(valid_min_deg=1.0, valid_max_deg=0.0), out, 1, n)]:
        assert _call(ctx, *args) == G.OPMM_EINVAL
    assert n.value == -1 and (out == GUARD).all()
