"""What the binding hands to the library for a list of host arrays: calls that
read no trace or one trace do not gather the others, long traces are pointed at
where they are, and every descriptor holds its saccade's values."""
import ctypes

import numpy as np
import pytest

import paper_2007_09884_gb300 as G

FIELDS = ("n_samples", "sample_rate_hz", "onset_index", "theta_start_deg", "theta_end_deg", "duration_ms")


class _Library:
    """Records the descriptors that a call passes on (with their samples)."""

    def __init__(self, n):
        self.n, self.got = n, None

    def _take(self, descs, n):
        self.got = [{f: getattr(descs[i], f) for f in FIELDS + ("trace_deg",)} for i in range(n)]
        for d in self.got:
            d["samples"] = None if not d["trace_deg"] else np.array(
                np.ctypeslib.as_array(ctypes.cast(d["trace_deg"], ctypes.POINTER(ctypes.c_float)), (d["n_samples"],)))
        return G.OPMM_OK

    def opmm_simulate(self, ctx, opc, n, descs, n_sacs, *rest):
        return self._take(descs, n_sacs)

    def opmm_nominal_opc(self, ctx, descs, n, *rest):
        return self._take(descs, n)

    def opmm_score(self, ctx, opc, m, desc, f):
        return self._take([desc._obj], 1)

    def opmm_serve_submit(self, ctx, desc, ticket):
        return self._take([desc._obj], 1)

    def opmm_fit_batch(self, ctx, descs, n, opts, res):
        return self._take(descs, n)


@pytest.fixture
def lib(monkeypatch):
    stub = _Library(0)
    monkeypatch.setattr(G, "load_library", lambda *a: stub)
    return stub


def _batch(n, L, dtype=np.float32):
    g = np.random.default_rng(n + L)
    sizes = g.integers(L // 2 + 1, L + 1, n)
    traces = [g.normal(size=k).astype(dtype) for k in sizes]
    return G.make_batch(traces, g.choice([250.0, 500.0, 1000.0], n), np.arange(n) % 5, g.normal(size=n), g.normal(size=n),
                        30.0 + g.random(n))


def _check(got, batch, i):
    for f in FIELDS:
        assert got[f] == getattr(batch, f)[i], f


@pytest.mark.parametrize("n", [1, 6, 7, 200])
@pytest.mark.parametrize("call", ["simulate", "nominal"])
def test_calls_that_read_no_trace_do_not_gather(lib, n, call):
    batch = _batch(n, 300)
    if call == "simulate":
        G.opmm_simulate(None, np.ones((n, 18), np.float32), batch)
    else:
        G.opmm_nominal_opc(None, batch)
    for i, d in enumerate(lib.got):
        _check(d, batch, i)
        assert not d["trace_deg"] or d["trace_deg"] == batch.traces[i].ctypes.data


@pytest.mark.parametrize("n,index", [(1, 0), (6, 2), (7, 6), (7, -1), (200, 101), (200, np.int64(-200))])
@pytest.mark.parametrize("call", ["score", "submit"])
def test_calls_that_read_one_trace_take_it_where_it_is(lib, n, index, call):
    batch = _batch(n, 300)

    def run(index):
        if call == "score":
            G.opmm_score(None, np.ones((3, 18), np.float32), batch, index=index)
        else:
            G.opmm_serve_submit(None, batch, index)

    run(index)
    _check(lib.got[0], batch, index)
    assert lib.got[0]["trace_deg"] == batch.traces[index].ctypes.data
    for outside in (n, -n - 1):
        with pytest.raises(IndexError):
            run(outside)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n,L", [(3, 9000), (7, 200), (7, 9000), (40, 5000), (40, 6200)])
def test_fits_read_every_trace(lib, n, L, dtype):
    batch = _batch(n, L, dtype)
    G.opmm_fit_batch(None, batch)
    long = np.mean(batch.n_samples) > 4000
    for i, d in enumerate(lib.got):
        _check(d, batch, i)
        np.testing.assert_array_equal(d["samples"], batch.traces[i].astype(np.float32))
        if dtype == np.float32 and (long or n <= 6):
            assert d["trace_deg"] == batch.traces[i].ctypes.data


# what indexes and converts entry by entry is taken at every size: lists, arrays of other types, tensors (of the
# device too: any that numpy does not read by itself)
@pytest.mark.parametrize("n", [3, 7, 50])
@pytest.mark.parametrize("kind", ["list", "float64", "tensor", "grad"])
def test_fields_and_offsets_of_every_kind(lib, n, kind):
    torch = pytest.importorskip("torch")
    ref = _batch(n, 300)
    offsets = np.concatenate([[0], np.cumsum(ref.n_samples)[:-1]])
    convert = {"list": lambda v: [x.item() for x in v], "float64": lambda v: v.astype(np.float64),
               "tensor": lambda v: torch.tensor(v.tolist()),
               "grad": lambda v: torch.tensor(v.tolist(), dtype=torch.float64, requires_grad=True)}[kind]
    packed = np.concatenate(ref.traces)
    batch = G.SaccadeBatch(packed, convert(offsets), *(convert(getattr(ref, f)) for f in FIELDS))
    G.opmm_fit_batch(None, batch)
    for i, d in enumerate(lib.got):
        _check(d, ref, i)
        np.testing.assert_array_equal(d["samples"], ref.traces[i])
    batch = G.SaccadeBatch(ref.traces, None, *(convert(getattr(ref, f)) for f in FIELDS))
    G.opmm_fit_batch(None, batch)
    for i, d in enumerate(lib.got):
        _check(d, ref, i)
        np.testing.assert_array_equal(d["samples"], ref.traces[i])
