"""Calls of mixed kinds and sizes on one context, whose buffers then hold other
calls' data, give what each gives on a context of its own, bit for bit."""
import numpy as np
import pytest

import paper_2007_09884_gb300 as G
import workloads as W
from _support import centres, oracle_inputs, to_batch

pytestmark = pytest.mark.gpu

SEEDED = dict(candidates=22 * 12, iterations=3, box_lo=0.95, box_hi=1.05, init_step=0.025)
PLAIN = dict(candidates=22 * 20, iterations=3)


@pytest.fixture(scope="module")
def items():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return oracle_inputs(W.uneven10k(B=40))


def _run(ctx, items, kind, n, device):
    some = (items * (n // len(items) + 1))[:n]
    batch = to_batch(some, device="cuda" if device else None)
    if kind == "predict":
        return [G.opmm_surrogate_predict(ctx, batch)]
    if kind == "featurize":
        return [G.opmm_featurize(ctx, batch)]
    if kind == "refine":
        return list(G.opmm_refine_batch(ctx, batch, centres(some), iterations=2).values())
    if kind == "seeded":
        r, fallbacks = G.opmm_fit_batch_seeded(ctx, batch, SEEDED, PLAIN, 0.1)
        return list(r.values()) + [np.array(fallbacks)]
    if kind == "seeded_centres":
        return list(G.opmm_fit_batch(ctx, batch, use_surrogate=True, init_opc=centres(some), **SEEDED).values())
    return list(G.opmm_fit_batch(ctx, batch, model=9 if kind == "fit9" else 18, candidates=600, iterations=3).values())


def _context():
    h = G.opmm_create(0)
    G.opmm_surrogate_init(h, 7)
    return h


def test_mixed_calls_on_one_context(items):
    kinds = ["predict", "featurize", "refine", "seeded", "seeded_centres", "fit", "fit9"]
    rng = np.random.default_rng(11)
    calls = [(k, int(n), bool(d)) for n in (300, 1, 129, 7, 128, 40) for k, d in
             zip(rng.permutation(kinds), rng.random(len(kinds)) < 0.5)]
    shared = _context()
    try:
        for kind, n, device in calls:
            got = _run(shared, items, kind, n, device)
            own = _context()
            try:
                want = _run(own, items, kind, n, device)
            finally:
                G.opmm_destroy(own)
            for a, b in zip(got, want):
                np.testing.assert_array_equal(a, b, err_msg=f"{kind} of {n}")
    finally:
        G.opmm_destroy(shared)
