"""A search's result does not depend on how its simplices are split over the
device, and its FP64 check holds at the edges of its blocks of 32 samples.

Tolerances: every walk performs the same single-precision operations on a
candidate and a simplex evolves alone, so results of different launch shapes
are compared bit for bit; the FP64 errors against the oracle's recomputation
of the same vector to 1e-9 relative (the bound of the other parity tests)."""
import numpy as np
import pytest

import oracle as O
import paper_2007_09884_gb300 as G
import workloads as W
from _support import centres, f32, oracle_inputs, to_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    h = G.opmm_create(0)
    yield h
    G.opmm_destroy(h)


@pytest.fixture(scope="module")
def items():
    return oracle_inputs(W.uneven10k(B=3))


def _same(a, b):
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


# one simplex, a few, one more or less than a group or a unit holds, several units
@pytest.mark.parametrize("model,simplices", [(18, s) for s in (1, 2, 31, 32, 33, 63, 64, 65, 190, 700)] +
                         [(9, s) for s in (1, 5, 27, 28, 107, 108, 109, 1000)])
@pytest.mark.parametrize("n", [1, 3])
def test_results_do_not_depend_on_the_split(ctx, items, model, simplices, n):
    batch = to_batch(items[:n])
    kw = dict(candidates=simplices * (model + 4), iterations=9, seed=7, model=model, init_opc=centres(items[:n]),
              tol_x=0.03, tol_f=0.02)   # loose enough for some simplices to stop early
    split = G.opmm_fit_batch(ctx, batch, **kw)
    variants = [v for v in range(G.opmm_search_variants())
                if G.opmm_search_variant_info(v)[1] == model and G.opmm_search_variant_walk(v) != G.OPMM_WALK_LEAN]
    for v in variants:
        G.opmm_set_search_variant(ctx, v)
        try:
            _same(split, G.opmm_fit_batch(ctx, batch, **kw))
        finally:
            G.opmm_set_search_variant(ctx, -1)


# small batches whose probes run every saccade, on each shape's own units
@pytest.mark.parametrize("model,simplices", [(18, 1), (18, 17), (18, 33), (18, 70), (18, 300), (9, 40), (9, 300)])
def test_tuned_plan_equals_the_one_shot_fit(ctx, items, model, simplices):
    batch = to_batch(items)
    kw = dict(candidates=simplices * (model + 4), iterations=5, seed=3, model=model, init_opc=centres(items))
    plan = G.opmm_plan_create(ctx, batch, **kw)
    try:
        got = plan.execute()
        if all(t["walk"] != "lean" or t["variant"] != plan.info()["variant"] for t in plan.tuning()):
            _same(got, G.opmm_fit_batch(ctx, batch, **kw))
    finally:
        plan.destroy()


# windows that end at the onset, that hold 1, 31, 32, 33, 64 and 65 samples after it, pulses shorter than a sample,
# ending on a block's edge and outlasting the window, and a vector whose substeps are refined
@pytest.mark.parametrize("fs,after,width", [(1000.0, 0, 20.0), (1000.0, 1, 20.0), (1000.0, 1, 0.3), (1000.0, 31, 16.05),
                                            (1000.0, 32, 31.0), (1000.0, 33, 32.0), (1000.0, 64, 90.0),
                                            (1000.0, 65, 33.5), (500.0, 65, 62.01), (250.0, 100, 0.05),
                                            (250.0, 390, 128.0), (1000.0, 120, -1.0)])
def test_fp64_check_at_its_block_edges(ctx, fs, after, width):
    A, onset = 12.0, 5
    L = onset + 1 + after
    p = f32(O.nominal_opc(A, 47.4, calibrated=False))
    if width < 0:                                  # stiff: more than 2.5 per 0.1 ms substep
        p[9] *= 0.02
    else:
        p[17] = np.float32(width)
    p = f32(p)
    y = f32(np.linspace(0.0, A, L) + np.random.default_rng(int(fs) + after).normal(0.0, 0.05, L))
    batch = to_batch([dict(y=y, fs=fs, onset=onset, th0=0.0, thf=A, dur=47.4, L=L)])
    r = G.opmm_fit_batch(ctx, batch, candidates=22, iterations=0, init_opc=p[None].astype(np.float32), box_lo=0.9,
                         box_hi=1.1, init_step=0.01)
    assert r["status"][0] == 0
    mse, mae = O.errors(r["opc"][0].astype(np.float64), L, fs, onset, 0.0, A, y)
    assert abs(r["rms_deg"][0] - np.sqrt(mse)) <= 1e-9 * np.sqrt(mse)
    assert abs(r["l1_deg"][0] - mae) <= 1e-9 * mae
