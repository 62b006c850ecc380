"""Refinement with its rows in shared memory and, for windows too long for
that, in global memory: short windows, the longest that fits, the next size up.

Tolerance: as in the refinement's parity tests, over three damped iterations
(lambda0 = 10) the refined RMS is within 1e-3 deg of the oracle's from the
same start, and the FP64 errors are the oracle's to 1e-9 relative."""
import numpy as np
import pytest

import oracle as O
import paper_2007_09884_gb300 as G
from _support import f32, to_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,L", [(18, 13), (18, 64), (18, 1224), (18, 1225), (9, 14), (9, 2232), (9, 2233)])
def test_rows_in_either_memory(model, L):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A, D, fs, onset = 10.0, 43.0, 1000.0, 5
    rng = np.random.default_rng(L)
    pn = f32(O.nominal_opc(A, D, calibrated=True))
    first = list(range(18)) if model == 18 else [0, 2, 7, 8, 6, 4, 5, 9, 14]
    y = f32(O.simulate_rk4(f32(pn * rng.uniform(0.95, 1.05, 18)), L, fs, onset, 0.0, A) + rng.normal(0.0, 0.05, L))
    start = pn.copy()
    start[first] *= np.exp(rng.uniform(-0.05, 0.05, len(first)))
    if model == 9:
        start[1], start[3] = start[0], start[2]
    start = f32(start)
    ctx = G.opmm_create(0)
    try:
        r = G.opmm_refine_batch(ctx, to_batch([dict(y=y, fs=fs, onset=onset, th0=0.0, thf=A, dur=D, L=L)]), start[None],
                                iterations=3, model=model, lambda0=10.0, centre_opc=pn[None])
    finally:
        G.opmm_destroy(ctx)
    want = O.refine(pn, L, fs, onset, 0.0, A, y, np.log(start[first] / pn[first]), 3, model=model, lambda0=10.0)
    assert r["status"][0] == 0
    assert abs(r["rms_deg"][0] - want["rms"]) <= 1e-3
    mse, mae = O.errors(r["opc"][0].astype(np.float64), L, fs, onset, 0.0, A, y)
    assert abs(r["rms_deg"][0] - np.sqrt(mse)) <= 1e-9 * np.sqrt(mse)
    assert abs(r["l1_deg"][0] - mae) <= 1e-9 * mae
