"""Trajectory rows, few (single stores) and many (stores in groups of four), at every alignment of their first sample, with as many
samples at rest as a group of four holds or fewer, and windows that end in any
part of a group.  A row is the same wherever it lies, bit for bit, and nothing
outside it is written; the values are the oracle's to the trajectory tolerance
of the other parity tests (1e-4 deg)."""
import numpy as np
import pytest

import oracle as O
import paper_2007_09884_gb300 as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [5, 47, 48, 131])
@pytest.mark.parametrize("onset", [0, 1, 2, 3, 4, 7, 40])
@pytest.mark.parametrize("after", [0, 1, 2, 3, 4, 5, 66])
def test_rows_at_every_alignment(m, onset, after):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    L = onset + 1 + after
    p = np.float32(O.nominal_opc(10.0, 43.0, calibrated=False))
    ref = O.simulate_rk4(p.astype(np.float64), L, 1000.0, onset, 2.0, -8.0)
    ctx = G.opmm_create(0)
    try:
        batch = G.make_batch([np.zeros(L, np.float32)], [1000.0], [onset], [2.0], [-8.0], [43.0])
        opc = torch.from_numpy(np.tile(p, (m, 1))).cuda()
        for lead in range(4):
            whole = torch.full((m * L + 16,), 777.0, device="cuda")
            out = whole[8 + lead:8 + lead + m * L]
            G.opmm_simulate(ctx, opc, batch, sac_index=np.zeros(m, np.int32), out=out)
            rows = out.cpu().numpy().reshape(m, L)
            np.testing.assert_array_equal(rows, np.tile(rows[0], (m, 1)))
            assert np.abs(rows[0] - ref).max() <= 1e-4
            assert (whole[:8 + lead] == 777.0).all() and (whole[8 + lead + m * L:] == 777.0).all()
    finally:
        G.opmm_destroy(ctx)


def test_writing_a_long_row_does_not_outweigh_its_walk():
    """One vector over 16,384 samples: its trajectory takes the walk's time, as
    its objective does (both one thread; the fastest of 20 calls each).  Stores
    that cost as much as the walk again would show as a factor above two."""
    import time
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    L = 16384
    opc = torch.from_numpy(np.float32(O.nominal_opc(10.0, 43.0, calibrated=False))[None]).cuda()
    batch = G.make_batch(torch.zeros(L, device="cuda"), [1000.0], [10], [0.0], [10.0], [43.0], n_samples=[L], offsets=[0])
    out, f = torch.zeros(L, device="cuda"), torch.zeros(1, device="cuda")
    ctx = G.opmm_create(0)

    def fastest(call):
        best = np.inf
        for _ in range(22):
            t = time.perf_counter()
            call()
            best = min(best, time.perf_counter() - t)
        return best

    try:
        assert fastest(lambda: G.opmm_simulate(ctx, opc, batch, out=out)) <= 1.7 * fastest(
            lambda: G.opmm_score(ctx, opc, batch, out=f))
    finally:
        G.opmm_destroy(ctx)
