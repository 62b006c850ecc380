"""Detection at the edges of its groups of 512 runs: kept and dropped runs
mixed, counts around one and two groups.  Every field of every kept event is
that of the reference definition, exactly (the decisions are FP32 on both
sides)."""
import numpy as np
import pytest

import paper_2007_09884_gb300 as G
from oracle.ivt import ivt

pytestmark = pytest.mark.gpu

FIELDS = {"onset": "onset", "end": "end", "window_start": "window_start", "n_samples": "n_samples",
          "onset_index": "onset_index", "theta_start_deg": "theta_start", "theta_end_deg": "theta_end",
          "amplitude_deg": "amplitude", "duration_ms": "duration_ms", "peak_velocity_dps": "peak_velocity"}


@pytest.mark.parametrize("runs", [1, 2, 511, 512, 513, 1024, 1025])
@pytest.mark.parametrize("small", [0, 1, 7])       # every small-th movement stays below 4 deg (0: none, 1: all)
def test_kept_events_in_order(runs, small):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(runs + small)
    parts, pos = [np.zeros(20, np.float32)], 0.0
    for i in range(runs):
        step = (2.0 if small and i % small == 0 else rng.uniform(4.5, 12.0)) * (1 if pos < 0 else -1)
        parts.append(pos + step * np.arange(1, 13) / 12.0)     # 12 fast steps
        pos += step
        parts.append(np.full(int(rng.integers(45, 70)), pos))  # shorter than some windows need
    x = np.concatenate(parts).astype(np.float32)
    ctx = G.opmm_create(0)
    try:
        got = G.opmm_detect_saccades(ctx, torch.from_numpy(x).cuda(), 1000.0)
        first = G.opmm_detect_saccades(ctx, x, 1000.0, max_events=3)
    finally:
        G.opmm_destroy(ctx)
    want = ivt(x, 1000.0)
    assert len(got) == len(want)
    for name, ref in FIELDS.items():
        np.testing.assert_array_equal(got[name], np.array([w[ref] for w in want]).astype(got.dtype[name]), err_msg=name)
    np.testing.assert_array_equal(first, got[:3])
