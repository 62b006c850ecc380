"""The featurizer at the edges of its launch (part blocks of one saccade per
warp; windows shorter than a warp and longer than the features reach; high and
low rates), and the training data's noisy form of it.

Tolerances: a feature as in test_gpu_surrogate.py (half a BF16 ulp, a sample
position off by 1e-4 samples, growing with the rate: eps (onset + 256 fs/1000)
stays below that up to 2 kHz).  A training loss is a sum of batch x 18 FP32
squares in a fixed order; the loss of 256 rows and the mean of the losses of
its halves differ by that order alone: 256 x 18 x 2^-24 = 2.7e-4 at worst, a
few 1e-6 in practice; 1e-5 is asked."""
import numpy as np
import pytest

import paper_2007_09884_gb300 as G
from _support import to_batch
from oracle import features as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    h = G.opmm_create(0)
    yield h
    G.opmm_destroy(h)


@pytest.mark.parametrize("n", [1, 3, 4, 5, 130])
def test_features_of_part_blocks(ctx, n):
    rng = np.random.default_rng(n)
    items = []
    for i in range(n):
        fs = (100.0, 250.0, 1000.0, 2000.0)[i % 4]
        L = (8, 31, 257, 1201)[(i // 4 + i) % 4]
        onset = min(3, L - 2)
        th0, A, sg = float(np.float32(rng.uniform(-10, 10))), float(np.float32(rng.uniform(0.2, 20))), (1.0, -1.0)[i & 1]
        ramp = np.clip(np.arange(L) - onset, 0, None) / max(1, L - onset)
        y = np.float32(th0 + sg * A * ramp + rng.normal(0, 0.05, L))
        items.append(dict(y=y, L=L, fs=fs, onset=onset, th0=th0, thf=float(np.float32(th0 + sg * A)), dur=30.0))
    got = G.opmm_featurize(ctx, to_batch(items))
    for j, it in enumerate(items):
        y = it["y"].astype(np.float64)
        ref = F.featurize(y, it["fs"], it["onset"], it["th0"], it["thf"])
        amp = max(abs(it["thf"] - it["th0"]), 0.5)
        d_pos = (1e-4 * np.abs(np.diff(y)).max() + 8 * 2.0 ** -24 * (np.abs(y).max() + abs(it["th0"]))) / amp
        tol = 2.0 ** -8 * np.abs(ref) + 1.01 * np.concatenate([np.full(256, d_pos), np.full(256, 20 * d_pos)])
        assert np.all(np.abs(got[j] - ref) <= tol), j


@pytest.mark.parametrize("base", [0, 4096, 2 ** 33])
def test_training_data_depend_on_the_sample_alone(ctx, base):
    def first_loss(batch, at):
        G.opmm_surrogate_init(ctx, 3)
        return float(G.opmm_surrogate_train(ctx, 1, batch=batch, sample_base=at)[0])

    whole = first_loss(256, base)
    halves = 0.5 * (first_loss(128, base) + first_loss(128, base + 128))
    assert whole > 0.0
    assert abs(whole - halves) <= 1e-5 * whole
