"""Training data of batches around the number of saccades that the features'
blocks take at once (two blocks of four warps on each of 152 SMs: 1,216): a
warp's later turns give each sample what a small batch gives it.

Tolerance: as for the halves of a batch in test_gpu_features_edges.py: losses
are sums of the same FP32 terms in other orders, 1e-5 relative."""
import pytest

import paper_2007_09884_gb300 as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1152, 1280, 2432, 2560, 4096])
def test_later_turns_give_the_same_samples(batch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = G.opmm_create(0)
    try:
        def first_loss(n, at):
            G.opmm_surrogate_init(ctx, 3)
            return float(G.opmm_surrogate_train(ctx, 1, batch=n, sample_base=at)[0])

        whole = first_loss(batch, 512)
        parts = [first_loss(128, 512 + at) for at in range(0, batch, 128)]
        assert abs(whole - sum(parts) / len(parts)) <= 1e-5 * whole
        assert max(parts) - min(parts) > 1e-3 * whole      # samples differ: a repeated or missed turn would show
    finally:
        G.opmm_destroy(ctx)
