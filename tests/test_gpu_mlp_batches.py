"""Training kernels at the edges of their tiles: batches around 32 rows (a block of the
forward / backward kernel), 128 rows (a stage of the weight sums) and multiples of 4 (its
16-byte copies), input counts around the 16-wide weight tiles, the largest of 68 and 96
inputs.  Loss and gradient against the FP64 oracle on the same BF16 weights.  A hidden
activation that FP32 and FP64 round to different BF16 neighbours differs by 2^-8 of
itself, so the gradient may by at most about that: relative 2-norm error below 4e-3."""
import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nf", [5, 15, 16, 28, 68, 96])
@pytest.mark.parametrize("n", [1, 3, 31, 33, 127, 130, 1000])
def test_loss_and_gradient(nf, n):
    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(nf * 1000 + n)
    ix = fg.Index(rng.standard_normal((64, 8)).astype(np.float32))
    w = mlp.quantize_weights(mlp.init(nf, 11) + rng.normal(0, 0.02, mlp.n_weights(nf)), nf)
    X = rng.standard_normal((n, nf)).astype(np.float32)
    T = rng.uniform(-1, 1, n).astype(np.float32)
    loss, g = ix.mlp_loss_grad(w.astype(np.float32), torch.from_numpy(X).cuda(),
                               torch.from_numpy(T).cuda())
    ol, og = mlp.loss_and_grad(w, X.astype(np.float64), T.astype(np.float64), nf, True)
    assert loss == pytest.approx(ol, rel=4e-3)
    assert np.linalg.norm(g - og) <= 4e-3 * np.linalg.norm(og)
    ix.close()
