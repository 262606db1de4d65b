"""kNN of so many queries that their lists take several passes: every query's result is
that of the one-pass call (small integers, exact)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,nq", [(3, 1_100_003), (20, 600_001)])
def test_passes(K, nq):
    import torch

    import paper_2206_11408_gb300 as fg

    g = torch.Generator("cuda").manual_seed(K)
    n = 300
    X = torch.randint(0, 6, (n, 5), device="cuda", generator=g).float()
    Q = torch.randint(0, 6, (nq, 5), device="cuda", generator=g).float()
    ix = fg.Index(X.cpu().numpy())
    ids, d = ix.knn(Q, K)
    ix.sync()
    for lo in range(0, nq, 1 << 17):
        q = Q[lo:lo + (1 << 17)]
        D = (q * q).sum(1)[:, None] + (X * X).sum(1)[None] - 2 * (q @ X.T)
        key = (D * 1024 + torch.arange(n, device="cuda")[None]).sort(1)[0][:, :K].long()
        assert torch.equal(ids[lo:lo + (1 << 17)], key % 1024)
        assert torch.equal(d[lo:lo + (1 << 17)], (key // 1024).float())
    ix.close()
