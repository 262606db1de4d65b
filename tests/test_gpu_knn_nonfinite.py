"""Exact kNN over a base with rows that are nobody's neighbour: NaN, infinite, or with a
norm that overflows.  Every other row ranks as if they were not there, for every query
(a zero query and queries that are not finite themselves among them).

Integer rows: distances are exact, so ids and distances must be exactly the K smallest
(distance, id) keys."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["nan_row", "nan_rows", "inf_row", "overflow_row", "all"])
@pytest.mark.parametrize("n,nq", [(5000, 40), (20011, 300)])
def test_other_rows_rank_as_without_them(kind, n, nq):
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(n)
    X = rng.integers(-3, 4, (n, 32)).astype(np.float32)
    Q = rng.integers(-3, 4, (nq, 32)).astype(np.float32)
    Q[1] = 0
    D = ((Q ** 2).sum(1)[:, None] + (X ** 2).sum(1)[None] - 2 * (Q @ X.T)).astype(np.int64)
    ok = np.ones(n, bool)
    if kind in ("nan_row", "all"):
        X[77, 3] = np.nan
        ok[77] = False
    if kind == "nan_rows":
        X[::3] = np.nan
        ok[::3] = False
    if kind in ("inf_row", "all"):
        X[200, 2] = -np.inf
        ok[200] = False
    if kind in ("overflow_row", "all"):
        X[n - 5] = 1e20
        ok[n - 5] = False
    order = np.argsort(np.where(ok, D, 1 << 30) * (1 << 20) + np.arange(n)[None], axis=1, kind="stable")
    Qn = Q.copy()
    Qn[5, 7] = np.nan
    Qn[6, 0] = np.inf
    ix = fg.Index(X)
    for K in (1, 10, 16, 17, 40, 41, 100):
        ids, d = ix.knn(torch.from_numpy(Q).cuda(), K)
        assert np.array_equal(ids.cpu().numpy(), order[:, :K]), K
        assert np.array_equal(d.cpu().numpy(), np.take_along_axis(D, order[:, :K], 1)), K
        ids, d = ix.knn(torch.from_numpy(Qn).cuda(), K)
        ids, d = ids.cpu().numpy(), d.cpu().numpy()
        rest = np.r_[0:5, 7:nq]
        assert np.array_equal(ids[rest], order[rest, :K]), K
        assert np.isinf(d[5:7]).all()
        assert (ids[5] == -1).all()
    ix.sync()
    ix.close()
