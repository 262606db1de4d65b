"""K <= 40 where the split products' error reaches over everything: the nearest all the same.

Rows far from the origin (their distances drown in the products' error), stored cluster by
cluster, so that one base segment holds all neighbours of a query and its list drops most of
them; batches of few long segments and of many short ones; norms that overflow, where no
approximate distance is finite; and a few such queries among ordinary ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def check(X, Q, K, ids, d):
    import torch

    x, q = torch.from_numpy(X).cuda().double(), torch.from_numpy(Q).cuda().double()
    for lo in range(0, len(Q), 64):
        got = torch.stack([((a - x[b]) ** 2).sum(1) for a, b in zip(q[lo:lo + 64], ids[lo:lo + 64])])
        ref = torch.stack([torch.topk(((a - x) ** 2).sum(1), K, largest=False)[0].sort()[0] for a in q[lo:lo + 64]])
        assert (ids[lo:lo + 64].sort(1)[0].diff(dim=1) > 0).all()
        torch.testing.assert_close(d[lo:lo + 64].double(), got, rtol=1e-5, atol=0)
        assert (d[lo:lo + 64].diff(dim=1) >= 0).all()
        torch.testing.assert_close(got.sort(1)[0], ref, rtol=1e-5, atol=0)


@pytest.mark.parametrize("K", [1, 10, 16, 17, 40])
@pytest.mark.parametrize("kind,n,nq", [("offset", 5000, 40), ("offset", 60_000, 2500), ("clusters", 60_000, 2500),
                                       ("clusters", 20_001, 3), ("overflow", 3000, 40), ("some", 60_000, 700),
                                       ("inf_row", 3000, 40)])
def test_nearest_by_their_own_differences(kind, n, nq, K):
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(n + nq)
    m = 33
    X = rng.standard_normal((n, m)).astype(np.float32)
    Q = rng.standard_normal((nq, m)).astype(np.float32)
    if kind == "offset":
        X += 3000
        Q += 3000
    elif kind == "clusters":   # runs of 500 rows around a centre
        X = (0.25 * X + 8 * rng.standard_normal((n // 500 + 1, m))[np.arange(n) // 500] + 2000).astype(np.float32)
        Q = (X[rng.integers(0, n, nq)] + 0.25 * Q).astype(np.float32)
    elif kind == "some":       # two of the queries, and the rows near them, lie far out
        X[1000:1900] += 5000
        Q[[3, 77]] += 5000
    elif kind == "inf_row":
        X[5, 5] = np.inf
        X[:, 0] += 1e19
        Q[:, 0] += 1e19
    else:
        X[:, 0] += 2e19
        Q[:, 0] += 2e19
    ix = fg.Index(X)
    for part in (Q, Q[:2]):
        ids, d = ix.knn(torch.from_numpy(part).cuda(), K)
        ix.sync()
        check(np.where(np.isinf(X), 1e30, X), part, K, ids, d)
    ix.close()


def test_fewer_rows_than_asked_for():
    import torch

    import paper_2206_11408_gb300 as fg

    X = np.full((7, 4), 3000, np.float32) + np.arange(7, dtype=np.float32)[:, None]
    X[2] = np.nan
    X[4, 1] = np.inf
    ix = fg.Index(X)
    ids, d = ix.knn(torch.from_numpy(X[[0, 5]]).cuda(), 10)
    ix.sync()
    assert ids.cpu().tolist() == [[0, 1, 3, 5, 6, -1, -1, -1, -1, -1], [5, 6, 3, 1, 0, -1, -1, -1, -1, -1]]
    assert d.cpu()[1].tolist() == [0, 4, 16, 64, 100] + [np.inf] * 5
    ix.close()
