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


@pytest.mark.parametrize("K", [10, 100])
def test_largest_error_of_the_parts(K):
    """The product of both operands' low parts, which is left out, at its largest: nearly
    2^-16 of |q| |x|.  The rows it moves away are the nearest all the same."""
    import torch

    import paper_2206_11408_gb300 as fg

    # a: high part 1, low part just under 2^-8.  Rows along a query a (A) lose the product of
    # the low parts, 1.5e-5, so that their approximate distance is 3.03e-5 too large; rows
    # at 1 lose nothing.  B: the next nearest, just behind A; C: where A appears to be
    a = np.float32(1 + 2.0 ** -8 - 2.0 ** -16)
    rng = np.random.default_rng(K)
    n = 20_000
    X = np.zeros((n, 16), np.float32)
    X[:, 0] = 0.5
    at = rng.permutation(n)[:300]
    A, B, C = at[:100], at[100:200], at[200:]
    own = float(a - 1) ** 2
    X[A, 0], X[A, 1] = a, np.sqrt(2.01e-5 + 1e-8 * np.arange(100))
    X[B, 0], X[B, 1] = 1, np.sqrt(2.31e-5 - own + 5e-9 * np.arange(100))
    X[C, 0], X[C, 1] = 1, np.sqrt(4.99e-5 - own + 1e-9 * np.arange(100))
    Q = np.zeros((3, 16), np.float32)
    Q[:, 0] = a
    ix = fg.Index(X)
    ids, d = ix.knn(torch.from_numpy(Q).cuda(), K)
    ix.sync()
    ix.close()
    check(X, Q, K, ids, d)


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


def test_roundings_of_long_rows():
    """A zero query over rows of 960 values: the norms' sums and the FP32 kernel's sums (one
    addition after the other) differ by hundreds of roundings, more than the distances by
    which a merge of K > 40 is decided.  Rows whose many small values vanish behind a large
    first one there are nearest by its sums, 1e-3 farther by the norms' (4,000 rows take that
    kernel whole, 5,000 the merge: the same results)."""
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(1)
    X = np.zeros((5000, 960), np.float32)
    X[:, 0] = 6.2 + 1e-5 * np.arange(5000)
    at = rng.permutation(4000)[:210]
    X[at[:40], 0] = np.sqrt(32.0)
    X[at[:40], 1:] = np.sqrt(1.8e-6)
    X[at[40:150], 0] = np.sqrt(32.0005)
    X[at[150:], 0] = np.sqrt(32.0015)
    Q = torch.zeros(2, 960, device="cuda")
    out = []
    for n in (4000, 5000):
        ix = fg.Index(X[:n])
        out.append(ix.knn(Q, 100))
        ix.sync()
        ix.close()
    assert set(out[0][0][0].cpu().tolist()[:40]) == set(at[:40].tolist())
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
