"""Candidate lists, segments and merges of the tensor-core kNN at their edges.

Rows and queries are small integers, so distances are exact in BF16 split products
and in FP32 and many are equal: ids and distances must be exactly the K smallest
(distance, id) keys.  Sizes: around a tile (128 rows), fewer rows than K or than the
32 / 64 kept, queries around a query tile, one chunk of columns, two (the largest
resident query tile) and three."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [3, 64, 65, 128, 129])
@pytest.mark.parametrize("n", [5, 127, 128, 129, 1000, 20011])
def test_exact_keys_with_ties(n, m):
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(n + m)
    X = rng.integers(0, 4, (n, m)).astype(np.float32)
    Q = rng.integers(0, 4, (300, m)).astype(np.float32)
    D = ((Q[:, None].astype(np.int64) - X[None, :2000].astype(np.int64)) ** 2).sum(-1) if n <= 2000 else \
        (Q ** 2).sum(1).astype(np.int64)[:, None] + (X ** 2).sum(1).astype(np.int64)[None] - 2 * (Q @ X.T).astype(np.int64)
    order = np.argsort(D * (1 << 20) + np.arange(n)[None], axis=1, kind="stable")
    ix = fg.Index(X)
    for nq in (1, 127, 129, 300):
        for K in (1, 10, 16, 17, 40):
            ids, d = ix.knn(torch.from_numpy(Q[:nq]).cuda(), K)
            ix.sync()
            k = min(K, n)
            assert np.array_equal(ids.cpu().numpy()[:, :k], order[:nq, :k])
            assert np.array_equal(d.cpu().numpy()[:, :k], np.take_along_axis(D[:nq], order[:nq, :k], 1))
            assert (ids.cpu().numpy()[:, k:] == -1).all() and np.isinf(d.cpu().numpy()[:, k:]).all()
    ix.close()


@pytest.mark.parametrize("m", [24, 130])
@pytest.mark.parametrize("n", [4095, 4096, 20011])
@pytest.mark.parametrize("clustered", [False, True])
def test_large_k(n, m, clustered):
    """K > 40: lists of 64 per segment merged, and the queries whose neighbours fill one
    segment's list (rows in runs of 300 copies of a few points) done again."""
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(n + m)
    X = rng.integers(0, 5, (n, m)).astype(np.float32)
    if clustered:
        X = X[np.arange(n) // 300 * 300] + rng.integers(0, 2, (n, m)) * (np.arange(m) < 3)
        X = X.astype(np.float32)
    Q = X[rng.integers(0, n, 130)] + rng.integers(0, 2, (130, m)).astype(np.float32)
    D = (Q ** 2).sum(1).astype(np.int64)[:, None] + (X ** 2).sum(1).astype(np.int64)[None] - 2 * (Q @ X.T).astype(np.int64)
    order = np.argsort(D * (1 << 20) + np.arange(n)[None], axis=1, kind="stable")
    ix = fg.Index(X)
    for nq, K in ((1, 41), (130, 100), (33, 256)):
        ids, d = ix.knn(torch.from_numpy(Q[:nq]).cuda(), K)
        ix.sync()
        assert np.array_equal(ids.cpu().numpy(), order[:nq, :K])
        assert np.array_equal(d.cpu().numpy(), np.take_along_axis(D[:nq], order[:nq, :K], 1))
    ix.close()


@pytest.mark.parametrize("candidates", [40, 64])
def test_graph_of_bounded_segments(candidates):
    """From 4 query tiles per SM on, the first segments' lists bound the later ones.  Up to
    64 candidates no list can drop one, so on integer rows (exact products, many equal
    distances) the graph must be the one that the FP32 candidates give."""
    import torch

    import paper_2206_11408_gb300 as fg

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(candidates)
    X = rng.integers(0, 40, (4 * sms * 128 + 77, 6)).astype(np.float32)
    graphs = []
    for fp32 in (False, True):
        ix = fg.Index(X)
        ix.build_graph(8, candidates=candidates, level_seed=3, fp32_candidates=fp32)
        graphs.append(ix.get_graph())
        ix.close()
    for key in ("adj0", "up_adj", "up_off", "level"):
        assert np.array_equal(graphs[0][key], graphs[1][key]), key


@pytest.mark.parametrize("kind,K", [("near", 10), ("near", 16), ("near", 40), ("near", 100),
                                    ("offset", 100), ("inf_query", 100), ("inf_row", 100),
                                    ("overflow", 100)])
def test_where_the_products_decide_little(kind, K):
    """Rows away from the origin: the split products' error reaches over the kept keys
    ("near": their order alone; "offset": everything); infinities; norms that overflow.
    The nearest by the rows' own FP32 differences all the same."""
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(5)
    X = rng.standard_normal((5000, 32)).astype(np.float32)
    Q = rng.standard_normal((40, 32)).astype(np.float32)
    if kind in ("near", "offset"):
        X += 60 if kind == "near" else 3000
        Q += 60 if kind == "near" else 3000
    elif kind == "inf_query":
        Q[3, 4] = np.inf
    elif kind == "inf_row":
        X[77, 2] = np.inf
    else:
        X[:, 0] += 2e19
        Q[:, 0] += 2e19
    ix = fg.Index(X)
    ids, d = ix.knn(torch.from_numpy(Q).cuda(), K)
    ix.sync()
    ix.close()
    ids, d = ids.cpu().numpy(), d.cpu().numpy()
    for i in range(len(Q)):
        with np.errstate(over="ignore", invalid="ignore"):
            diff = (Q[i] - X).astype(np.float64)
            ref = (diff ** 2).sum(1)
        if np.isnan(ref).any() or np.isinf(ref).all():
            assert np.array_equal(ids[i], np.arange(K)) and np.isinf(d[i]).all()
            continue
        # every returned distance is the row's own, ascending, and none nearer is missing
        got = ref[ids[i]]
        np.testing.assert_allclose(d[i], got, rtol=1e-5)
        assert (np.diff(d[i]) >= 0).all() and len(set(ids[i])) == K
        assert np.sort(ref)[K - 1] >= got.max() * (1 - 1e-5)
