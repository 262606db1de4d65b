"""Output of many keys: from 64 on the result list is sorted instead of scanned once per key.

A small base that a search reaches whole (ef above its size, so no gate): the output must be
all rows by exact (distance, id), then padding.  Integer rows with many equal distances;
sizes around the change and around powers of two; the reduced-precision mode ranks the
sorted head again by its FP32 rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["PLAIN", "FINGER_F16", "FINGER_LP"])
@pytest.mark.parametrize("n", [40, 63, 64, 65, 127, 129, 500, 1000])
def test_all_rows_in_order(n, mode):
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(n)
    X = rng.integers(0, 4, (n, 20)).astype(np.float32)
    Q = rng.integers(0, 4, (400, 20)).astype(np.float32)
    D = ((Q[:, None] - X[None]) ** 2).sum(-1).astype(np.int64)
    order = np.argsort(D * 4096 + np.arange(n)[None], axis=1)
    ix = fg.Index(X)
    ix.build_graph(24, candidates=min(n - 1, 200), level_seed=1)
    if mode != "PLAIN":
        ix.build_tables(8, 3, half_codes=mode == "FINGER_F16", build_lp=mode == "FINGER_LP")
    ix.set_mode(getattr(fg, "MODE_" + mode), 5)
    for K in sorted({32, 62, 63, 64, 65, n - 1, n, min(n + 7, 1024)}):
        ids, d = ix.search(torch.from_numpy(Q).cuda(), K, 1024)
        k = min(K, n)
        assert np.array_equal(ids.cpu().numpy()[:, :k], order[:, :k]), K
        assert np.array_equal(d.cpu().numpy()[:, :k], np.take_along_axis(D, order[:, :k], 1)), K
        assert (ids.cpu().numpy()[:, k:] == -1).all() and np.isinf(d.cpu().numpy()[:, k:]).all()
        one = ix.search(torch.from_numpy(Q[:1]).cuda(), K, 1024)   # (several warps per query)
        assert torch.equal(one[0], ids[:1]) and torch.equal(one[1], d[:1])
    ix.sync()
    ix.close()
