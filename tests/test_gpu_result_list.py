"""The unsorted result list against the oracle at the sizes where its scans change.

A scan covers 32 entries per step and 160 per round, so ef takes the values on both
sides of those; rows are small integers, so distances are exact in FP32 and many
are equal, which leaves the order to the ids: ids and distances must equal the
oracle's exactly."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def integer_index():
    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(11)
    X = rng.integers(0, 6, (3000, 24)).astype(np.float32)
    Q = rng.integers(0, 6, (40, 24)).astype(np.float32)
    g = oracle.hnsw_build(X, 8, 60, 21)
    ix = fg.Index(X)
    ix.set_graph(g.adj0, g.level, g.up_off, g.up_adj, g.entry, g.maxlevel, g.M)
    yield ix, g, X, Q
    ix.close()


@pytest.mark.parametrize("ef", [1, 2, 31, 32, 33, 159, 160, 161, 320, 321, 1024])
def test_ties_and_scan_edges(integer_index, ef):
    import torch

    import paper_2206_11408_gb300 as fg

    ix, g, X, Q = integer_index
    ix.set_mode(fg.MODE_PLAIN, 5)
    for K in sorted({1, min(33, ef), ef}):
        cnt = torch.zeros((len(Q), 8), dtype=torch.int32, device="cuda")
        ix.set_counters(cnt)
        ids, d = ix.search(torch.from_numpy(Q).cuda(), K, ef)
        ix.sync()
        ix.set_counters(None)
        oi, od, oc = oracle.search(g, X, Q, K, ef, None)
        assert np.array_equal(ids.cpu().numpy(), oi)
        assert np.array_equal(d.cpu().numpy(), od.astype(np.float32))
        assert np.array_equal(cnt.cpu().numpy()[:, :7], np.asarray(oc)[:, :7])
