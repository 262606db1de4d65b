"""The 32-bit visited set at its fullest: tens of thousands of queries whose expansions add
up to 64 new ids at a time to a table of 512 or 1,024 slots that is nearly three quarters full.  No
node may be taken as new twice, so the counters equal those of the 16-bit set (other
buckets, other losses of the lanes' compare-and-swaps)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,ef", [(250, 32), (500, 64)])
def test_no_node_twice(m, ef):
    import torch

    import paper_2206_11408_gb300 as fg

    n = 9000
    rng = np.random.default_rng(m)
    X = rng.standard_normal((n, m)).astype(np.float32)   # (no clusters: 64 links to most nodes)
    ix = fg.Index(X)
    ix.build_graph(32, candidates=64, level_seed=5)
    ix.set_mode(fg.MODE_PLAIN, 5)
    g = torch.Generator("cuda").manual_seed(m)
    x = torch.from_numpy(X).cuda()
    q = x[torch.randint(0, n, (40_000,), device="cuda", generator=g)] + torch.randn(40_000, m, device="cuda", generator=g)

    def search(bits):
        ix.set_visited_slots(bits)
        cnt = torch.zeros((len(q), 8), dtype=torch.int32, device="cuda")
        ix.set_counters(cnt)
        out = ix.search(q, ef, ef)
        ix.sync()
        ix.set_counters(None)
        return (*out, cnt)

    a, b = search(0), search(32)
    assert (b[0].sort(1)[0].diff(dim=1) > 0).all()
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    ix.close()
