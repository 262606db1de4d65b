"""Long rows in the modes without codes: a smaller visited table where that brings a batch into
one wave of five blocks per SM.  The same queries in a small batch (several warps per query, the full table), with
32-bit slots, and tuned (any table size) give the same ids, distances and counters."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["PLAIN", "FINGER"])
@pytest.mark.parametrize("n,m,M", [(300, 1000, 8), (3000, 600, 32), (9000, 960, 32)])
def test_table_sizes_agree(mode, n, m, M):
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(m)
    X = rng.standard_normal((n, m)).astype(np.float32)
    ix = fg.Index(X)
    ix.build_graph(M, candidates=64, level_seed=5)
    if mode == "FINGER":
        ix.build_tables(16, 6)
    ix.set_mode(getattr(fg, "MODE_" + mode), 5)
    wave = 18 * torch.cuda.get_device_properties(0).multi_processor_count   # more than four blocks of 4
    q = torch.from_numpy((X[rng.integers(0, n, wave)] + rng.standard_normal((wave, m))).astype(np.float32)).cuda()

    def search(nq, ef):
        cnt = torch.zeros((nq, 8), dtype=torch.int32, device="cuda")
        ix.set_counters(cnt)
        out = ix.search(q[:nq].contiguous(), 10, ef)
        ix.sync()
        ix.set_counters(None)
        return (*out, cnt)

    for ef in (290, 320, 500, 560, 640, 700):
        whole = search(wave, ef)
        for a, b in zip(whole, search(100, ef)):
            assert torch.equal(a[:100], b), ef
        ix.set_visited_slots(32)
        for a, b in zip(whole, search(wave, ef)):
            assert torch.equal(a, b), ef
        ix.set_visited_slots(0)
    ix.autotune(q, 10, 500)
    for a, b in zip(search(wave, 500), search(100, 500)):
        assert torch.equal(a[:100], b)
    ix.close()
