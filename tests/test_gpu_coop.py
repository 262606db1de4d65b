"""Several warps per query (small batches) against one warp per query.

A batch too small to fill the GPU runs the cooperative kernel form: the exact
rows of an expansion are shared by the block's warps.  Every row's sum keeps its
order, so ids, distances and counters must be bit-identical to the same queries
inside a batch large enough for one warp per query.  Sizes: one query, and both
sides of each change of block width (2, 4 and 8 queries per SM)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MODES = ("PLAIN", "FINGER", "FINGER_F16", "FINGER_F8", "FINGER_LP")


@pytest.mark.parametrize("m,M,r", [(20, 4, 5), (100, 24, 32), (300, 8, 40), (960, 32, 64)])
@pytest.mark.parametrize("mode", MODES)
def test_small_batches_equal_the_large_one(m, M, r, mode):
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(m)
    X = rng.standard_normal((1500, m)).astype(np.float32)
    ix = fg.Index(X)
    ix.build_graph(M, candidates=max(M, 40), level_seed=5)
    if mode != "PLAIN":
        ix.build_tables(r, 6, half_codes=mode == "FINGER_F16", fp8_codes=mode == "FINGER_F8",
                        build_lp=mode == "FINGER_LP")
    ix.set_mode(getattr(fg, "MODE_" + mode), 5)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    total = 16 * sms + 5
    q = torch.from_numpy((X[rng.integers(0, 1500, total)] +
                          0.5 * rng.standard_normal((total, m))).astype(np.float32)).cuda()

    def search(lo, hi, K, ef):
        cnt = torch.zeros((hi - lo, 8), dtype=torch.int32, device="cuda")
        ix.set_counters(cnt)
        ids, d = ix.search(q[lo:hi].contiguous(), K, ef)
        ix.sync()
        ix.set_counters(None)
        return ids, d, cnt

    for K, ef in ((1, 1), (10, 37), (100, 150)):
        whole = search(0, total, K, ef)
        for nq in (1, 2 * sms - 1, 2 * sms + 1, 4 * sms + 1, 8 * sms - 3):
            part = search(total - nq, total, K, ef)
            for a, b in zip(whole, part):
                assert torch.equal(a[total - nq:], b), (K, ef, nq)
        # an uneven batch of the same queries
        nq = 2 * sms + 1
        Ks = torch.full((nq,), K, dtype=torch.int32, device="cuda")
        efs = torch.full((nq,), ef, dtype=torch.int32, device="cuda")
        if mode != "FINGER_LP":   # (its re-ranked head differs between the two calls)
            ids, d, _ = ix.search_batch(q[:nq].contiguous(), Ks, efs, max_ef=ef)
            assert torch.equal(ids.view(nq, K), whole[0][:nq])
            assert torch.equal(d.view(nq, K), whole[1][:nq])
    ix.close()
