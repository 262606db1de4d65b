"""Link selection on both sides of the row length where its kernel changes (256 floats): the
graph is that of the candidates' own definition, computed on the host.

Integer rows with many equal distances, so that every distance is exact and the order of
candidates and the selection's strict comparison are decided by it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [255, 256, 257, 512, 513, 960, 1024])
def test_flat_graph(m):
    import paper_2206_11408_gb300 as fg

    n, M, cand = 300, 6, 40
    rng = np.random.default_rng(m)
    X = (rng.integers(0, 3, (n, m)) * (rng.random((n, m)) < 0.05)).astype(np.float32)
    D = ((X[:, None].astype(np.int64) - X[None].astype(np.int64)) ** 2).sum(-1)
    ix = fg.Index(X)
    ix.build_graph(M, candidates=cand, level_seed=1, flat=True, symmetric=True, fp32_candidates=True)
    adj = ix.get_graph()["adj0"]
    ix.close()
    order = np.argsort(D * 4096 + np.arange(n)[None] + (1 << 40) * np.eye(n, dtype=np.int64), axis=1)[:, :cand]

    def select(i, cands, limit):
        kept = []
        for c in cands:
            if len(kept) == limit:
                break
            if all(D[i, c] < D[c, k] for k in kept):
                kept.append(int(c))
        return kept

    fwd = [select(i, order[i], M) for i in range(n)]
    into = [[] for _ in range(n)]
    for i, f in enumerate(fwd):
        for c in f:
            into[c].append(i)
    for i in range(n):
        cands = sorted(set(fwd[i]) | set(into[i]), key=lambda c: (D[i, c], c))
        if len(into[i]) <= 64:   # (more reverse links than that: the closest are considered)
            assert [c for c in adj[i] if c >= 0] == select(i, cands, adj.shape[1]), i
