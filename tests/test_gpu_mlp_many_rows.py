"""Predictions of more rows than the GPU has blocks for: a block goes on to further rows,
and every prediction has the bits it has in a small call."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 24, 64])
@pytest.mark.parametrize("rows", [38_913, 100_003, (1 << 20) + 33])
def test_many_rows_equal_few(r, rows):
    import torch

    import paper_2206_11408_gb300 as fg

    rng = np.random.default_rng(r)
    ix = fg.Index(rng.standard_normal((500, 64)).astype(np.float32))
    ix.build_graph(8, candidates=32, level_seed=3)
    ix.build_tables(r, 4)
    ix.set_predictor((0.2 * rng.standard_normal(ix.mlp_size())).astype(np.float32), 0.05)
    g = torch.Generator("cuda").manual_seed(rows)
    feat = torch.randn(rows, r + 4, device="cuda", generator=g)
    out = ix.mlp_predict(feat)
    for lo in (0, 1000, rows // 2, rows - 77):
        part = feat[lo:lo + 77].contiguous()
        assert torch.equal(out[lo:lo + 77], ix.mlp_predict(part))
    assert len(torch.unique(out)) > 0.5 * min(rows, 100_000)
    ix.close()
