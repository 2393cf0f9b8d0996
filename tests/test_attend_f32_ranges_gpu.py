"""The f32 attention at the edges of its tiles and of its key splits."""
import pytest
import torch

from oracle import scalekv_oracle as orc
from paper_2505_19602_b200 import binding
from parity_util import ParityRun

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,heads,sides,budget", [
    (1, 1, (1, 8, 9, 23), 30),           # 64 and 65 rows of keys and queries; clusters of up to 8 CTAs, some without a tile
    (2, 3, (3, 16, 20), -1),             # full cache
    (4, 9, (2, 12, 27), 100),            # 36 slices: three CTAs per slice and tile of queries, then one
])
def test_f32_attention_matches_oracle(batch, heads, sides, budget):
    n = orc.scale_token_counts(sides)
    g = torch.Generator().manual_seed(23)
    data = [tuple(torch.randn(batch, heads, nk, 64, generator=g) for _ in range(3)) for nk in n]
    data = [(3.0 * Q, K, V) for Q, K, V in data]           # (rows that a few keys dominate)
    budgets = [[budget] * len(sides)]
    kv = binding.ScaleKV(1, batch, heads, 64, "f32", sides, sides, budgets)
    run = ParityRun(kv, "f32", sides, budgets, lambda l, k: data[k], lambda k: orc.window_centroids(sides[k], sides[k], 16),
                    sorted({(0, 0, 0), (0, batch - 1, heads - 1)}), compress_last=True).run()
    assert run.compared == len(sides) * len(run.slices)
    kv.close()
