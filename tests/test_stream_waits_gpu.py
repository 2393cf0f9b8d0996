"""Compresses that run beside later layers' attends: the same values, bit for bit, as with everything on one stream."""
import pytest
import torch

from oracle import scalekv_oracle as orc
from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu

SIDES = (2, 6, 12, 20, 24)


def _pass(budgets, heads, data, side_stream):
    n = orc.scale_token_counts(SIDES)
    kv = binding.ScaleKV(len(budgets), 1, heads, 128, "bf16", SIDES, SIDES, budgets, side_stream=side_stream)
    out = [[torch.empty_like(data[l][k][0]) for l in range(len(budgets))] for k in range(len(n))]
    torch.cuda.synchronize()
    for _ in range(2):                     # the second pass finds every layer's and every page set's last compress to wait for
        kv.scalekv_reset()
        for k in range(len(n)):
            window = orc.window_centroids(SIDES[k], SIDES[k], 16)
            for l in range(len(budgets)):
                kv.scalekv_step(l, k, *data[l][k], out[k][l], window_pos=window)
    kv.scalekv_join()
    kv.scalekv_sync()
    kv.close()
    return out


# budgets of the layers in turn (-1: nothing is evicted): fewer layers than page sets, one more, all sets twice over, layers of which
# some compress and some do not, so that the last compress of a layer and of its set's owner are near and far
@pytest.mark.parametrize("layers,budget_of", [(1, (40,)), (3, (40,)), (5, (40, 200)), (9, (40,)), (9, (40, -1, -1)), (8, (-1, 40, 40, -1))])
def test_overlapped_compresses_change_nothing(layers, budget_of):
    heads = 16
    budgets = [[budget_of[l % len(budget_of)]] * len(SIDES) for l in range(layers)]
    gen = torch.Generator(device="cuda").manual_seed(17)
    data = [[tuple(torch.randn(1, heads, nk, 128, generator=gen, device="cuda", dtype=torch.bfloat16) for _ in range(3))
             for nk in orc.scale_token_counts(SIDES)] for _ in range(layers)]
    beside, alone = (_pass(budgets, heads, data, s) for s in (True, False))
    for k in range(len(SIDES)):
        for l in range(layers):
            assert torch.equal(beside[k][l], alone[k][l]), (k, l)
