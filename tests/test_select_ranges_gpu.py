"""The selection's histogram levels, its ranking and its ties, and the pruning."""
import pytest
import torch

from oracle import scalekv_oracle as orc
from paper_2505_19602_b200 import binding
from parity_util import ParityRun

pytestmark = pytest.mark.gpu


def levels_inputs(B, H, d, n, distinct, seed):
    """Queries of one direction and keys with `distinct` different products with it (1: every entry ties with every other)."""
    def fn(layer, scale):
        g = torch.Generator().manual_seed(seed * 100 + scale)
        Q = torch.zeros(B, H, n[scale], d)
        Q[..., 0] = 1.0
        K = 0.1 * torch.randn(B, H, n[scale], d, generator=g)
        K[..., 0] = torch.randint(0, distinct, (B, H, n[scale]), generator=g).float() * 0.25
        V = torch.randn(B, H, n[scale], d, generator=g)
        return tuple(t.to(torch.bfloat16) for t in (Q, K, V))
    return fn


@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("heads", [1, 17])
@pytest.mark.parametrize("distinct,budget", [
    (1, 1),        # all keys equal, more of them than there are threads: the last level runs out of bits
    (1, 700),
    (2, 900),      # two keys: whole bins stay, or the tie runs through one
    (300, 500),    # a bin with repeated keys, ranked
])
def test_ties_at_every_level(distinct, budget, heads, separate):
    sides = (2, 40, 13)
    n = orc.scale_token_counts(sides)
    budgets = [[budget] * len(sides)]
    kv = binding.ScaleKV(1, 1, heads, 128, "bf16", sides, sides, budgets)
    run = ParityRun(kv, "bf16", sides, budgets, levels_inputs(1, heads, 128, n, distinct, 3),
                    lambda k: orc.window_centroids(sides[k], sides[k], 16), sorted({(0, 0, 0), (0, 0, heads - 1)}), compress_last=True,
                    max_rows=32)
    run.separate_kernels = separate
    run.run()
    assert run.resyncs == 0 and run.evictions >= 2
    kv.close()


@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("distinct", [3, 4096])           # ties through the whole slice; hardly any
@pytest.mark.parametrize("entries,budget", [
    (127, 60), (128, 60), (129, 60),                       # every key ranked against all, up to 128 entries
    (128, 0), (128, 112), (40, 23),                        # nothing but the window; all but none; a block mostly idle
    (700, 112), (700, 113),                                # 128 and 129 rows: one chunk of the gather, and one row more
    (1200, 496), (1200, 497),                              # 512 and 513: one round of look-ups, and one row more
])
def test_edges_of_ranking_and_gather(entries, budget, distinct, separate):
    n = [24, entries - 24, 1]
    budgets = [[binding.KEEP_ALL, budget, binding.KEEP_ALL]]
    window = list(range(0, n[1], max(1, n[1] // 16)))[:16]
    kv = binding.ScaleKV(1, 1, 3, 128, "bf16", [1, 1, 1], n, budgets)
    run = ParityRun(kv, "bf16", [1, 1, 1], budgets, levels_inputs(1, 3, 128, n, distinct, entries),
                    lambda k: window if k == 1 else [0], [(0, 0, 0), (0, 0, 2)], max_rows=16, sides_w=n)
    run.separate_kernels = separate
    run.run()
    assert run.resyncs == 0
    kv.close()


@pytest.mark.parametrize("heads", [2, 17])
@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("budget", [5, 129, 2100])         # around the sinks, a chunk of rows, everything but a few
def test_positional_rule_over_long_slices(budget, separate, heads):
    sides = (20, 42, 3)
    n = orc.scale_token_counts(sides)
    budgets = [[budget] * len(sides)]
    g = torch.Generator().manual_seed(8)
    data = [tuple(torch.randn(1, heads, nk, 128, generator=g).to(torch.bfloat16) for _ in range(3)) for nk in n]
    kv = binding.ScaleKV(1, 1, heads, 128, "bf16", sides, sides, budgets)
    run = ParityRun(kv, "bf16", sides, budgets, lambda l, k: data[k], lambda k: None, sorted({(0, 0, 0), (0, 0, heads - 1)}),
                    compress_last=True, max_rows=16)
    run.policy, run.n_sink, run.separate_kernels = "recent", 4, separate
    run.run()
    kv.close()


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f32", 64)])
@pytest.mark.parametrize("how", ["skipped", "sinks"])
def test_slices_longer_than_their_budgets_lead_to(how, dtype, d):
    """Pages hold more than the budgets' plan needs, and append accepts what they hold: the first scale is never compressed, or its
    100 sinks outnumber the budget of 10."""
    sides, page = (10, 11, 4), 512
    n = orc.scale_token_counts(sides)
    budgets = [[10] * len(sides)]
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator().manual_seed(41)
    kv = binding.ScaleKV(1, 1, 2, d, dtype, sides, sides, budgets, page_tokens=page)
    caches = [orc.SliceCache(n, d) for _ in range(2)]
    for k, nk in enumerate(n):
        Q, K, V = (torch.randn(1, 2, nk, d, generator=g).to(dt) for _ in range(3))
        Qd, Kd, Vd = Q.cuda(), K.cuda(), V.cuda()
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, Kd, Vd)
        O = kv.scalekv_attend(0, Qd)
        window = orc.window_centroids(sides[k], sides[k], 16)
        if k > 0:
            kv.scalekv_compress(0, Qd, window, qw_is_full_map=True)
        elif how == "sinks":
            kv.scalekv_compress_ex(0, Qd, policy="recent", n_sink=100)      # all of them: nothing is evicted
        kv.scalekv_sync()
        for h in range(2):
            c = caches[h]
            c.append(K[0, h].double().numpy(), V[0, h].double().numpy())
            want, _ = c.attend(Q[0, h].double().numpy())
            assert abs(want - O[0, h].double().cpu().numpy()).max() <= (2e-2 if dtype == "bf16" else 1e-4)
            if k > 0:
                pos, _ = c.compress(Q[0, h].double().numpy()[window], window, budgets[0][k])
                assert (kv.scalekv_export_slice(0, 0, h).numpy() == pos).all()
    kv.close()
