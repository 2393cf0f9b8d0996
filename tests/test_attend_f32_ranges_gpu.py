"""The f32 attention at the edges of its tiles and of its key splits."""
import pytest
import torch

from oracle import scalekv_oracle as orc
from paper_2505_19602_b200 import binding
from parity_util import ParityRun

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,heads,sides,budget", [
    (1, 1, (1, 8, 9, 23), 30),           # 64 and 65 rows of keys and queries; clusters of two to five CTAs
    (1, 1, (2, 22), -1),                 # eight key tiles: clusters of eight
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


@pytest.mark.parametrize("heads", [1, 40])             # keys shared by a cluster, and not
def test_f32_rows_of_scores_near_the_lowest_number(heads):
    """Every score near the type's lowest value: they differ by less than it resolves, so all keys weigh the same."""
    sides = (3, 17)
    g = torch.Generator(device="cuda").manual_seed(7)
    kv = binding.ScaleKV(1, 1, heads, 64, "f32", sides, sides, [[binding.KEEP_ALL] * len(sides)])
    values = []
    for k, a in enumerate(sides):
        Q, K, V = (torch.randn(1, heads, a * a, 64, generator=g, device="cuda") for _ in range(3))
        Q[..., 0], K[..., 0] = 1.0, -3e38
        values.append(V)
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, K, V)
        O = kv.scalekv_attend(0, Q)
        kv.scalekv_sync()
        want = torch.cat(values, 2).mean(2, keepdim=True)
        assert (O - want).abs().max().item() <= 1e-5
    kv.close()


@pytest.mark.parametrize("heads", [2, 40])
def test_f32_log_sum_exp_is_rounded_twice(heads):
    """lse lies in [4, 8) and so does the logarithm of the sum, its largest part: two roundings of 2^-21 / sqrt(12) rms make 1.95e-7.  A
    third, or one of numbers above 8, would show: 3e-7 where the logarithm is taken to base 2 and converted."""
    sides = (5, 40)
    g = torch.Generator(device="cuda").manual_seed(9)
    kv = binding.ScaleKV(1, 1, heads, 64, "f32", sides, sides, [[binding.KEEP_ALL] * len(sides)])
    keys = []
    for k, a in enumerate(sides):
        Q, K, V = (torch.randn(1, heads, a * a, 64, generator=g, device="cuda") for _ in range(3))
        Q *= 0.25
        keys.append(K)
        lse = torch.empty(1, heads, a * a, device="cuda")
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, K, V)
        kv.scalekv_attend(0, Q, lse=lse)
        kv.scalekv_sync()
    want = (Q.double() @ torch.cat(keys, 2).double().transpose(2, 3) / 8).logsumexp(-1)
    assert 4 < want.min().item() and want.max().item() < 8
    assert (lse.double() - want).pow(2).mean().sqrt().item() <= 2.4e-7
    kv.close()


@pytest.mark.parametrize("heads", [1, 40])
@pytest.mark.parametrize("key", [-2.0 ** 33, -1.125 * 2.0 ** 33, 1.125 * 2.0 ** 33, -2.0 ** 40, -2.0 ** 100])
def test_f32_rows_of_equal_scores_far_from_zero(heads, key):
    """Equal scores, exact in 32 bits: equal weights, however far from zero they lie, to the roundings of sums over 340 values."""
    sides = (4, 18)
    g = torch.Generator(device="cuda").manual_seed(13)
    kv = binding.ScaleKV(1, 1, heads, 64, "f32", sides, sides, [[binding.KEEP_ALL] * len(sides)])
    values = []
    for k, a in enumerate(sides):
        Q, K, V = (torch.randn(1, heads, a * a, 64, generator=g, device="cuda") for _ in range(3))
        Q[...], K[..., 0] = 0.0, key
        Q[..., 0] = 1.0
        values.append(V)
        lse = torch.empty(1, heads, a * a, device="cuda")
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, K, V)
        O = kv.scalekv_attend(0, Q, lse=lse)
        kv.scalekv_sync()
    want = torch.cat(values, 2).double().mean(2, keepdim=True)
    # means of size 1/18 of values of size 1, whose sums are rounded by a few 2^-24 of their size: 2e-7 sqrt(a few) of the means
    assert ((O.double() - want).norm() / (O.shape[2] ** 0.5 * want.norm())).item() <= 2e-6
    assert (lse.double() - (key / 8 + torch.log(torch.tensor(340.0, dtype=torch.float64)).item())).abs().max().item() <= abs(key) / 8 * 2e-7 + 1e-6
    kv.close()


@pytest.mark.parametrize("batch,heads,hist,n", [
    (1, 3, 300, 1),            # one block of queries, more key tiles than that: rows of the grid behind the slices'
    (1, 3, 70, 129),           # a last row of the grid that is not full
    (2, 40, 500, 300),         # clusters of none, more CTAs than SMs
    (128, 128, 300, 1),        # more rows than a grid has: the compress scores from K
])
def test_window_logits_behind_the_slices(batch, heads, hist, n):
    sides_w, budget = [hist, n, 1], 40
    kv = binding.ScaleKV(1, batch, heads, 64, "f32", [1, 1, 1], sides_w, [[binding.KEEP_ALL, budget, binding.KEEP_ALL]], window_patches=16,
                         window_kind="last")
    g = torch.Generator().manual_seed(hist + n)
    slices = sorted({(0, 0), (batch - 1, heads - 1), (batch // 2, heads // 2)})
    caches = {s: orc.SliceCache(sides_w, 64) for s in slices}
    for k, nk in enumerate(sides_w):
        base = [torch.randn(1, 3, nk, 64, generator=g) for _ in range(3)]          # head h of any image has what head h mod 3 has here
        Q, K, V = (x.cuda()[:, torch.arange(heads) % 3].repeat(batch, 1, 1, 1) for x in base)
        O = torch.empty_like(Q)
        window = list(range(max(0, nk - 16), nk))
        torch.cuda.synchronize()
        kv.scalekv_step(0, k, Q, K, V, O, window_pos=window if k == 1 else None)
        kv.scalekv_sync()
        for b, h in slices:
            q, key, value = (x[0, h % 3].double().numpy() for x in base)
            caches[b, h].append(key, value)
            want, _ = caches[b, h].attend(q)
            assert abs(want - O[b, h].double().cpu().numpy()).max() <= 1e-4
            if k == 1:
                pos, _ = caches[b, h].compress(q[window], window, budget)
                assert (kv.scalekv_export_slice(0, b, h).numpy() == pos).all()
    kv.close()
