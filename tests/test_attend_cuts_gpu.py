"""How the tensor-core attention cuts a launch: pairs of query tiles, single tiles whose keys the two warpgroups share, single
tiles whose keys a cluster of CTAs shares, and launches whose last items are worked on tile by tile (and the clusters of the f32
attention, where slices differ in length)."""
import pytest
import torch

from oracle import scalekv_oracle as orc
from paper_2505_19602_b200 import binding
from parity_util import ParityRun

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,heads,sides,budget", [
    (1, 1, (1, 11, 12, 16, 37), 40),       # one slice: clusters of two to six CTAs, rows that do not divide among them
    (1, 1, (2, 43), 40),                   # 16 key tiles: clusters of eight, 57 rows in the last tile
    (1, 3, (2, 16, 17, 29), -1),           # full cache: odd numbers of key tiles
    (1, 2, (1, 63), -1),                   # 31 tiles and one row
    (1, 16, (3, 9, 33), 70),               # 144 single tiles: every SM has one, nothing is left to split
    (7, 10, (2, 12, 25), 150),             # 70 slices x 5 tiles: 210 items, the last 62 tile by tile from inside a slice
    (5, 15, (1, 18), 25),                  # 75 slices x 3 tiles: 150 items, one whole slice tile by tile
    (6, 16, (2, 20), 30),                  # 96 slices x 4 tiles: 192 pairs, the last 44 tile by tile
    (4, 16, (1, 8, 20), 30),               # 64 slices x 4 tiles: 128 pairs, no more than one wave
    (4, 16, (2, 8, 11), -1),               # 64 single tiles with two key tiles: shared by the two warpgroups
    (5, 13, (2, 8, 11), -1),               # 65: one warpgroup takes both
])
def test_every_way_of_cutting_a_launch(batch, heads, sides, budget):
    n = orc.scale_token_counts(sides)
    B, H, d = batch, heads, 128
    gen = torch.Generator().manual_seed(91)
    data = [tuple(torch.randn(B, H, nk, d, generator=gen).to(torch.bfloat16) for _ in range(3)) for nk in n]
    slices = [(0, b, h) for b in range(B) for h in range(H)]
    followed = slices if len(slices) <= 3 else slices[:2] + slices[len(slices) * 2 // 3:][:2] + slices[-3:]
    for run in ("run", "run_pipelined"):   # with the map's rows copied by the attention kernel, and left to the compress
        budgets = [[budget] * len(sides)]
        kv = binding.ScaleKV(1, B, H, d, "bf16", sides, sides, budgets)
        p = ParityRun(kv, "bf16", sides, budgets, lambda l, k: data[k], lambda k: orc.window_centroids(sides[k], sides[k], 16),
                      followed, compress_last=True)
        getattr(p, run)()
        kv.close()


@pytest.mark.parametrize("batch,heads", [(1, 16), (4, 15), (8, 16)])      # clusters, singles, pairs
@pytest.mark.parametrize("first", [0, 128, 256])                          # the masked keys open a tile of the map: every part's first
def test_keys_masked_with_minus_infinity(first, batch, heads):
    """32 keys at the head of a tile whose products are -inf: no weight, whichever part of the keys starts with them."""
    sides, d = (8, 18), 128
    gen = torch.Generator(device="cuda").manual_seed(5)
    kv = binding.ScaleKV(1, batch, heads, d, "bf16", sides, sides, [[binding.KEEP_ALL] * len(sides)])
    keys, values = [], []
    for k, a in enumerate(sides):
        Q, K, V = (torch.randn(batch, heads, a * a, d, generator=gen, device="cuda", dtype=torch.bfloat16) for _ in range(3))
        Q[..., 0] = 1.0
        if k == 1:
            K[:, :, first: first + 32, 0] = -float("inf")
        keys.append(K), values.append(V)
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, K, V)
        O = kv.scalekv_attend(0, Q)
        kv.scalekv_sync()
        S = Q.double() @ torch.cat(keys, 2).double().transpose(2, 3) / d ** 0.5
        want = S.softmax(-1) @ torch.cat(values, 2).double()
        assert (O.double() - want).abs().max().item() <= 2e-2
    kv.close()


@pytest.mark.parametrize("dtype,d,tol", [("bf16", 128, 2e-2), ("f32", 64, 1e-4)])
def test_clusters_sized_for_a_longer_slice(dtype, d, tol):
    """Per-head budgets leave one head 49 times as long as the other; the launch is cut for the longer one, and most CTAs of the
    shorter one's clusters have no key tile."""
    sides, budgets, heads = (40, 3), [[1200] * 2], [1200, 0]
    n = orc.scale_token_counts(sides)
    g = torch.Generator().manual_seed(37)
    kv = binding.ScaleKV(1, 1, 2, d, dtype, sides, sides, budgets)
    caches = [orc.SliceCache(n, d) for _ in heads]
    for k, nk in enumerate(n):
        Q, K, V = (torch.randn(1, 2, nk, d, generator=g).to(kv.torch_dtype) for _ in range(3))
        Qd, Kd, Vd = Q.cuda(), K.cuda(), V.cuda()
        lse = torch.empty(1, 2, nk, device="cuda")
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, Kd, Vd)
        O = kv.scalekv_attend(0, Qd, lse=lse)
        if k == 0:
            kv.scalekv_compress_ex(0, Qd, orc.window_centroids(sides[0], sides[0], 16), qw_is_full_map=True, head_budgets=heads)
        kv.scalekv_sync()
        for h, c in enumerate(caches):
            c.append(K[0, h].double().numpy(), V[0, h].double().numpy())
            want, want_lse = c.attend(Q[0, h].double().numpy())
            assert abs(want - O[0, h].double().cpu().numpy()).max() <= tol
            assert abs(want_lse - lse[0, h].double().cpu().numpy()).max() <= 1e-4
            if k == 0:
                c.adopt_positions(kv.scalekv_export_slice(0, 0, h).numpy())
    assert [len(c) for c in caches] == [1216 + 9, 16 + 9]
    kv.close()
