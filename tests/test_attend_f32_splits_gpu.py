"""The f32 attention where the CTAs that share a slice's keys come in several waves, with the window's behind them."""
import pytest
import torch

from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,hist,n", [
    (88, 195, 120),            # 5 key tiles, three CTAs each: all at once
    (99, 195, 120),            # more of them than run at once as clusters
    (50, 700, 310),            # 16 key tiles x 150 CTAs: two waves of clusters
    (22, 1030, 1130),          # 34 x 198: three
    (150, 370, 290),           # 450 CTAs, a slice each
])
def test_f32_splits_match_64_bits(heads, hist, n):
    kv = binding.ScaleKV(1, 1, heads, 64, "f32", [1, 1, 1], [hist, n, 1], [[binding.KEEP_ALL, 40, binding.KEEP_ALL]], window_kind="last")
    g = torch.Generator(device="cuda").manual_seed(heads + n)
    maps = [tuple(torch.randn(1, heads, m, 64, generator=g, device="cuda") for _ in range(3)) for m in (hist, n)]
    lse = torch.empty(1, heads, n, device="cuda")
    O = torch.empty(1, heads, n, 64, device="cuda")
    torch.cuda.synchronize()
    kv.scalekv_append(0, 0, *maps[0][1:])
    kv.scalekv_step(0, 1, *maps[1], O, window_pos=list(range(n - 16, n)), lse=lse)
    kv.scalekv_sync()
    kv.close()
    K, V = (torch.cat([m[i] for m in maps], 2).double() for i in (1, 2))
    S = maps[1][0].double() @ K.transpose(2, 3) / 8
    assert (lse.double() - S.logsumexp(-1)).abs().max().item() <= 1e-5        # sums near 2^3 .. 2^4, rounded a few times: some 2^-20
    assert (O.double() - S.softmax(-1) @ V).abs().max().item() <= 1e-4        # as against the oracle
