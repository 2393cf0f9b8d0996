"""scalekv_layer_stats_ex over its two kernels: few and many rows, splits that are no power of two, K' on either side of 16, more rows
than the scratch takes."""
import numpy as np
import pytest
import torch

from oracle import scalekv_oracle as orc
from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,topk,stride,sides", [
    (1, 16, 1, (1, 3, 9)),            # fewer rows than a warp's 16, a history shorter than K', ragged key tiles
    (3, 16, 1, (8, 16, 13)),          # tiles that are history, map and both; five and eight key ranges
    (2, 1, 3, (5, 31, 8)),
    (16, 15, 2, (2, 20, 33)),         # nine blocks of rows
    (5, 0, 4, (4, 11)),               # three key ranges
    (2, 17, 1, (3, 18, 7)),           # K' > 16: the other kernel
])
def test_statistics_match_the_oracle(heads, topk, stride, sides):
    d = 128
    n = orc.scale_token_counts(sides)
    g = torch.Generator().manual_seed(17)
    kv = binding.ScaleKV(1, 1, heads, d, "bf16", sides, sides, [[binding.KEEP_ALL] * len(sides)])
    caches = [orc.SliceCache(n, d) for _ in range(heads)]
    for k, nk in enumerate(n):
        Q, K, V = (torch.randn(1, heads, nk, d, generator=g).to(torch.bfloat16) for _ in range(3))
        K[:, :, 0] *= 4.0
        Qd, Kd, Vd = Q.cuda(), K.cuda(), V.cuda()
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, Kd, Vd)
        car, htk, cs, ts, ns = kv.scalekv_layer_stats_ex(0, Qd, topk, stride)
        want_c, want_t = [], []
        for h in range(heads):
            caches[h].append(K[0, h].double().numpy(), V[0, h].double().numpy())
            y = Q[0, h].double().numpy()[::stride] @ caches[h].K.T / np.sqrt(d)
            a = np.exp(y - y.max(1, keepdims=True))
            a /= a.sum(1, keepdims=True)
            hist = a.shape[1] - nk
            want_c.append(a[:, hist:].sum(1).mean())
            want_t.append(np.sort(a[:, :hist], axis=1)[:, ::-1][:, :topk].sum(1).mean())
        # logits are sums of 128 exact products in fp32: ~1e-6 of their size (up to ~40 here), which is what a weight is off by
        assert np.allclose(cs[0], want_c, rtol=1e-4, atol=1e-7) and np.allclose(ts[0], want_t, rtol=1e-4, atol=1e-7)
        assert np.allclose(ns[0], np.array(want_c) * (hist + nk) / nk, rtol=1e-4)
        assert abs(car - np.mean(want_c)) <= 1e-4 * abs(car) and abs(htk - np.mean(want_t)) <= 1e-4 * abs(htk) + 1e-7
        assert kv.scalekv_lengths(0) == [[sum(n[:k + 1])] * heads]
    kv.close()


def test_rows_of_scores_near_the_lowest_number():
    """Every score near the type's lowest value: they differ by less than it resolves, so all entries weigh the same."""
    sides, heads, d, topk = (4, 9), 3, 128, 16
    n = orc.scale_token_counts(sides)
    g = torch.Generator(device="cuda").manual_seed(19)
    kv = binding.ScaleKV(1, 1, heads, d, "bf16", sides, sides, [[binding.KEEP_ALL] * len(sides)])
    for k, nk in enumerate(n):
        Q, K, V = (torch.randn(1, heads, nk, d, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(3))
        Q[..., 0], K[..., 0] = 1.0, -3e38
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, K, V)
        _, _, cs, ts, _ = kv.scalekv_layer_stats_ex(0, Q, topk, 1)
        L = sum(n[: k + 1])
        assert np.allclose(cs, nk / L, rtol=1e-5) and np.allclose(ts, min(topk, L - nk) / L, rtol=1e-5, atol=1e-7)
    kv.close()


def test_nothing_is_expected_of_the_workspace_between_calls():
    """The workspace is borrowed: its owner may have used it for something else between two calls."""
    sides, heads, d = (4, 20), 2, 128
    g = torch.Generator(device="cuda").manual_seed(23)
    kv = binding.ScaleKV(1, 1, heads, d, "bf16", sides, sides, [[binding.KEEP_ALL] * len(sides)])
    inputs = [tuple(torch.randn(1, heads, a * a, d, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(3)) for a in sides]
    passes = []
    for fill in (0, 0x2b):
        kv.scalekv_reset()
        passes.append([])
        for k, (Q, K, V) in enumerate(inputs):
            kv.workspace.fill_(fill)
            torch.cuda.synchronize()
            kv.scalekv_append(0, k, K, V)
            passes[-1].append(kv.scalekv_layer_stats_ex(0, Q, 16, 1))
    kv.close()
    assert passes[0] == passes[1]


def test_more_records_than_the_scratch_holds():
    """33 slices x 4 096 rows: the tensor-core kernel's records do not fit, the other kernel takes the call although K' <= 16."""
    sides, batch, heads, d, topk = (2, 64), 3, 11, 128, 5
    g = torch.Generator(device="cuda").manual_seed(31)
    kv = binding.ScaleKV(1, batch, heads, d, "bf16", sides, sides, [[binding.KEEP_ALL] * len(sides)])
    keys = []
    for k, a in enumerate(sides):
        Q, K, V = (torch.randn(batch, heads, a * a, d, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(3))
        keys.append(K)
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, K, V)
        _, _, cs, ts, _ = kv.scalekv_layer_stats_ex(0, Q, topk, 1)
    for b in range(batch):
        for h in range(heads):
            A = (Q[b, h].double() @ torch.cat([K[b, h] for K in keys]).double().T / d ** 0.5).softmax(-1)
            hist = sides[0] ** 2
            # (the bound of the test above)
            assert abs(cs[b][h] - A[:, hist:].sum(1).mean().item()) <= 1e-4 * cs[b][h] + 1e-7
            assert abs(ts[b][h] - A[:, :hist].topk(min(topk, hist))[0].sum(1).mean().item()) <= 1e-4 * ts[b][h] + 1e-7
    kv.close()
