"""bf16 attention where tiles end early: chunks of 32 keys that hold none, behind an end inside a chunk or at its edge."""
import pytest
import torch

from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slices", [1, 16, 160])                        # clusters, shared singles, more items than SMs
@pytest.mark.parametrize("hist", [1, 32, 33, 97, 128])
@pytest.mark.parametrize("n", [1, 100, 161, 289])
def test_ragged_tiles(slices, hist, n):
    """A pass before leaves values far from zero in the pages behind the history's end: a weight that should not be there would show.  (What lies
    behind the map's end is filled with zeros on its way into shared memory.)"""
    heads = slices if slices < 16 else 16
    g = torch.Generator(device="cuda").manual_seed(hist * 1000 + n)
    kv = binding.ScaleKV(1, slices // heads, heads, 128, "bf16", [1, 1], [hist, n], [[binding.KEEP_ALL] * 2])
    for first in (True, False):
        keys, values = [], []
        kv.scalekv_reset()
        for k, m in enumerate((hist, n)):
            Q, K, V = (torch.randn(slices // heads, heads, m, 128, generator=g, device="cuda") for _ in range(3))
            if k == 1:
                K[:, :, -1] *= 3                                          # the last key of the last tile counts
                if first:
                    V += 1000
            Q, K, V = (x.to(torch.bfloat16) for x in (Q, K, V))
            keys.append(K), values.append(V)
            torch.cuda.synchronize()
            kv.scalekv_append(0, k, K, V)
            lse = torch.empty(slices // heads, heads, m, device="cuda")
            O = kv.scalekv_attend(0, Q, lse=lse)
            kv.scalekv_sync()
    kv.close()
    s = Q.float() @ torch.cat(keys, 2).float().transpose(2, 3) / 128 ** 0.5
    want = s.softmax(-1) @ torch.cat(values, 2).float()
    # P and O are rounded to bf16, 2^-9 each relative to values of up to max |O|
    assert (O.float() - want).abs().max().item() <= max(2e-2, 2.0 ** -7 * want.abs().max().item())
    assert (lse - s.logsumexp(-1)).abs().max().item() <= 1e-3
