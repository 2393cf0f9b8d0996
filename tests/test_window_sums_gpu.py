"""The log-sum-exps of a window that attend has not left: taken by the compress of a short slice, or by a launch of their own."""
import pytest
import torch

from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f32", 64)])
@pytest.mark.parametrize("hist,n,w", [
    (1, 2, 1), (20, 44, 5),              # a row of less than a warp, of two rounds
    (200, 312, 16), (200, 312, 40),      # 512 entries, the longest that the compress sums; more rows than warps
    (200, 313, 16),                      # one more: a launch of its own both times
])
def test_sums_are_the_same_to_the_bit(dtype, d, hist, n, w):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(hist + n + w)
    data = [tuple(torch.randn(1, 3, m, d, generator=g, device="cuda").to(dt) for _ in range(3)) for m in (hist, n)]
    window = list(range(0, n, max(1, n // w)))[:w]
    out = []
    for separate in (False, True):
        kv = binding.ScaleKV(1, 1, 3, d, dtype, [1, 1, 1], [hist, n, 1], [[binding.KEEP_ALL, (hist + n) // 3, binding.KEEP_ALL]], max_window=64)
        torch.cuda.synchronize()
        for k, (Q, K, V) in enumerate(data):
            kv.scalekv_append(0, k, K, V)
            kv.scalekv_attend(0, Q)
            if k == 1:
                kv.scalekv_compress_ex(0, Q, window, qw_is_full_map=True, separate_kernels=separate)
        kv.scalekv_sync()
        out.append([(kv.scalekv_export_scores(0, h), kv.scalekv_export_slice(0, 0, h)) for h in range(3)])
        kv.close()
    for one, other in zip(*out):
        assert all(torch.equal(torch.as_tensor(a), torch.as_tensor(b)) for a, b in zip(one, other))
