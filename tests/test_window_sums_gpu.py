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


@pytest.mark.parametrize("heads,hist,n,w,launches", [
    (3, 200, 312, 32, 1), (3, 200, 312, 33, 2),      # two rounds of rows; a third costs more than a launch of its own where few slices wait for it
    (8, 200, 312, 64, 2), (9, 200, 312, 64, 1),      # eight slices are few
    (1, 100, 156, 64, 1), (1, 100, 157, 64, 2),      # and rows of up to 256 entries short
    (3, 31, 33, 33, 1),
])
@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f32", 64)])
def test_wide_windows_of_few_slices_are_summed_by_a_launch(dtype, d, heads, hist, n, w, launches):
    """One answer whoever sums the rows, and the launch where it is the quicker way."""
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(hist + n + w)
    data = [tuple(torch.randn(1, heads, m, d, generator=g, device="cuda").to(dt) for _ in range(3)) for m in (hist, n)]
    window = list(range(n - w, n))
    out = []
    for separate in (False, True):
        kv = binding.ScaleKV(1, 1, heads, d, dtype, [1, 1, 1], [hist, n, 1], [[binding.KEEP_ALL, (hist + n) // 3, binding.KEEP_ALL]], max_window=64)
        torch.cuda.synchronize()
        kv.scalekv_append(0, 0, *data[0][1:])
        kv.scalekv_append(0, 1, *data[1][1:])
        kv.scalekv_attend(0, data[1][0])
        before = kv.scalekv_launch_count()
        kv.scalekv_compress_ex(0, data[1][0], window, qw_is_full_map=True, separate_kernels=separate)
        if not separate:
            assert kv.scalekv_launch_count() - before == launches + 1        # (the logits' first: this window has not been recorded)
        kv.scalekv_sync()
        out.append([(kv.scalekv_export_scores(0, h), kv.scalekv_export_slice(0, 0, h)) for h in range(heads)])
        kv.close()
    for one, other in zip(*out):
        assert all(torch.equal(torch.as_tensor(a), torch.as_tensor(b)) for a, b in zip(one, other))
