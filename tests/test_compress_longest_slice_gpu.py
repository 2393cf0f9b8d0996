"""The longest slice whose keys and keep list fit one CTA's shared memory beside the selection's own state."""
import pytest
import torch

from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entries,launches", [
    (27712, 1),            # 433 pages of 64 entries: 4 (2 x 27 712 + 433) of 232 448 bytes less 8 864
    (27776, 3),            # a page more
])
def test_longest_slice_of_the_one_launch_compress(entries, launches):
    g = torch.Generator(device="cuda").manual_seed(5)
    n = [24, entries - 24, 1]
    maps = [tuple(torch.randn(1, 2, m, 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3)) for m in n[:2]]
    kept = []
    for separate in (False, True):
        kv = binding.ScaleKV(1, 1, 2, 128, "bf16", [1, 1, 1], n, [[binding.KEEP_ALL, 300, binding.KEEP_ALL]], page_tokens=64, window_kind="last")
        torch.cuda.synchronize()
        kv.scalekv_append(0, 0, *maps[0][1:])
        kv.scalekv_append(0, 1, *maps[1][1:])
        kv.scalekv_attend(0, maps[1][0])
        before = kv.scalekv_launch_count()
        kv.scalekv_compress_ex(0, maps[1][0], list(range(n[1] - 16, n[1])), qw_is_full_map=True, separate_kernels=separate)
        assert kv.scalekv_launch_count() - before == (3 if separate else launches)
        kv.scalekv_sync()
        kept.append([kv.scalekv_export_slice(0, 0, h) for h in range(2)])
        kv.close()
    assert all((a == b).all() and len(a) == 316 for a, b in zip(*kept))
