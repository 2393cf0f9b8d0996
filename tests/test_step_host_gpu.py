"""scalekv_step_host over growing maps: the staging halves of consecutive scales must not meet."""
import pytest
import torch

from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shrink", [False, True])
def test_growing_maps_do_not_overwrite_the_step_before(shrink):
    """Two layers, maps that quadruple: the input copies of layer 0's next scale run while layer 1's is being attended.  Outputs
    equal those of the device calls bit for bit.  shrink: the caller passes only as much of its staging area as the scale needs, so
    the halves lie elsewhere from step to step."""
    sides, B, H, d = (4, 8, 16, 32, 64), 2, 16, 128
    n = [a * a for a in sides]
    g = torch.Generator().manual_seed(5)
    data = [tuple(torch.randn(B, H, nk, d, generator=g).to(torch.bfloat16).pin_memory() for _ in range(3)) for nk in n]
    kv = binding.ScaleKV(2, B, H, d, "bf16", sides, sides, [[64] * len(sides)] * 2)
    windows = [binding.scalekv_window_centroids(a, a, 16) for a in sides]
    staging = torch.empty(8 * B * H * max(n) * d, dtype=torch.bfloat16, device="cuda")
    device = [tuple(t.cuda() for t in qkv) for qkv in data]
    want = [[torch.empty_like(Q) for Q, _, _ in device] for _ in range(2)]
    out = [[torch.empty_like(Q).pin_memory() for Q, _, _ in data] for _ in range(2)]
    torch.cuda.synchronize()
    window = lambda k: windows[k] if k + 1 < len(sides) else None
    for k in range(len(sides)):
        for l in range(2):
            kv.scalekv_step(l, k, *device[k], want[l][k], window_pos=window(k))
    for _ in range(3):
        kv.scalekv_reset()
        for k, (Q, K, V) in enumerate(data):
            area = staging[: 8 * Q.numel()] if shrink else staging
            for l in range(2):
                kv.scalekv_step_host(l, k, Q, K, V, out[l][k], area, window_pos=window(k))
        kv.scalekv_sync()
        for k in range(len(sides)):
            for l in range(2):
                assert torch.equal(out[l][k], want[l][k].cpu()), (l, k)
    kv.close()
