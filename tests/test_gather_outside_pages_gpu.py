"""The pruning where the current map has not been copied into the pages: its survivors come from the caller's tensors, the others from the pages."""
import pytest
import torch

from oracle import scalekv_oracle as orc
from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f32", 64)])
@pytest.mark.parametrize("padding", [0, 16])               # columns between a row's end and the next row
@pytest.mark.parametrize("hist,entries,budget", [
    (24, 700, 112), (24, 700, 113),                        # 128 and 129 rows: one chunk of the gather, and one row more
    (24, 1200, 496), (24, 1200, 497),                      # 512 and 513: one round of look-ups, and one row more
    (500, 700, 112), (700, 1200, 497),                     # most rows from the pages, the rest from the tensors
    (24, 40, 0),                                           # the window alone
])
def test_rows_moved_at_the_edges_of_the_gather(hist, entries, budget, padding, dtype, d):
    """Slot 0 goes, so that every kept row moves: as many as are kept."""
    dt, heads, w = (torch.bfloat16 if dtype == "bf16" else torch.float32), 3, 16
    n = [hist, entries - hist, 1]
    g = torch.Generator().manual_seed(entries + budget + hist)
    maps = []
    for m in n[:2]:
        Q, K, V = torch.zeros(1, heads, m, d), 0.1 * torch.randn(1, heads, m, d, generator=g), torch.randn(1, heads, m, d, generator=g)
        Q[..., 0] = 1.0
        for h in range(heads):
            K[0, h, :, 0] = 0.25 * torch.randperm(m, generator=g).float() / 8
        maps.append([Q, K, V])
    maps[0][1][:, :, 0, 0] = -8.0                          # the lowest product of all
    def rows(x):
        at = torch.full((*x.shape[:3], d + padding), 7.0, device="cuda", dtype=dt)
        at[..., :d] = x.to("cuda", dt)
        return at[..., :d]
    dev = [[rows(x) for x in m] for m in maps]
    kv = binding.ScaleKV(1, 1, heads, d, dtype, [1, 1, 1], n, [[binding.KEEP_ALL, budget, binding.KEEP_ALL]], window_kind="last")
    window = list(range(n[1] - w, n[1]))
    O = torch.empty(1, heads, n[1], d, device="cuda", dtype=dt)
    torch.cuda.synchronize()
    kv.scalekv_append(0, 0, *dev[0][1:])
    kv.scalekv_attend(0, dev[0][0])
    before = kv.scalekv_launch_count()
    kv.scalekv_step(0, 1, *dev[1], O, window_pos=window)
    # attend, compress and, of long f32 slices, the sums of the window's rows: nothing has copied the map
    assert kv.scalekv_launch_count() - before == (3 if dtype == "f32" and entries > 512 else 2)
    kv.scalekv_sync()
    for h in range(heads):
        pos, K, V = kv.scalekv_export_slice(0, 0, h, with_kv=True)
        assert len(pos) == budget + w and pos[0] > 0       # all of them have moved
        c = orc.SliceCache(n, d)
        for _, *map_kv in maps:
            c.append(*(x[0, h].to(dt).double().numpy() for x in map_kv))
        want, _ = c.compress(maps[1][0][0, h].to(dt).double().numpy()[window], window, budget)
        assert (pos.numpy() == want).all()
        for got, i in ((K, 1), (V, 2)):
            assert torch.equal(got, torch.cat([m[i][0, h] for m in dev]).cpu()[pos.long()])
    kv.close()
