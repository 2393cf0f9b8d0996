"""layer_stats on a map that is still in the caller's tensors: same numbers, rows in the pages, tensors free when it returns."""
import pytest
import torch

from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,height,width,stride", [
    (16, 1, 1, 1), (3, 1, 63, 1), (16, 1, 128, 3), (5, 3, 43, 1),        # copied beside: blocks of 128 rows, one row more
    (16, 32, 32, 16), (16, 25, 41, 16),                                  # two copying CTAs per slice of 512 rows; a row more than they take
    (2, 40, 40, 7),                                                      # several blocks of rows
    (32, 20, 20, 16), (300, 2, 5, 1),                                    # launches that are full without them
])
def test_a_map_outside_the_pages(heads, height, width, stride):
    n, first = height * width, 37
    g = torch.Generator(device="cuda").manual_seed(3)
    maps = [[torch.randn(1, heads, m, 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3)] for m in (first, n)]
    answers = []
    for outside in (True, False):
        kv = binding.ScaleKV(1, 1, heads, 128, "bf16", [1, height], [first, width], [[binding.KEEP_ALL] * 2])
        for k, (Q, K, V) in enumerate(maps):
            K, V = K.clone(), V.clone()
            torch.cuda.synchronize()
            kv.scalekv_append(0, k, K, V)
            if not outside:
                kv.scalekv_export_slice(0, 0, 0)             # (copies the map)
            got = kv.scalekv_layer_stats_ex(0, Q, 16, stride)
            K.zero_(), V.zero_()                             # on another stream, at once
            torch.cuda.synchronize()
        answers.append(torch.tensor([list(got[:2]) + sum((x[0] for x in got[2:]), [])], dtype=torch.float64))
        for h in {0, heads // 2, heads - 1}:
            pos, Kh, Vh = kv.scalekv_export_slice(0, 0, h, with_kv=True)
            assert pos.tolist() == list(range(first + n))
            assert torch.equal(Kh, torch.cat([m[1][0, h] for m in maps]).cpu())
            assert torch.equal(Vh, torch.cat([m[2][0, h] for m in maps]).cpu())
        kv.close()
    # (the keys may be split over another number of CTAs: sums of fp32 weights in another order)
    assert torch.allclose(answers[0], answers[1], rtol=1e-5, atol=0)


def test_every_word_of_an_answer_has_one_writer():
    """Behind a refused selection the device's slices outgrow their pages, and every call answers that it has no numbers - at once, with
    many CTAs per block of rows still to come: none of them may write into the next call's words."""
    sides, heads = (2, 5, 9, 24), 3
    kv = binding.ScaleKV(1, 1, heads, 128, "bf16", sides, sides, [[10] * 4], page_tokens=16)
    g = torch.Generator(device="cuda").manual_seed(43)
    for k, a in enumerate(sides):
        Q, K, V = (torch.randn(1, heads, a * a, 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, K, V)
        if k < 3:                                                            # the heads part at scale 1; their common selection is refused at scale 2
            kv.scalekv_attend(0, Q)
            kv.scalekv_compress_ex(0, Q, binding.scalekv_window_centroids(a, a, 16), qw_is_full_map=True, head_shared=k == 2)
    for _ in range(200):
        car, htk, cars, htks, ncas = kv.scalekv_layer_stats_ex(0, Q, 16, 1)
        assert all(x != x for x in [car, htk] + cars[0] + htks[0] + ncas[0])
    with pytest.raises(binding.ScaleKVError):
        kv.scalekv_sync()
    kv.close()
