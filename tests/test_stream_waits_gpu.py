"""Compresses that run beside later layers' attends: the same values, bit for bit, as with everything on one stream."""
import time

import pytest
import torch

from oracle import scalekv_oracle as orc
from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu

SIDES = (2, 6, 12, 20, 24)


def _pass(budgets, heads, data, side_stream, dtype="bf16"):
    n = orc.scale_token_counts(SIDES)
    kv = binding.ScaleKV(len(budgets), 1, heads, data[0][0][0].shape[-1], dtype, SIDES, SIDES, budgets, side_stream=side_stream)
    out = [[torch.empty_like(data[l][k][0]) for l in range(len(budgets))] for k in range(len(n))]
    torch.cuda.synchronize()
    for _ in range(2):                     # the second pass finds every layer's and every page set's last compress to wait for
        kv.scalekv_reset()
        for k in range(len(n)):
            window = orc.window_centroids(SIDES[k], SIDES[k], 16)
            for l in range(len(budgets)):
                kv.scalekv_step(l, k, *data[l][k], out[k][l], window_pos=window)
    kv.scalekv_join()
    kv.scalekv_sync()
    kv.close()
    return out


# budgets of the layers in turn (-1: nothing is evicted): fewer layers than page sets, one more, all sets twice over, layers of which
# some compress and some do not, so that the last compress of a layer and of its set's owner are near and far
@pytest.mark.parametrize("layers,budget_of", [(1, (40,)), (3, (40,)), (5, (40, 200)), (9, (40,)), (9, (40, -1, -1)), (8, (-1, 40, 40, -1))])
def test_overlapped_compresses_change_nothing(layers, budget_of):
    heads = 16
    budgets = [[budget_of[l % len(budget_of)]] * len(SIDES) for l in range(layers)]
    gen = torch.Generator(device="cuda").manual_seed(17)
    data = [[tuple(torch.randn(1, heads, nk, 128, generator=gen, device="cuda", dtype=torch.bfloat16) for _ in range(3))
             for nk in orc.scale_token_counts(SIDES)] for _ in range(layers)]
    beside, alone = (_pass(budgets, heads, data, s) for s in (True, False))
    for k in range(len(SIDES)):
        for l in range(layers):
            assert torch.equal(beside[k][l], alone[k][l]), (k, l)


# f32 steps record into the sets' buffers by CTAs of the attend's launch, and their compresses take rows from the caller's tensors
@pytest.mark.parametrize("layers,budget_of", [(5, (40, 200)), (9, (40,)), (8, (-1, 40, 40, -1))])
def test_overlapped_f32_compresses_change_nothing(layers, budget_of):
    heads = 16
    budgets = [[budget_of[l % len(budget_of)]] * len(SIDES) for l in range(layers)]
    gen = torch.Generator(device="cuda").manual_seed(19)
    data = [[tuple(torch.randn(1, heads, nk, 64, generator=gen, device="cuda") for _ in range(3)) for nk in orc.scale_token_counts(SIDES)]
            for _ in range(layers)]
    beside, alone = (_pass(budgets, heads, data, s, "f32") for s in (True, False))
    for k in range(len(SIDES)):
        for l in range(layers):
            assert torch.equal(beside[k][l], alone[k][l]), (k, l)


# Layers 0 and 4 share their logit buffer.  Layer 0 scores from K, into that buffer, because layer 4 has appended in between:
# "kept": while the attend of layer 4, whose compress has evicted nothing, may still record there
# "late": and layer 4 only attends then
def _shared_buffer_pass(order, data, windows, sides, side_stream):
    budgets = [[5] * len(sides)] * 4 + [[-1 if order == "kept" else 5] * len(sides)]
    kv = binding.ScaleKV(5, 4, 16, 128, "bf16", sides, sides, budgets, page_tokens=4096, side_stream=side_stream)
    out = []
    torch.cuda.synchronize()
    for k in range(len(sides)):
        O = [torch.empty_like(Q) for Q, _, _ in data[k]]
        append = lambda l: kv.scalekv_append(l, k, *data[k][l > 0][1:])
        attend = lambda l: kv.scalekv_attend(l, data[k][l > 0][0], O[l > 0])
        compress = lambda l: kv.scalekv_compress(l, data[k][l > 0][0], windows[k], qw_is_full_map=True)
        append(0), attend(0), append(4)
        if order == "kept":
            attend(4), compress(4), compress(0)
        else:
            compress(0), attend(4), compress(4)
        out.append(O)
    kv.scalekv_join()
    kv.scalekv_sync()
    kept = [kv.scalekv_export_slice(l, b, h) for l in (0, 4) for b in range(4) for h in range(16)]
    kv.close()
    return [o for O in out for o in O] + kept


@pytest.mark.parametrize("order", ["kept", "late"])
def test_layers_that_share_a_logit_buffer_wait_for_each_other(order):
    sides = (8, 32, 40)
    gen = torch.Generator(device="cuda").manual_seed(29)
    data = [[tuple(torch.randn(4, 16, a * a, 128, generator=gen, device="cuda", dtype=torch.bfloat16) for _ in range(3))
             for _ in range(2)] for a in sides]
    windows = [orc.window_centroids(a, a, 16) for a in sides]
    beside, alone = (_shared_buffer_pass(order, data, windows, sides, s) for s in (True, False))
    for x, y in zip(beside, alone, strict=True):
        assert torch.equal(x, y)


@pytest.mark.parametrize("calls", ["attend", "step"])        # a map that the attend has copied, one that the statistics copy
def test_a_compress_waits_for_the_statistics_before_it(calls):
    """layer_stats returns when its sums have arrived, before stream_main's end is known: the compress waits for what stream_main
    has been given since the attend, as work behind the statistics shows."""
    sides, heads = (4, 12), 16
    n = orc.scale_token_counts(sides)
    gen = torch.Generator(device="cuda").manual_seed(37)
    data = [tuple(torch.randn(1, heads, nk, 128, generator=gen, device="cuda", dtype=torch.bfloat16) for _ in range(3)) for nk in n]
    kept = []
    for side_stream in (True, False):
        kv = binding.ScaleKV(1, 1, heads, 128, "bf16", sides, sides, [[30] * len(n)], side_stream=side_stream)
        torch.cuda.synchronize()
        for k, (Q, K, V) in enumerate(data):
            if calls == "attend" or k + 1 < len(n):
                kv.scalekv_append(0, k, K, V)
                kv.scalekv_attend(0, Q)
            else:
                kv.scalekv_step(0, k, Q, K, V, torch.empty_like(Q))
            kv.scalekv_layer_stats_ex(0, Q)
            with torch.cuda.stream(kv.stream_main):
                torch.cuda._sleep(200_000_000)                # about a tenth of a second
            kv.scalekv_compress(0, Q, orc.window_centroids(sides[k], sides[k], 16), qw_is_full_map=True)
            done = torch.cuda.Event()
            done.record(kv.stream_side)
            time.sleep(0.02)
            evicts = n[k] > 30 + 16
            assert not (evicts and done.query())
            kv.scalekv_sync()
        kept.append([torch.cat([x.float().reshape(len(x), -1) for x in kv.scalekv_export_slice(0, 0, h, with_kv=True)], 1) for h in range(heads)])
        kv.close()
    for x, y in zip(*kept, strict=True):
        assert torch.equal(x, y)


def test_an_f32_attend_records_no_window():
    """It does not know what compress follows, if any: it waits for no other layer's compress, and writes O over Q where it is asked to."""
    sides, heads = (8, 32), 16
    gen = torch.Generator(device="cuda").manual_seed(41)
    data = [tuple(torch.randn(1, heads, a * a, 64, generator=gen, device="cuda") for _ in range(3)) for a in sides]
    window = orc.window_centroids(32, 32, 16)
    kept = []
    for in_place in (True, False):
        kv = binding.ScaleKV(5, 1, heads, 64, "f32", sides, sides, [[5, 50]] * 5, page_tokens=4096)
        torch.cuda.synchronize()
        for l in (0, 4):
            kv.scalekv_step(l, 0, *data[0], torch.empty_like(data[0][0]), window_pos=orc.window_centroids(8, 8, 16))
        kv.scalekv_sync()
        Q, K, V = data[1]
        kv.scalekv_append(0, 1, K, V)
        beside = kv.scalekv_attend(0, Q)                      # (held: what it is written to must not be given to `out`)
        kv.scalekv_append(4, 1, K, V)
        out, done = Q.clone(), torch.cuda.Event()
        torch.cuda.synchronize()
        with torch.cuda.stream(kv.stream_side):
            torch.cuda._sleep(200_000_000)                    # about a tenth of a second
        kv.scalekv_compress(0, Q, window, qw_is_full_map=True)
        O = kv.scalekv_attend(4, out if in_place else Q, out)
        done.record(kv.stream_main)
        time.sleep(0.02)
        assert done.query()
        kv.scalekv_compress(4, Q, window, qw_is_full_map=True)
        kv.scalekv_sync()
        kept.append([O, beside] + [kv.scalekv_export_slice(l, 0, h) for l in (0, 4) for h in range(heads)])
        kv.close()
    for x, y in zip(*kept, strict=True):
        assert torch.equal(x, y)
