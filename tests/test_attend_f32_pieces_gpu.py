"""The f32 attention by products of bf16 pieces: edges of its tiles, its error, numbers it cannot split, maps outside the pages."""
import pytest
import torch

from oracle import scalekv_oracle as orc
from paper_2505_19602_b200 import binding
from parity_util import ParityRun

pytestmark = pytest.mark.gpu


def full_cache(heads, sides, make, sides_w=None, lse=False):
    """Attends map after map behind a full cache; the last map's queries, all keys and values, and what came out."""
    kv = binding.ScaleKV(1, 1, heads, 64, "f32", sides, sides_w or sides, [[binding.KEEP_ALL] * len(sides)])
    keys, values = [], []
    for k, n in enumerate(kv.n):
        Q, K, V = make(k, n)
        keys.append(K), values.append(V)
        out = torch.empty(1, heads, n, device="cuda") if lse else None
        torch.cuda.synchronize()
        kv.scalekv_append(0, k, K, V)
        O = kv.scalekv_attend(0, Q, lse=out)
        kv.scalekv_sync()
    kv.close()
    return Q, torch.cat(keys, 2), torch.cat(values, 2), O, out


def normal(seed, heads):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return lambda n: (torch.randn(1, heads, n, 64, generator=g, device="cuda") for _ in range(3))


@pytest.mark.parametrize("page", [16, 128])
@pytest.mark.parametrize("heights,widths,budget", [
    ((1, 1, 1), (1, 63, 64), 20),        # a tile of keys, one less, one more
    ((1, 1, 1), (3, 127, 129), 50),      # a block of queries and one row
    ((1, 5, 16), (2, 13, 24), 33),
])
def test_one_call_steps_match_oracle(heights, widths, budget, page):
    """Maps that the attention reads in the caller's tensors: a step that evicts nothing copies them into the pages, from one that does the
    compress takes the rows that stay."""
    n = orc.scale_token_counts(heights, widths)
    g = torch.Generator().manual_seed(31)
    data = [tuple(torch.randn(2, 3, nk, 64, generator=g) for _ in range(3)) for nk in n]
    budgets = [[budget] * len(n)]
    kv = binding.ScaleKV(1, 2, 3, 64, "f32", heights, widths, budgets, page_tokens=page)
    run = ParityRun(kv, "f32", heights, budgets, lambda l, k: data[k], lambda k: orc.window_centroids(heights[k], widths[k], 16),
                    [(0, b, h) for b in range(2) for h in range(3)], compress_last=True, sides_w=widths)
    run.run_pipelined()
    kv.close()


# by queries' gain: a score of size s is off by about 2^-24 s per rounding of its sum and of its exponent, at random from key to key, and
# a weight by as much; a few such for scores of 0.25, 1 and 3, whose larger ones carry the weight.  Measured: 1.4 to 1.7e-7, 2.2 to
# 2.4e-7 and 3.9 to 4.0e-7; plain fp32 sums over these keys give 4.6 to 11.9e-7, 5.5 to 12.3e-7 and 10.7 to 15.2e-7.
BOUND = {0.25: 3.5e-7, 1.0: 5e-7, 3.0: 8e-7}


@pytest.mark.parametrize("heads", [1, 40])             # keys shared by a cluster, and not
@pytest.mark.parametrize("gain", [0.25, 1.0, 3.0])
def test_error_is_that_of_fp32_arithmetic(heads, gain):
    """Against 64 bits.  A score s is off by some 2^-24 of the larger ones' size per rounding, and so is a weight; sums over thousands of
    keys may not add to that."""
    draw = normal(11, heads)

    def make(k, n):
        Q, K, V = draw(n)
        return Q * gain, K, V

    Q, K, V, O, lse = full_cache(heads, (24, 60), make, lse=True)
    s = Q.double() @ K.double().transpose(2, 3) / 8
    want = s.softmax(-1) @ V.double()
    assert ((O.double() - want).norm() / want.norm()).item() <= BOUND[gain]
    assert (lse.double() - s.logsumexp(-1)).pow(2).mean().sqrt().item() <= 1e-6


@pytest.mark.parametrize("heads", [1, 40])
@pytest.mark.parametrize("q,k,v", [(0, 0, -118), (0, 0, 99), (0, 0, 110), (-118, 118, 0), (118, -118, 0), (-118, 95, 0), (95, -105, 0), (100, -100, 0)])
def test_numbers_at_the_ends_of_the_range(heads, q, k, v):
    """Gains of 2^q, 2^k and 2^v: pieces that would be subnormal, operands that cannot be lifted.  The bound of scores of size 1."""
    draw = normal(12, heads)

    def make(_, n):
        Q, K, V = draw(n)
        return Q * 2.0 ** q, K * 2.0 ** k, V * 2.0 ** v

    Q, K, V, O, lse = full_cache(heads, (8, 18), make, lse=True)
    s = Q.double() @ K.double().transpose(2, 3) / 8
    want = s.softmax(-1) @ V.double()
    assert ((O.double() - want).norm() / want.norm()).item() <= BOUND[1.0]
    assert (lse.double() - s.logsumexp(-1)).pow(2).mean().sqrt().item() <= 1e-6


@pytest.mark.parametrize("heads", [1, 40])
@pytest.mark.parametrize("first", [0, 40, 64])
def test_keys_masked_with_minus_infinity(heads, first):
    """Keys whose products are -inf have no weight, whatever the signs of the queries' pieces."""
    draw = normal(5, heads)

    def make(k, n):
        Q, K, V = draw(n)
        Q[..., 0] = Q[..., 0].abs() + 0.01
        if k == 1:
            K[:, :, first: first + 32, 0] = -float("inf")
        return Q, K, V

    Q, K, V, O, _ = full_cache(heads, (8, 18), make)
    s = (Q.double() @ K.double().transpose(2, 3) / 8).masked_fill(torch.isinf(K[..., 0])[:, :, None], -float("inf"))
    assert (O.double() - s.softmax(-1) @ V.double()).abs().max().item() <= 1e-5


@pytest.mark.parametrize("heads", [1, 40])
def test_infinite_values_reach_their_column_only(heads):
    draw = normal(6, heads)

    def make(k, n):
        Q, K, V = draw(n)
        if k == 1:
            V[:, :, 70, 5] = float("inf")
        return Q, K, V

    Q, K, V, O, _ = full_cache(heads, (8, 18), make)
    want = (Q.double() @ K.double().transpose(2, 3) / 8).softmax(-1) @ V.double()
    assert torch.isinf(O[..., 5]).all() and (O[..., 5] > 0).all()
    rest = [c for c in range(64) if c != 5]
    assert (O.double() - want)[..., rest].abs().max().item() <= 1e-5


@pytest.mark.parametrize("heads", [1, 40])
@pytest.mark.parametrize("masked", [1, 3, 64, 1500])
def test_masked_keys_among_thousands(heads, masked):
    """-inf in one of their columns, here and there: the others' weights are those of fp32 arithmetic."""
    draw = normal(14, heads)
    g = torch.Generator(device="cuda").manual_seed(15)

    def make(k, n):
        Q, K, V = draw(n)
        Q[..., 7] = Q[..., 7].abs() + 0.01
        K[:, :, torch.randperm(n, generator=g, device="cuda")[:masked if k == 0 else 1], 7] = -float("inf")
        return Q, K, V

    Q, K, V, O, lse = full_cache(heads, (60, 12), make, lse=True)
    s = (Q.double() @ K.double().transpose(2, 3) / 8).masked_fill(torch.isinf(K[..., 7])[:, :, None], -float("inf"))
    want = s.softmax(-1) @ V.double()
    assert ((O.double() - want).norm() / want.norm()).item() <= BOUND[1.0]
    assert (lse.double() - s.logsumexp(-1)).pow(2).mean().sqrt().item() <= 1e-6


@pytest.mark.parametrize("heads", [1, 40])
def test_infinite_columns_of_either_sign(heads):
    """The sign of a score with infinite columns is its query's, or it has none: where both signs meet, and where the query is zero."""
    draw = normal(20, heads)

    def make(k, n):
        Q, K, V = draw(n)
        Q[..., 3], Q[..., 40], Q[..., 63] = Q[..., 3].abs() + 0.01, -Q[..., 40].abs() - 0.01, Q[..., 63].abs() + 0.01
        for first, second in ((5, 6), (n - 1, n - 2)):
            K[:, :, first, 3], K[:, :, first, 40] = -float("inf"), float("inf")
            K[:, :, second, 3], K[:, :, second, 63] = -float("inf"), -float("inf")
        K[:, 0, 9, 40] = float("inf")
        Q[:, :, 2, 3] = 0.0
        Q[:, :, 4, 40] = 1e-30
        Q[:, :, 6, 3], Q[:, :, 6, 40], Q[:, :, 6, 63] = -1.0, 1.0, -1.0
        return Q, K, V

    Q, K, V, O, lse = full_cache(heads, (60, 12), make, lse=True)
    s = Q.double() @ K.double().transpose(2, 3) / 8
    want = s.softmax(-1) @ V.double()
    assert torch.isnan(want).any(-1).sum().item() == 3 * heads and (torch.isnan(O) == torch.isnan(want)).all()
    there = torch.isfinite(want)
    assert ((O.double() - want)[there].norm() / want[there].norm()).item() <= BOUND[1.0]
    assert (lse.double() - s.logsumexp(-1))[there[..., 0]].pow(2).mean().sqrt().item() <= 1e-6


@pytest.mark.parametrize("heads", [1, 40])
def test_rows_that_are_done_again_are_as_exact_as_plain_sums(heads):
    """An infinite value spoils all rows, an infinite query its own, a key that is no number all of its head's."""
    draw = normal(16, heads)

    def make(k, n):
        Q, K, V = draw(n)
        if k == 0:
            V[:, 0, 70, 5] = float("inf")
            if heads > 1:
                K[:, 1, 3000, 9] = float("nan")
        else:
            Q[:, -1, 3, 2] = float("inf")
        return Q, K, V

    Q, K, V, O, lse = full_cache(heads, (60, 12), make, lse=True)
    s = Q.double() @ K.double().transpose(2, 3) / 8
    want = s.softmax(-1) @ V.double()
    assert (torch.isnan(O) == torch.isnan(want)).all() and (torch.isinf(O) == torch.isinf(want)).all()
    there = torch.isfinite(want)
    # sums of 3 744 terms one behind the other: half a unit of 2^-24 each of a growing sum, at random, sqrt(3744 / 3) / 2 of them
    assert ((O.double() - want)[there].norm() / want[there].norm()).item() <= 2e-6
    finite = torch.isfinite(s).all(-1)
    assert (lse.double() - s.logsumexp(-1))[finite].abs().max().item() <= 2e-6


def test_a_map_whose_keys_and_values_are_laid_out_differently():
    """A one-call step takes it, evicting or not."""
    sides, heads = (4, 12, 15), 3
    g = torch.Generator(device="cuda").manual_seed(8)
    outs = []
    maps = [[torch.randn(1, heads, a * a, 64, generator=g, device="cuda") for _ in range(3)] for a in sides]
    for spread in (False, True):
        kv = binding.ScaleKV(1, 1, heads, 64, "f32", sides, sides, [[40] * 3])
        for k, (Q, K, V) in enumerate(maps):
            if spread:
                wide = torch.zeros(1, K.shape[2], heads, 64, device="cuda")
                wide.copy_(V.transpose(1, 2))
                V = wide.transpose(1, 2)
            O = torch.zeros_like(Q)
            window = kv.window_array(binding.scalekv_window_centroids(sides[k], sides[k], 16)) if k < 2 else None
            torch.cuda.synchronize()
            kv.scalekv_step(0, k, Q, K, V, O, window_pos=window)
            kv.scalekv_sync()
        outs.append(O.clone())
        kv.close()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("policy", ["recent", "score"])
def test_maps_laid_out_differently_are_pruned_like_others(dtype, policy):
    """In the steps, and by a compress of its own behind the last one, which leaves its map in the caller's tensors."""
    sides, heads, d = (4, 12, 15), 3, 64 if dtype == "f32" else 128
    g = torch.Generator(device="cuda").manual_seed(8)
    maps = [[torch.randn(1, heads, a * a, d, generator=g, device="cuda") for _ in range(3)] for a in sides]
    left = []
    for spread in (False, True):
        kv = binding.ScaleKV(1, 1, heads, d, dtype, sides, sides, [[40] * 3])
        for k, tensors in enumerate(maps):
            Q, K, V = (x.to(kv.torch_dtype) for x in tensors)
            if spread:
                V = V.transpose(1, 2).contiguous().transpose(1, 2)
            O = torch.zeros_like(Q)
            window = binding.scalekv_window_centroids(sides[k], sides[k], 16)
            torch.cuda.synchronize()
            kv.scalekv_step_ex(0, k, Q, K, V, O, compress=k < 2, window_pos=kv.window_array(window), policy=policy)
            if k == 2:
                kv.scalekv_compress_ex(0, Q, window, qw_is_full_map=True, policy=policy)
            kv.scalekv_sync()
            left.append(O.clone())
        left.append([kv.scalekv_export_slice(0, 0, h, with_kv=True) for h in range(heads)])
        kv.close()
    for x, y in zip(left[:3], left[4:7]):
        assert torch.equal(x, y)
    for x, y in zip(left[3], left[7]):
        assert all(torch.equal(a, b) for a, b in zip(x, y))


@pytest.mark.parametrize("refused", ["attend", "compress"])
def test_a_step_that_is_refused_half_way_keeps_its_map(refused):
    """In the pages, as an append by itself would have: the caller goes on without the tensors."""
    heads, n = 3, (20, 150)
    draw = normal(18, heads)
    kv = binding.ScaleKV(1, 1, heads, 64, "f32", [1, 1], n, [[30] * 2], page_tokens=16)
    Q, K, V = draw(n[0])
    torch.cuda.synchronize()
    kv.scalekv_append(0, 0, K, V)
    kv.scalekv_attend(0, Q)
    kv.scalekv_sync()
    keys, values = [K], [V]
    Q, K, V = draw(n[1])
    keys.append(K.clone()), values.append(V.clone())
    O = torch.empty_like(Q)
    torch.cuda.synchronize()
    with pytest.raises(binding.ScaleKVError):
        if refused == "attend":                            # rows that start between 16-byte boundaries
            kv.scalekv_step(0, 1, torch.empty(Q.numel() + 1, device="cuda")[1:].view_as(Q), K, V, O, window_pos=[3, 70])
        else:                                              # more sinks than the pages were planned for
            kv.scalekv_step_ex(0, 1, Q, K, V, O, policy="recent", n_sink=140)
    kv.scalekv_sync()
    K.zero_(), V.zero_()
    torch.cuda.synchronize()
    O = kv.scalekv_attend(0, Q)
    kv.scalekv_sync()
    want = (Q.double() @ torch.cat(keys, 2).double().transpose(2, 3) / 8).softmax(-1) @ torch.cat(values, 2).double()
    assert (O.double() - want).abs().max().item() <= 1e-5
    kv.close()
