"""How many CTAs share a slice's keys in the f32 attention: the host's rule, compiled by itself."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_19602_b200", "csrc")
SMS = 148


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    at = tmp_path_factory.mktemp("key_split")
    (at / "rule.cpp").write_text('#include "key_split.h"\nextern "C" int rule(int ctas, int tiles, int n_sm) { return scalekv::f32::key_split(ctas, tiles, n_sm); }\n')
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(at / "rule.cpp"), "-o", str(at / "rule.so")], check=True)
    rule = ctypes.CDLL(str(at / "rule.so")).rule
    return lambda ctas, tiles: rule(ctas, tiles, SMS)


def test_slices_of_two_tiles_are_shared_where_every_cta_finds_an_sm(split):
    assert [split(ctas, 2) for ctas in (1, 4, 73, 74, 75, 148, 149, 296, 297, 5000)] == [2, 2, 2, 2, 1, 1, 1, 1, 1, 1]


@pytest.mark.parametrize("tiles,first,last", [
    # key tiles, CTAs of the unsplit launch: sizes that are not shared, since nobody has measured that they should be
    (3, 50, 74), (5, 75, 98), (6, 99, 148), (9, 99, 148), (8, 297, 444), (11, 297, 444), (12, 149, 197), (16, 149, 197),
    (14, 149, 197), (14, 593, 740), (28, 198, 222), (31, 198, 222), (34, 198, 222), (37, 198, 222), (50, 223, 236), (54, 223, 236), (58, 223, 236), (62, 223, 236),
])
def test_longer_slices_are_not_shared_on_the_model_s_word_alone(split, tiles, first, last):
    assert {split(ctas, tiles) for ctas in range(first, last + 1)} == {1}


def test_a_split_charges_one_and_a_half_tiles_above_two(split):
    def charged(ctas, tiles):
        def cost(c):
            n, per = ctas * c, -(-tiles // c)
            return (1 if n <= SMS else 1.35) * (-(-n // (2 * SMS)) * (per + 3)) + (1.5 if c > 1 else 0)
        costs = [cost(c) for c in range(1, min(8, tiles) + 1)]
        near = [c + 1 for c in range(len(costs)) if costs[c] <= min(costs) + 1e-3]       # (32 bits may break a tie either way)
        return near
    for tiles in list(range(3, 40)) + [50, 62, 80, 165]:
        for ctas in list(range(1, 760, 7)) + [1000, 1199, 4096]:
            assert split(ctas, tiles) in charged(ctas, tiles), (tiles, ctas)
