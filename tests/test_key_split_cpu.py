"""How many CTAs share a slice's keys in the f32 attention: the host's rule, compiled by itself."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_19602_b200", "csrc")
SMS, FIT = 148, (0, 0, 148, 93, 71, 56, 45, 37, 33)         # what a B200 has room for: clusters of 2, 3, .. CTAs, two CTAs to an SM


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    at = tmp_path_factory.mktemp("key_split")
    (at / "rule.cpp").write_text('#include "key_split.h"\nextern "C" int rule(int ctas, int tiles, int n_sm, const int *fit) '
                                 '{ return scalekv::f32::key_split(ctas, tiles, n_sm, fit); }\n')
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(at / "rule.cpp"), "-o", str(at / "rule.so")], check=True)
    rule = ctypes.CDLL(str(at / "rule.so")).rule
    return lambda tiles, ctas, fit=FIT: rule(ctas, tiles, SMS, (ctypes.c_int * 9)(*fit))


def test_slices_of_two_tiles_are_shared_where_every_cta_finds_an_sm(split):
    assert [split(2, ctas) for ctas in (1, 4, 73, 74, 75, 148, 149, 296, 297, 5000)] == [2, 2, 2, 2, 1, 1, 1, 1, 1, 1]


@pytest.mark.parametrize("tiles,ctas,more", [
    (5, 91, 3), (14, 189, 3), (13, 94, 3), (28, 216, 4), (24, 72, 4), (29, 57, 5), (50, 234, 5), (35, 46, 6), (28, 41, 7), (32, 36, 8),
])
def test_no_wave_of_clusters_for_the_last_few(split, tiles, ctas, more):
    """`more` CTAs for one fit 296 places, but not as clusters."""
    assert ctas * more <= 2 * SMS * -(-ctas * more // (2 * SMS))
    chosen = split(tiles, ctas)
    assert chosen != more or -(-ctas // FIT[more]) == -(-ctas * more // (2 * SMS))


@pytest.mark.parametrize("tiles,ctas,want", [
    (3, 74, 2), (5, 75, 3), (5, 90, 3), (6, 148, 2), (9, 100, 2), (12, 149, 3), (16, 178, 3), (34, 198, 4), (28, 213, 4),
    (8, 297, 1), (8, 444, 1), (11, 360, 1), (14, 600, 1), (14, 740, 1), (27, 972, 1),            # more than a wave, one CTA each
])
def test_sizes_with_both_sides_measured(split, tiles, ctas, want):
    assert split(tiles, ctas) == want


def test_bounds(split):
    for tiles in list(range(1, 24)) + [80, 165, 1000]:
        for ctas in (1, 7, 33, 37, 38, 148, 149, 296, 297, 4096):
            assert 1 <= split(tiles, ctas) <= min(8, tiles)
            assert split(tiles, ctas, (0,) * 9) == 1        # a device that cannot run clusters
