"""The tables of the table-driven logarithm, made again from their recipe (the comment at the head of
rt_lntab.cuh) and compared with the committed ones entry by entry, with the ranges that the evaluation
(ln_tab in rt_rng.cuh) takes for granted."""
import os
import re

import pytest

mp = pytest.importorskip("mpmath")

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_00405_gb300", "csrc",
                      "rt_lntab.cuh")
TOL = 48  # an entry's own rounding is below 1 / TOL of its last place


def _round64(v):
    """The nearest multiple of 2^-64 as an integer, and how far v lies from it in those units."""
    x = mp.ldexp(v, 64)
    n = int(mp.floor(x + mp.mpf(1) / 2))
    return n, abs(x - n)


def make_tables():
    with mp.workprec(300):
        ln2 = mp.log(2)
        first, zmax = [], mp.mpf(0)
        for i in range(64, 128):  # f in [i / 128, (i + 1) / 128)
            s = 1 if i <= 90 else 0
            r = (128 << 15) // (i + 1)  # the largest with f r 2^-15 <= 1 in the whole bucket
            while True:
                L, e = _round64(mp.log(mp.ldexp(r, -15)) - s * ln2)
                if e * TOL <= 1:
                    break
                r -= 1
            zmax = max(zmax, 1 - mp.mpf(i * r) / (128 << 15))
            below, above = 1 - s, s  # m = 2 f > 1 below sqrt(1/2), m = f < 1 above it
            if i == 90:  # holds sqrt(1/2)
                below = above = 1
            first.append((L % (1 << 64), r, s | below << 1 | above << 2))
        second, size = [], int(mp.floor(zmax * 4096)) + 1
        for j in range(size):  # z in [j / 4096, (j + 1) / 4096)
            t = (j << 24) // (4096 - j)  # the largest with (1 - z)(1 + t 2^-24) <= 1
            while True:
                L, e = _round64(mp.log(1 + mp.ldexp(t, -24)))
                if e * TOL <= 1:
                    break
                t -= 1
            second.append((L, t << 8))
    return first, second


def committed():
    text = open(HEADER).read()
    a, b = text.split("kLn1[64] = {")[1].split("kLn2[kLn2Size] = {")
    first = [(int(x, 16), int(y), int(z)) for x, y, z in re.findall(r"\{(0x[0-9A-F]+)ull, (\d+)u, (\d+)u\}", a)]
    second = [(int(x, 16), int(y, 16)) for x, y in re.findall(r"\{(0x[0-9A-F]+)ull, (0x[0-9A-F]+)u, 0u\}", b)]
    return first, second, int(re.search(r"kLn2Size = (\d+);", text).group(1))


def test_tables_follow_their_recipe():
    first, second, size = committed()
    assert (len(first), len(second)) == (64, size)
    assert make_tables() == (first, second)


def test_ranges_the_evaluation_relies_on():
    first, second, size = committed()
    z_end = [(1 << 53) - (i << 46) * r // (1 << 15) for i, (_, r, _) in zip(range(64, 128), first)]  # 2^-53
    assert all(((i + 1) << 46) * r <= 1 << 68 for i, (_, r, _) in zip(range(64, 128), first))  # z >= 0
    assert max(z_end) < 2.0 ** (53 - 5.9) and max(z_end) >> 41 < size  # the second table's index
    for j, (_, t) in enumerate(second):
        assert t >> 32 == 0 and t % 256 == 0
        one = 1 << 44  # (1 - z)(1 + t) with z in 2^-12 and t in 2^-32
        assert ((4096 - j) * ((1 << 32) + t)) <= one  # z' >= 0
        assert one - (4096 - j - 1) * ((1 << 32) + t) < 2.0 ** (44 - 11.9)  # z' at the far end
