"""CPU test of the warp-tile step's table of words per species: the packed
bytes and shifts of a tet's lookup (emulated here, 1 to 32 species) give every
word that decides a molecule its species, and every other word of its last
Philox block an index that the block's table of species scales holds."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1610_02258_gb300", "csrc")
MAX_WORDS = 127  # beyond, the lookup walks the trial counts


def _constant(text, name):
    value = re.search(rf"constexpr int {name} = ([^;]+);", text).group(1)
    for other in re.findall(r"k\w+", value):
        value = value.replace(other, str(_constant(text, other)))
    return eval(value)  # an integer expression


def _scale_entries():
    with open(os.path.join(CSRC, "steps_device.h")) as f:
        header = f.read()
    with open(os.path.join(CSRC, "steps_warp.cuh")) as f:
        size = re.search(r"__shared__ uint32_t s_scale\[(\w+)\];", f.read()).group(1)
    return _constant(header, size)


def _species_of(ends, v):
    """species_of on the packed prefix bytes of `ends` (words up to and including each species)."""
    rows = (len(ends) + 3) // 4
    pre = np.full(4 * rows, 0x80, np.uint64)
    pre[: len(ends)] = ends
    words = [int(sum(int(b) << (8 * k) for k, b in enumerate(pre[4 * j: 4 * j + 4]))) for j in range(rows)]
    v4 = v * 0x01010101 + 0x80808080
    u = 0
    for j, w in enumerate(words):
        u |= (((v4 - w) & 0xFFFFFFFF) >> j) & (0x80808080 >> j)
    return bin(u).count("1")


@pytest.mark.parametrize("S", range(1, 33))
def test_every_word_finds_its_species_and_a_scale(S):
    entries = _scale_entries()
    rng = np.random.default_rng(S)
    for _ in range(40):
        counts = rng.integers(0, 16, S) * (rng.random(S) < rng.random())
        while counts.sum() > MAX_WORDS:
            counts[rng.integers(0, S)] = 0
        ends = np.cumsum(counts)
        W = int(ends[-1])
        owner = np.repeat(np.arange(S), counts)
        for v in range((W + 3) // 4 * 4):
            s = _species_of(ends, v)
            if v < W:
                assert s == owner[v]
            assert 0 <= s < entries, f"word {v} of {W} looks up scale {s} of {entries}"
