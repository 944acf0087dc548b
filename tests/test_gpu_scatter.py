"""The multi-block distribution at its edges: tiles of 8 to 32 rounds that are
full, ragged or all of one bucket (the largest counts), and subsets whose common prefix ends
anywhere in a key, against the oracle."""
import numpy as np
import pytest

import gen
import oracle
from gpu_util import gpu_sort

pytestmark = pytest.mark.gpu


def from_rows(rows, cap=0):
    """One string per row of a byte matrix (0 ends it early)."""
    n, w = rows.shape
    chars = np.zeros((n, w + 1), np.uint8)
    chars[:, :w] = rows
    return gen.StringSet(chars.reshape(-1), (np.arange(n) * (w + 1)).astype(np.uint64), cap)


def check(s, **opts):
    p, l = gpu_sort(s, big_threshold=4096, small_cutoff=64, **opts)
    wp, wl = oracle.sort(s.chars, s.offsets, s.max_len)
    np.testing.assert_array_equal(p, wp)
    np.testing.assert_array_equal(l, wl)


@pytest.mark.parametrize("rounds", [0, 8, 16, 32])
@pytest.mark.parametrize("extra", [-1, 0, 1])
@pytest.mark.parametrize("kinds", [1, 3, 5000])
def test_tile_edges(rounds, extra, kinds):
    rng = np.random.default_rng(kinds)
    n = 2 * 256 * 32 + extra
    words = rng.integers(97, 123, (kinds, 30)).astype(np.uint8)
    rows = words[rng.integers(0, kinds, n)]
    rows[rng.random(n) < 0.2, 17] = 122  # some differ behind the first 16 characters
    check(from_rows(rows), tile_rounds=rounds)


@pytest.mark.parametrize("cap", [0, 7, 9, 12, 13, 16, 20])
@pytest.mark.parametrize("alphabet", [b"ab", b"ACGT", None])
def test_prefix_ends_inside_the_key(alphabet, cap):
    # 40 subsets of 500 strings each: the strings of subset k agree in 6 + k % 12
    # characters (DNA keys: up to three times as many)
    rng = np.random.default_rng(cap)
    letters = np.frombuffer(alphabet, np.uint8) if alphabet else np.arange(1, 256, dtype=np.uint8)
    rows = letters[rng.integers(0, len(letters), (20000, 70))]
    step = 3 if alphabet == b"ACGT" else 1
    for k in range(40):
        share = (6 + k % 12) * step
        rows[500 * k:500 * (k + 1), :share] = rows[500 * k, :share]
    rows[rng.random(20000) < 0.1, 11] = 0  # ends inside and before the shared part
    rows = rows[rng.permutation(20000)]
    check(from_rows(rows, cap))
    if alphabet == b"ACGT":
        check(from_rows(rows, cap), dna=True)
