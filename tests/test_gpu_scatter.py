"""The multi-block distribution at its edges: tiles of 8 to 32 rounds that are
full, ragged or all of one bucket (the largest counts), against the oracle."""
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
