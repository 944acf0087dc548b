"""The doubling rounds of the suffix array at their edges: groups just below,
at and above the size up to which a round compares the members of a group with
one another (256), alone and mixed, and texts around the tiles of the naming
passes, against the oracle's sort of all suffixes."""
import numpy as np
import pytest

import oracle
from test_gpu_sa import gpu_sa

pytestmark = pytest.mark.gpu


def grouped_text(sizes, seed, tail=6):
    """Words of 12 characters, word g sizes[g] times, each followed by random
    characters: at depth 4 word g makes groups of sizes[g] suffixes."""
    rng = np.random.default_rng(seed)
    units = []
    for k in sizes:
        word = rng.integers(1, 256, 12)
        units += [np.concatenate([word, rng.integers(1, 256, tail)]) for _ in range(k)]
    return bytes(np.concatenate([units[i] for i in rng.permutation(len(units))]).astype(np.uint8))


def check(text, depth):
    sa, lcp = gpu_sa(text, initial_depth=depth)
    want_sa, want_lcp = oracle.suffix_array(text)
    np.testing.assert_array_equal(sa, want_sa)
    np.testing.assert_array_equal(lcp, want_lcp)
    return want_lcp


@pytest.mark.parametrize("sizes", [[2] * 500, [64] * 20, [255] * 6, [256] * 6, [257] * 6, [2, 255, 256, 257, 3, 500], [64, 2000]],
                         ids=lambda s: "-".join(map(str, sorted(set(s)))))
@pytest.mark.parametrize("tail", [0, 6])
def test_group_sizes(sizes, tail):
    lcp = check(grouped_text(sizes, 5 + tail, tail), 4)
    run = np.diff(np.nonzero(np.concatenate([lcp < 4, [True]]))[0])  # sizes of the groups at depth 4
    assert run.max() >= max(sizes)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 255, 256, 257, 4095, 4096, 4097, 8193, 304 * 4096 + 1])
def test_tile_edges(n):
    rng = np.random.default_rng(n)
    text = bytes(rng.integers(ord("a"), ord("e"), n).astype(np.uint8))
    for depth in (2, 7):  # large groups first, small ones from the start
        check(text, depth)
