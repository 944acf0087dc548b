"""Block sorts of subsets of 33..small_cutoff strings: sizes at the edges of
the two block sizes, runs of equal caches around the limits at which they are
handed on (32 and 256 strings) or ranked by ballots (64), few and many subsets."""
import numpy as np
import pytest

from gpu_util import assert_parity, from_strings, gpu_sort

pytestmark = pytest.mark.gpu


def _runs(rng, n, sizes, tail):
    """n strings: runs of the given sizes sharing an 8-character key each (and `tail` more characters), the rest
    random, shuffled."""
    out = []
    for k, size in enumerate(sizes):
        key = bytes(rng.integers(97, 123, 8 + tail).astype(np.uint8))
        for _ in range(size):
            out.append(key + bytes(rng.integers(97, 100, int(rng.integers(0, 4))).astype(np.uint8)))
    while len(out) < n:
        out.append(bytes(rng.integers(97, 123, int(rng.integers(0, 14))).astype(np.uint8)))
    out = out[:n]
    return [out[i] for i in rng.permutation(n)]


@pytest.mark.parametrize("tail", [0, 70])
@pytest.mark.parametrize("n", [33, 64, 65, 255, 256, 257, 513, 1023, 1024])
def test_runs_of_equal_caches(n, tail):
    rng = np.random.default_rng(n + tail)
    sizes = [s for s in (2, 31, 32, 33, 63, 64, 65, 66, 128, 255, 256, 257, 300)]
    rng.shuffle(sizes)
    s = from_strings(_runs(rng, n, sizes, tail))
    assert_parity(s, *gpu_sort(s))


@pytest.mark.parametrize("kind", ["equal", "one_other_first", "one_other_last", "two_keys", "ended", "ladder"])
@pytest.mark.parametrize("n", [40, 256, 300, 1024, 4000])
def test_degenerate_subsets(n, kind):
    rng = np.random.default_rng(n)
    a, b = b"abcdefgh" * 10, b"abcdefgi"
    strs = {"equal": [a] * n, "one_other_first": [b] + [a] * (n - 1), "one_other_last": [a] * (n - 1) + [b],
            "two_keys": [(a, b)[int(x)] for x in rng.integers(0, 2, n)],
            "ended": [b"abc"] * (n // 2) + [b"abcd"] * (n - n // 2),
            "ladder": [a[:int(x)] for x in rng.integers(0, 80, n)]}[kind]
    s = from_strings(strs)
    assert_parity(s, *gpu_sort(s, small_cutoff=4096))


@pytest.mark.parametrize("groups", [3, 40, 3000])
def test_few_and_many_subsets(groups):
    # groups of 33..600 strings behind distinct prefixes: as many block-sort subsets, few enough for
    # the large blocks to take them all, and more than that
    rng = np.random.default_rng(groups)
    strs = []
    for g in range(groups):
        pre = b"%06d" % g + bytes(rng.integers(97, 123, 2).astype(np.uint8))
        for _ in range(int(rng.integers(33, 60 if groups > 100 else 600))):
            strs.append(pre + bytes(rng.integers(97, 99, int(rng.integers(0, 30))).astype(np.uint8)))
    strs = [strs[i] for i in rng.permutation(len(strs))]
    s = from_strings(strs)
    assert_parity(s, *gpu_sort(s))
