"""The block sorts on sets of 33..4096 strings.  A plain sort of so few strings
is ranked by counting; an option that sizes the distribution steps keeps it on
the block sorts, with the whole mixed set as one subset."""
import numpy as np
import pytest

from gpu_util import assert_parity, from_strings, gpu_sort
from test_gpu_blocksort import _runs
from test_gpu_windows import _placed

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cutoff", [1024, 4096])
@pytest.mark.parametrize("tail", [0, 70])
@pytest.mark.parametrize("n", [33, 34, 64, 65, 127, 255, 256, 257, 513, 1023, 1024])
def test_runs_of_equal_caches(n, tail, cutoff):
    rng = np.random.default_rng(n + tail)
    sizes = [2, 31, 32, 33, 63, 64, 65, 66, 128, 255, 256, 257, 300]
    rng.shuffle(sizes)
    s = from_strings(_runs(rng, n, sizes, tail))
    assert_parity(s, *gpu_sort(s, small_cutoff=cutoff))


@pytest.mark.parametrize("n", [1025, 2048, 3000, 4095, 4096])
@pytest.mark.parametrize("tail", [0, 70])
def test_runs_in_large_subsets(n, tail):
    rng = np.random.default_rng(n + tail)
    sizes = [int(x) for x in rng.choice([31, 32, 33, 64, 65, 255, 256, 257, 600], 30)]
    s = from_strings(_runs(rng, n, sizes, tail))
    assert_parity(s, *gpu_sort(s, small_cutoff=4096))


@pytest.mark.parametrize("cap", [0, 1, 7, 8, 9, 15, 16, 17, 24, 70])
@pytest.mark.parametrize("n, cutoff", [(200, 1024), (600, 1024), (600, 64), (3000, 4096)])
def test_windows_around_block_boundaries(n, cutoff, cap):
    rng = np.random.default_rng(cap + n)
    pre = bytes(rng.integers(97, 99, 100).astype(np.uint8))
    starts, strings = [], []
    for k in range(n):
        length = int(rng.integers(0, 96))
        share = int(rng.integers(0, length + 1))
        starts.append((k + 1) * 4096 - int(rng.integers(0, 96)))
        strings.append(pre[:share] + bytes(rng.integers(97, 99, length - share).astype(np.uint8)))
    s = _placed(starts, strings, (n + 2) * 4096)
    s.max_len = cap
    assert_parity(s, *gpu_sort(s, small_cutoff=cutoff))


@pytest.mark.parametrize("cutoff", [64, 1024])
def test_every_alignment_and_length(cutoff):
    pre = b"abcdefghijklmnopqrstuvwxyzabcdefghijklmnopqrstuvwxyz"
    starts, strings, at = [], [], 0
    for align in range(16):
        for length in range(40):
            at = (at + 15) // 16 * 16 + align
            starts.append(at)
            strings.append(pre[:length])
            at += length + 1
    s = _placed(starts, strings, at + 64)
    assert_parity(s, *gpu_sort(s, small_cutoff=cutoff))


@pytest.mark.parametrize("n, cutoff", [(33, 1024), (100, 1024), (3000, 1024), (3000, 4096)])
def test_long_common_prefix(n, cutoff):
    rng = np.random.default_rng(n)
    pre = bytes(rng.integers(97, 123, size=600).astype(np.uint8))
    strs = [pre + bytes(rng.integers(97, 99, size=int(rng.integers(0, 20))).astype(np.uint8)) for _ in range(n)]
    strs[::7] = [pre] * len(strs[::7])
    s = from_strings(strs)
    assert_parity(s, *gpu_sort(s, small_cutoff=cutoff))
    assert_parity(s, *gpu_sort(s, small_cutoff=cutoff, with_lcp=False))
