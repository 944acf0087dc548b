"""The time of a block sort does not hang on the order of its strings: sets in
which every k-th string has one key, in that order and shuffled."""
import numpy as np
import pytest

import gen
import oracle
from gpu_util import to_device

pytestmark = pytest.mark.gpu

LENGTH = 24


def _rows(rows):
    """Strings of equal length from a matrix of characters."""
    n = rows.shape[0]
    chars = np.concatenate([rows, np.zeros((n, 1), np.uint8)], axis=1)
    return gen.StringSet(chars.reshape(-1).copy(), np.arange(n, dtype=np.uint64) * (rows.shape[1] + 1))


def _batch(sets, cutoff):
    import torch

    import paper_1808_00963_gb300 as ss
    dev = []
    for s in sets:
        chars, offsets = to_device(s)
        dev.append((chars, offsets, 0, *(torch.empty(s.n, dtype=torch.int32, device="cuda") for _ in range(2))))
    return ss.Batch(dev, small_cutoff=cutoff)


def _us(batch):
    """Shortest time of a run among 15."""
    import torch
    best = float("inf")
    for _ in range(15):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        batch.run()
        b.record()
        torch.cuda.synchronize()
        best = min(best, 1000 * a.elapsed_time(b))
    batch.status()
    return best


@pytest.mark.parametrize("period", [4, 16])
@pytest.mark.parametrize("n, cutoff", [(256, 1024), (1024, 1024), (2048, 2048), (4096, 4096)])
def test_periodic_order(n, cutoff, period):
    # a set whose sample is all one key compares every string with all others: 4 to 12 times as long
    rng = np.random.default_rng(n + period)
    ordered, shuffled = [], []
    for _ in range(600):
        rows = rng.integers(97, 123, (n, LENGTH)).astype(np.uint8)
        rows[::period] = rows[0]
        ordered.append(_rows(rows))
        shuffled.append(_rows(rows[rng.permutation(n)]))
    runs = [_batch(x, cutoff) for x in (ordered, shuffled)]
    in_order, in_none = (_us(b) for b in runs)
    for sets, batch in zip((ordered, shuffled), runs):
        for k in (0, 1, 599):
            _, _, _, p, l = batch.keep[k]
            want_p, want_l = oracle.sort(sets[k].chars, sets[k].offsets, 0)
            assert np.array_equal(p.cpu().numpy().view(np.uint32), want_p)
            assert np.array_equal(l.cpu().numpy().view(np.uint32), want_l)
        batch.close()
    assert in_order < 1.5 * in_none, (in_order, in_none)


def test_large_subsets():
    # as many strings in subsets of 1024 and of 4096: few enough for every subset to have a block, which then takes
    # the larger one four times as many steps, most of them short ones; with the same number of splitters for both
    # a string of the larger one is compared with four times as many others, and it takes 2.7 times as long
    rng = np.random.default_rng(4)
    sets = [_rows(rng.integers(97, 123, (4096, LENGTH)).astype(np.uint8)) for _ in range(60)]
    quarters = [gen.StringSet(s.chars, s.offsets[k:k + 1024].copy()) for s in sets for k in range(0, 4096, 1024)]
    whole, parts = _us(_batch(sets, 4096)), _us(_batch(quarters, 4096))
    assert whole < 2 * parts, (whole, parts)


@pytest.mark.parametrize("kind", ["letters", "bits"])
@pytest.mark.parametrize("n", [1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096])
def test_splitter_counts(n, kind):
    from gpu_util import assert_parity, gpu_sort
    lo, hi, length = (97, 123, LENGTH) if kind == "letters" else (97, 99, 10)  # bits: four equal strings each
    s = _rows(np.random.default_rng(n).integers(lo, hi, (n, length)).astype(np.uint8))
    assert_parity(s, *gpu_sort(s, small_cutoff=4096))
    assert_parity(s, *gpu_sort(s, small_cutoff=4096, with_lcp=False))
