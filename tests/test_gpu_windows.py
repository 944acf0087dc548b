"""Character reads at the edges of their 16-byte words and 4 KiB blocks: every
alignment of a window's first byte, windows that end just before, at and past
a block boundary, terminators and caps at every place inside a window."""
import numpy as np
import pytest

import gen
import oracle

pytestmark = pytest.mark.gpu


def _placed(starts, strings, size):
    """A buffer with string k at starts[k] (random letters elsewhere)."""
    chars = np.random.default_rng(9).integers(97, 123, size).astype(np.uint8)
    for at, s in zip(starts, strings):
        chars[at:at + len(s)] = np.frombuffer(s, np.uint8)
        chars[at + len(s)] = 0
    return gen.StringSet(chars, np.array(starts, np.uint64), 0)


def _check(s, **opts):
    from gpu_util import gpu_sort
    p, l = gpu_sort(s, **opts)
    wp, wl = oracle.sort(s.chars, s.offsets, s.max_len)
    assert np.array_equal(p, wp) and np.array_equal(l, wl)


@pytest.mark.parametrize("cap", [0, 1, 7, 8, 9, 15, 16, 17, 24, 70])
@pytest.mark.parametrize("path", ["small", "queue", "big"])
def test_windows_around_block_boundaries(path, cap):
    # strings of 0..95 characters over two letters starting 0..95 bytes before
    # a 4 KiB boundary (relative to the 512-byte aligned device buffer), 12 000
    # in all; long common prefixes make every path read deep windows
    rng = np.random.default_rng(cap + 1)
    n = {"small": 600, "queue": 6000, "big": 12000}[path]
    pre = bytes(rng.integers(97, 99, 100).astype(np.uint8))
    starts, strings = [], []
    for k in range(n):
        before = int(rng.integers(0, 96))
        length = int(rng.integers(0, 96))
        share = int(rng.integers(0, length + 1))
        starts.append((k + 1) * 4096 - before)
        strings.append(pre[:share] + bytes(rng.integers(97, 99, length - share).astype(np.uint8)))
    s = _placed(starts, strings, (n + 2) * 4096)
    s.max_len = cap
    _check(s, **({"big_threshold": 4096, "small_cutoff": 64} if path == "big" else {}))


def test_every_alignment_and_length():
    # one string per (alignment, length) pair, all sharing one prefix, packed
    # back to back with a pad so that each alignment of 0..15 occurs
    pre = b"abcdefghijklmnopqrstuvwxyzabcdefghijklmnopqrstuvwxyz"
    starts, strings, at = [], [], 0
    for align in range(16):
        for length in range(40):
            at = (at + 15) // 16 * 16 + align
            starts.append(at)
            strings.append(pre[:length])
            at += length + 1
    _check(_placed(starts, strings, at + 64))


@pytest.mark.parametrize("runs", [2, 5])
def test_merge_windows(runs):
    import torch

    import paper_1808_00963_gb300 as ss
    rng = np.random.default_rng(runs)
    n = 4000
    starts = [(k + 1) * 4096 - int(rng.integers(0, 48)) for k in range(n)]
    pre = bytes(rng.integers(97, 99, 48).astype(np.uint8))
    strings = [pre[:int(rng.integers(0, 48))] + bytes(rng.integers(97, 99, int(rng.integers(0, 20))).astype(np.uint8))
               for _ in range(n)]
    s = _placed(starts, strings, (n + 2) * 4096)
    chars = torch.from_numpy(s.chars).cuda()
    offs = torch.from_numpy(s.offsets.view(np.int64)).cuda()
    own = torch.from_numpy(rng.integers(0, runs, n)).cuda()
    parts = []
    for k in range(runs):
        sub = torch.nonzero(own == k).flatten()
        p, l = ss.sort(chars, offs[sub].contiguous())
        parts.append((sub.to(torch.int32)[p.long()], l))
    p, l = ss.merge(chars, offs, parts)
    wp, wl = oracle.sort(s.chars, s.offsets)
    assert np.array_equal(p.cpu().numpy().view(np.uint32), wp)
    assert np.array_equal(l.cpu().numpy().view(np.uint32), wl)
