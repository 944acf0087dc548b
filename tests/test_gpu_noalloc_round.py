"""ss_sort_noalloc above the multi-block threshold: its root takes one
multi-block step inside the fixed scratch, everything after it the work queue;
equal to ss_sort_ex at the edges of its range and on inputs whose children stay
large (shared prefixes, equal strings)."""
import numpy as np
import pytest

import gen
from gpu_util import from_strings, to_device

pytestmark = pytest.mark.gpu


def _set(kind, n):
    rng = np.random.default_rng(n)
    if kind == "url":
        return gen.url_set(n, n)
    if kind == "bytes":
        return gen.random_set(n, n, 0, 40, 1, 255)
    if kind == "binary":
        return gen.random_set(n, n, 0, 24, ord("0"), ord("1"))
    if kind == "equal":
        return from_strings([b"abcdefghijklmnopqrstuvwxyz"] * n)
    pre = bytes(rng.integers(97, 123, 100).astype(np.uint8))
    return from_strings([pre + bytes(x) for x in rng.integers(97, 99, (n, 6)).astype(np.uint8)])


@pytest.mark.parametrize("n", [8191, 8192, 8193, 20011, 65535, 65536])
@pytest.mark.parametrize("kind", ["url", "bytes", "binary", "prefix", "equal"])
def test_same_as_sort(kind, n):
    import torch

    import paper_1808_00963_gb300 as ss
    s = _set(kind, n)
    chars, offsets = to_device(s)
    want_p, want_l = ss.sort(chars, offsets)
    for _ in range(2):  # the second call finds the first one's leftovers in the scratch
        p = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        l = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        ss.sort_noalloc(chars, offsets, out=(p, l))
        assert torch.equal(p, want_p) and torch.equal(l, want_l)
