"""Host sets that cannot be sorted in parts: strings that reach into
characters that are still on their way.  They are left out of the parts' sorts
and the whole set is sorted afterwards."""
import numpy as np
import pytest

import gen
from gpu_util import assert_parity, from_strings

pytestmark = pytest.mark.gpu


def _set(layout):
    rng = np.random.default_rng(len(layout))
    if layout == "suffixes":  # to the end of the text, no cap
        s = gen.dna_suffix_set(300_000, 3)
        s.max_len = 0
        return s
    s = gen.url_set(200_000, 5)
    if layout == "shuffled":
        s.offsets = s.offsets[rng.permutation(s.n)]
    elif layout == "reversed":
        s.offsets = s.offsets[::-1].copy()
    elif layout == "last_first":  # only the last part is not packed
        s.offsets[-1] = s.offsets[0]
    elif layout == "first_last":  # ... or the first one
        s.offsets[0] = s.offsets[-1]
    elif layout == "one_string":  # a million characters, then short strings; an offset inside the long one
        s = from_strings([b"ab" * 500_000] + [b"%07d" % k for k in rng.integers(0, 10**7, 100_000)])
        s.offsets[5] = 1000
    return s


@pytest.mark.parametrize("parts", [2, 4, 16])
@pytest.mark.parametrize("layout", ["suffixes", "shuffled", "reversed", "last_first", "first_last", "one_string"])
def test_not_packed(layout, parts):
    import torch

    import paper_1808_00963_gb300 as ss
    s = _set(layout)
    chars = torch.from_numpy(s.chars.copy()).pin_memory()
    offsets = torch.from_numpy(s.offsets.view(np.int64).copy()).pin_memory()
    for _ in range(2):
        p, l = ss.sort_host(chars, offsets, s.max_len, host_parts=parts)
        assert_parity(s, p, l)


def test_packed_with_long_and_empty_strings():
    import paper_1808_00963_gb300 as ss
    rng = np.random.default_rng(1)
    strs = [b"x" * int(k) for k in rng.integers(0, 40, 30_000)]
    strs[12_345] = b"y" * 300_000
    s = from_strings(strs)
    for parts in (2, 8):
        p, l = ss.sort_host(s.chars, s.offsets.view(np.int64), 0, host_parts=parts)
        assert_parity(s, p, l)
