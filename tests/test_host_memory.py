"""Device memory that a call holds at once, against what the header states
(counted on a stand-in for the CUDA runtime)."""
import ctypes
import re

import numpy as np
import pytest

import fake_util
import paper_1808_00963_gb300 as ss


def _stated():
    text = " ".join(line.strip(" *") for line in open(ss.HEADER).read().splitlines())
    return int(re.search(r"At most about (\d+) bytes of device memory per text character", text).group(1))


@pytest.mark.parametrize("with_lcp", [True, False])
@pytest.mark.parametrize("n", [1000, 4096, 33_000, 100_000, 1_000_000])
def test_suffix_array(tmp_path, n, with_lcp):
    lib = fake_util.load(tmp_path)
    text, sa, lcp = np.ones(n + 1, np.uint8), np.zeros(n, np.uint32), np.zeros(n, np.uint32)
    for _ in range(2):  # (the first call also allocates what is kept)
        lib.fake_peak()
        assert lib.ss_suffix_array(text.ctypes.data, n, sa.ctypes.data, lcp.ctypes.data if with_lcp else None, 0,
                                   ctypes.c_void_p(0x99)) == 0
    peak, stated = lib.fake_peak(), n * _stated() + 100_000
    assert peak <= 1.03 * stated and (n < 100_000 or peak >= 0.9 * stated), peak / n
