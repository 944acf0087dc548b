"""Shared-memory limits of the kernels: every device has its own, and threads
whose first sorts run at the same time do not undo each other's (checked on a
stand-in for the CUDA runtime that refuses launches above a kernel's limit)."""
import ctypes
import itertools

import pytest

import fake_util
from test_host_streams import Set


@pytest.fixture
def lib(tmp_path):
    return fake_util.load(tmp_path)


@pytest.mark.parametrize("device", [0, 1])
@pytest.mark.parametrize("opts", [{}, {"splitters_log2": 10}, {"small_cutoff": 4096}, {"tile_rounds": 32}])
def test_every_device(lib, device, opts):
    assert Set(20_000).sort(lib) == 0
    lib.fake_set_device(device)
    assert Set(20_000).sort(lib, **opts) == 0


@pytest.mark.parametrize("dna", [0, 1])
def test_first_sorts_at_the_same_time(lib, dna):
    def sort(cutoff):
        s = Set(20_000)
        if not dna:
            return s.sort(lib, stream=cutoff, small_cutoff=cutoff)
        o = fake_util.ss.make_options(small_cutoff=cutoff)
        chars, offsets, perm, lcp = s.ptrs
        return lib.ss_sort_dna(chars, s.n, offsets, s.n, perm, lcp, ctypes.byref(o),
                               ctypes.c_void_p(cutoff))

    assert sort(300) == 0  # everything but the block sorts' limit
    lib.fake_slow_attributes(20_000)
    assert fake_util.in_threads(lambda: sort(1024), lambda: sort(4096)) == [0, 0]
    assert sort(4096) == 0


def test_options_one_after_the_other(lib):
    for logv, cutoff, rounds in itertools.product((7, 10), (4096, 64), (32, 8)):
        assert Set(20_000).sort(lib, splitters_log2=logv, small_cutoff=cutoff, tile_rounds=rounds) == 0
