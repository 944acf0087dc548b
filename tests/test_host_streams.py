"""What the host code does when several threads sort on one stream, checked on
a stand-in for the CUDA runtime that logs the launches."""
import ctypes
import time

import numpy as np
import pytest

import fake_util
import paper_1808_00963_gb300 as ss

STREAM = 0x77
BIG = 20_000  # strings: above the multi-block threshold


@pytest.fixture
def lib(tmp_path):
    return fake_util.load(tmp_path)


class Set:
    def __init__(self, n):
        self.n = n
        self.bufs = [np.zeros(n + 16, np.uint64) for _ in range(4)]
        self.ptrs = [ctypes.c_void_p(b.ctypes.data) for b in self.bufs]

    def sort(self, lib, stream=STREAM, **opts):
        chars, offsets, perm, lcp = self.ptrs
        return lib.ss_sort_ex(chars, offsets, self.n, perm, lcp, ctypes.byref(ss.make_options(**opts)),
                              ctypes.c_void_p(stream))

    def desc(self):
        chars, offsets, perm, lcp = (p.value for p in self.ptrs)
        return ss.SetDesc(chars, offsets, self.n, 0, perm, lcp)


def multi_block_parts(lib):
    """(thread, what) of the launches that use the stream's control block, in order: "begin" writes it, the loop
    graph or the kernels of a round work on it."""
    names = {"k_begin": "begin", "k_big_": "round", "k_scan_": "round", "graph": "graph"}
    return [(tag, kind) for tag, _, stream, what, _ in fake_util.log(lib) if stream == STREAM
            for part, kind in names.items() if part in what]


@pytest.mark.parametrize("graph_loop", [1, 0])
@pytest.mark.parametrize("second", ["sort", "batch"])
def test_sorts_of_two_threads_on_one_stream(lib, graph_loop, second):
    """A sort's multi-block rounds run on the stream's control block, which the sort has written: no other sort of
    the stream may write it in between."""
    lib.ss_set_graph_loop(graph_loop)
    sets = [Set(BIG) for _ in range(2)]
    assert sets[0].sort(lib) == 0  # the stream's slot and its loop graph
    batch = ctypes.c_void_p()
    descs = (ss.SetDesc * 2)(sets[1].desc(), Set(100).desc())
    assert lib.ss_batch_create(descs, 2, None, ctypes.byref(batch)) == 0
    lib.fake_delay(b"k_begin", 2000)
    lib.fake_delay(b"k_big_classify", 500)
    lib.fake_clear_log()

    def first():
        lib.fake_set_tag(1)
        return [sets[0].sort(lib) for _ in range(8)]

    def other():
        lib.fake_set_tag(2)
        if second == "batch":
            return [lib.ss_batch_run(batch, ctypes.c_void_p(STREAM)) for _ in range(8)]
        return [sets[1].sort(lib) for _ in range(8)]

    assert fake_util.in_threads(first, other) == [[0] * 8] * 2
    owner = None
    parts = multi_block_parts(lib)
    assert sum(kind == "begin" for _, kind in parts) == 16
    for tag, kind in parts:
        if kind == "begin":
            owner = tag
        assert tag == owner, parts
    lib.ss_batch_destroy(batch)


def test_status_set_while_it_is_read(lib):
    """A kernel's error bit that arrives while a thread takes the stream's status word is still reported: by that
    thread or by the next one, never by none.  (Two bits one after the other, the second with the higher rank: it
    is reported whether the two are taken together or apart.)"""
    assert Set(100).sort(lib) == 0
    take = ctypes.cast(lib.ss_stream_status, ctypes.c_void_p)
    lib.fake_status_episodes.restype = ctypes.c_uint64
    lib.fake_status_episodes.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint32,
                                         ctypes.c_int, ctypes.c_uint64]
    timeout, too_deep, too_large = 1 << 1, 1 << 2, 4
    assert lib.fake_status_episodes(take, STREAM, timeout, too_deep, too_large, 300_000) == 0


def test_noalloc_of_two_threads(lib):
    """The calls without allocation share one scratch array: a call's launches and its wait come before the next
    call's first launch, on one stream or on two."""
    sets = [Set(BIG), Set(300)]
    for s in sets:
        assert lib.ss_sort_noalloc(s.ptrs[0], s.ptrs[1], s.n, 0, s.ptrs[2], s.ptrs[3], ctypes.c_void_p(STREAM)) == 0
    lib.fake_delay(b"k_begin", 1000)
    lib.fake_delay(b"k_rank_keys", 1000)
    lib.fake_clear_log()

    def call(tag, s, stream):
        lib.fake_set_tag(tag)
        return [lib.ss_sort_noalloc(s.ptrs[0], s.ptrs[1], s.n, 0, s.ptrs[2], s.ptrs[3], ctypes.c_void_p(stream))
                for _ in range(8)]

    assert fake_util.in_threads(lambda: call(1, sets[0], STREAM), lambda: call(2, sets[1], STREAM),
                                lambda: call(3, Set(BIG), STREAM + 1)) == [[0] * 8] * 3
    calls, fresh = 0, True
    for tag, _, _, what, _ in fake_util.log(lib):
        if fresh:
            owner, calls = tag, calls + 1
        assert tag == owner
        fresh = what == "wait"
    assert calls == 24


def test_captured_sort_has_its_own_control_block(lib):
    """A captured graph can be replayed on any stream at any time: its rounds run on a control block in the sort's
    workspace, not on that of the stream it was captured on, where other sorts may be running then."""
    s = Set(BIG)
    size = lib.ss_workspace_size(BIG, None)
    buf = np.zeros(size + 256, np.uint8)
    ws = (buf.ctypes.data + 255) & ~255
    opts = dict(workspace=ws, workspace_bytes=size)

    def control_blocks():
        lib.fake_clear_log()
        assert s.sort(lib, **opts) == 0
        return {first for _, _, _, what, first in fake_util.log(lib) if "k_big_" in what}

    plain = control_blocks()  # built with the stream's loop graph
    assert len(plain) == 1 and not ws <= min(plain) < ws + size
    lib.fake_capture(STREAM, 1)
    captured = control_blocks()
    lib.fake_capture(STREAM, 0)
    assert len(captured) == 1 and ws <= min(captured) < ws + size


def test_batch_destroyed_while_its_stream_is_asked(lib):
    """The status of a stream includes that of the last batch run on it, which another thread may destroy while the
    stream is waited for: its workspace, gone by then, is not read."""
    stop = []
    descs = (ss.SetDesc * 2)(Set(50).desc(), Set(100).desc())

    def run():
        for _ in range(100):
            batch = ctypes.c_void_p()
            assert lib.ss_batch_create(descs, 2, None, ctypes.byref(batch)) == 0
            assert lib.ss_batch_run(batch, ctypes.c_void_p(STREAM)) == 0
            time.sleep(0.001)
            assert lib.ss_batch_destroy(batch) == 0
        stop.append(True)
        return True

    def ask():
        return {lib.ss_stream_status(ctypes.c_void_p(STREAM)) for _ in iter(lambda: bool(stop), True)}

    lib.fake_delay(b"wait", 1500)
    assert fake_util.in_threads(run, ask, ask) == [True, {0}, {0}]
    assert lib.fake_stray_copies() == 0


@pytest.mark.parametrize("parts", [2, 4, 16])
def test_parts_are_checked_before_they_are_sorted(lib, parts):
    """A part of a host set is sorted while the characters of later ones are on their way.  Strings that reach into
    those must not be read: each part's layout is checked, and such strings left out, before its sort begins."""
    s = Set(BIG * parts)
    chars = np.zeros(s.n * 2, np.uint8)
    offsets = np.arange(s.n, dtype=np.uint64) * 2
    lib.fake_clear_log()
    o = ss.make_options(host_parts=parts)
    assert lib.ss_sort_host(chars.ctypes.data, chars.size, offsets.ctypes.data, s.n, s.ptrs[2], s.ptrs[3],
                            ctypes.byref(o), ctypes.c_void_p(STREAM)) == 0
    names = {"k_layout_check": "check", "k_layout_guard": "guard", "k_begin": "sort", "k_merge_prep": "records"}
    order = [kind for _, _, stream, what, _ in fake_util.log(lib) if stream == STREAM
             for part, kind in names.items() if part in what]
    assert order == ["check", "guard", "sort", "records"] * parts
