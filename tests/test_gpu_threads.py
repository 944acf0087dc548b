"""Several threads sorting on one stream, threads of the call without
allocation, and a captured sort replayed while its stream sorts: every result
equals that of the sort alone."""
import threading

import numpy as np
import pytest

import gen
from gpu_util import assert_parity, to_device

pytestmark = pytest.mark.gpu

SIZES = [20_000, 90_000, 9_000, 300_000, 500, 40_000]


@pytest.fixture(scope="module")
def alone():
    """[(chars, offsets, (perm, lcp))] of sets sorted one at a time."""
    import torch

    import paper_1808_00963_gb300 as ss
    out = []
    for i, n in enumerate(SIZES):
        s = gen.url_set(n, 60 + i) if i % 2 else gen.random_set(n, 60 + i)
        chars, offsets = to_device(s)
        p, l = ss.sort(chars, offsets)
        torch.cuda.synchronize()
        assert_parity(s, p.cpu().numpy().view(np.uint32), l.cpu().numpy().view(np.uint32))
        out.append((chars, offsets, (p, l)))
    return out


def _run(threads, work):
    failed = []

    def guarded(w):
        try:
            failed.extend(work(w))
        except Exception as e:  # (would end its thread only)
            failed.append((w, e))

    ts = [threading.Thread(target=guarded, args=(w,)) for w in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failed


def _same(out, want):
    import torch
    return all(torch.equal(a, b) for a, b in zip(out, want))


def test_sorts_and_batches_of_many_threads_on_one_stream(alone):
    import torch

    import paper_1808_00963_gb300 as ss
    stream = torch.cuda.Stream()

    def work(w):
        done = []
        with torch.cuda.stream(stream):
            for r in range(20):
                k = (w + r) % len(alone)
                chars, offsets, want = alone[k]
                out = tuple(torch.empty_like(x) for x in want)
                if w % 3 == 2:
                    batch = ss.Batch([(chars, offsets, 0, *out)], own_workspace=True)
                    batch.run(stream)
                    done.append((k, out, batch))
                else:
                    ss.sort(chars, offsets, out=out, stream=stream, sync=False)
                    done.append((k, out, None))
        stream.synchronize()
        return [(w, k) for k, out, _ in done if not _same(out, alone[k][2])]

    _run(6, work)
    ss.stream_status(stream)


def test_noalloc_of_many_threads(alone):
    import torch

    import paper_1808_00963_gb300 as ss
    shared = torch.cuda.Stream()
    small = [x for x in alone if x[1].numel() <= ss.NOALLOC_MAX_STRINGS]

    def work(w):
        stream = shared if w % 2 else torch.cuda.Stream()
        bad = []
        for r in range(20):
            chars, offsets, want = small[(w + r) % len(small)]
            with torch.cuda.stream(stream):
                out = tuple(torch.empty_like(x) for x in want)
                ss.sort_noalloc(chars, offsets, out=out, stream=stream)
                if not _same(out, want):
                    bad.append((w, r))
        return bad

    _run(4, work)


def test_replay_beside_sorts_of_the_captured_stream(alone):
    import torch

    import paper_1808_00963_gb300 as ss
    home, other = torch.cuda.Stream(), torch.cuda.Stream()
    chars, offsets, want = alone[1]
    out = tuple(torch.empty_like(x) for x in want)
    need = ss.workspace_size(offsets.numel())
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    args = dict(out=out, sync=False, workspace=ws.data_ptr(), workspace_bytes=need)
    with torch.cuda.stream(home):
        ss.sort(chars, offsets, stream=home, **args)  # the stream's slot
    home.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=home):
        ss.sort(chars, offsets, stream=home, **args)
    done = []
    for r in range(20):
        for x in out:
            x.fill_(-1)
        torch.cuda.synchronize()
        k = r % len(alone)
        mine = tuple(torch.empty_like(x) for x in alone[k][2])
        with torch.cuda.stream(other):
            graph.replay()
        with torch.cuda.stream(home):
            ss.sort(*alone[k][:2], out=mine, stream=home, sync=False)
        torch.cuda.synchronize()
        done.append(_same(out, want) and _same(mine, alone[k][2]))
    assert all(done)
    ss.stream_status(home)
