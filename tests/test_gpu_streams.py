"""Sorts of several streams at once: their kernels share the GPU, so blocks of
one kernel start late, also after others of the same kernel have ended."""
import threading

import numpy as np
import pytest

import gen
from gpu_util import assert_parity, to_device

pytestmark = pytest.mark.gpu


def test_sorts_on_many_streams():
    import torch

    import paper_1808_00963_gb300 as ss
    sets = [gen.url_set(n, 40 + i) if i % 2 else gen.random_set(n, 40 + i)
            for i, n in enumerate([3_000, 60_000, 150_000, 250_000, 400_000, 20_000])]
    dev = [to_device(s) for s in sets]
    want = [ss.sort(c, o, max_len=s.max_len) for s, (c, o) in zip(sets, dev)]
    torch.cuda.synchronize()
    for s, (p, l) in zip(sets, want):
        assert_parity(s, p.cpu().numpy().view(np.uint32), l.cpu().numpy().view(np.uint32))
    failed = []

    def work(w):
        stream = torch.cuda.Stream()
        out = []
        with torch.cuda.stream(stream):
            for r in range(24):
                k = (w + r) % len(sets)
                res = tuple(torch.empty_like(x) for x in want[k])
                ss.sort(*dev[k], max_len=sets[k].max_len, out=res, stream=stream, sync=False)
                out.append((k, res))
        stream.synchronize()
        for k, res in out:
            if not all(torch.equal(a, b) for a, b in zip(res, want[k])):
                failed.append((w, k))

    threads = [threading.Thread(target=work, args=(w,)) for w in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
