"""The work queue's ring taken round more than once: subsets that are put back
at every level, since at each of them one more string leaves the others.  (A
subset whose keys are all equal is taken further in place, without the queue:
identical strings, however long, make no such pushes.)"""
import numpy as np
import pytest

import gen
import oracle
from gpu_util import to_device

pytestmark = pytest.mark.gpu

TAIL_WORD = 4  # the workspace starts with the control words; this one counts the pushes


def _ladders(groups, rest, levels, shared, seed):
    """Per group `rest` copies of one string of 8 * levels characters behind `shared` characters, and for every level
    a string that leaves it there; `rest + levels` strings a group, in a mixed order."""
    rng = np.random.default_rng(seed)
    parts, offsets, at = [], [], 0
    for g in range(groups):
        stem = b"%08d" % (g * 7919 % 100000) + bytes(rng.integers(97, 123, shared - 8 + 8 * levels).astype(np.uint8))
        texts = [stem] + [stem[:shared + 8 * k + int(rng.integers(0, 8))] + b"A" for k in range(levels)]
        for k, t in enumerate(texts):
            offsets += [at] * (rest if k == 0 else 1)
            parts.append(t + b"\0")
            at += len(t) + 1
    chars = np.frombuffer(b"".join(parts), np.uint8).copy()
    return gen.StringSet(chars, rng.permutation(np.array(offsets, np.uint64)))


@pytest.mark.parametrize("shape", ["cutoff_64", "default"])
def test_more_pushes_than_slots(shape):
    import torch

    import paper_1808_00963_gb300 as ss
    # more strings than the cutoff stay together to the last level: groups * levels pushes, 4096 slots
    s, opts = {"cutoff_64": (_ladders(128, 65, 64, 8, 1), dict(small_cutoff=64, big_threshold=1 << 20)),
               "default": (_ladders(8, 1025, 640, 16, 2), {})}[shape]
    chars, offsets = to_device(s)
    need = ss.workspace_size(s.n, **opts)
    for _ in range(2):
        ws = torch.full((need,), 0xAB, dtype=torch.uint8, device="cuda")
        perm, lcp = ss.sort(chars, offsets, workspace=ws.data_ptr(), workspace_bytes=need, **opts)
        pushes = int(ws[:256].view(torch.int32)[TAIL_WORD])
        slots = max(4096, s.n // (opts.get("small_cutoff", 1024) + 1) + 1024)
        assert pushes > slots == 4096, (pushes, slots)
        want_p, want_l = oracle.sort(s.chars, s.offsets, 0)
        assert np.array_equal(perm.cpu().numpy().view(np.uint32), want_p)
        assert np.array_equal(lcp.cpu().numpy().view(np.uint32), want_l)
    if shape == "default":  # the same steps in the fixed scratch of the call without allocation
        for _ in range(2):
            p, l = ss.sort_noalloc(chars, offsets)
            assert torch.equal(p, perm) and torch.equal(l, lcp)
