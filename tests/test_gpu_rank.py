"""Sorts of a few thousand strings by counting (33..4096 strings with default
options): sizes at the edges of the tiles, strings told apart inside, at the
end of and past the 32 characters that are compared, caps, both encodings;
against the oracle and against the distribution steps (which explicit options
select)."""
import numpy as np
import pytest

import gen
from gpu_util import assert_parity, from_strings, gpu_sort, to_device

pytestmark = pytest.mark.gpu

SIZES = [33, 34, 127, 128, 129, 255, 256, 257, 1000, 1025, 4095, 4096]


def _set(kind, n):
    rng = np.random.default_rng(n)
    if kind == "url":
        return gen.url_set(n, n)
    if kind == "bytes":
        return gen.random_set(n, n, 0, 40, 1, 255)
    if kind == "binary":  # many equal strings
        return gen.random_set(n, n, 0, 9, ord("0"), ord("1"))
    if kind == "dna":
        return gen.dna_suffix_set(n, n, nblocks=min(1, n // 3000), blocklen=1000)
    if kind == "ladder":  # prefixes of one string, ends on and around the word edges
        a = bytes(rng.integers(97, 123, 90).astype(np.uint8))
        return from_strings([a[:int(x)] for x in rng.integers(0, 90, n)])
    pre = bytes(rng.integers(97, 123, int(kind)).astype(np.uint8))
    return from_strings([pre + bytes(rng.integers(97, 99, int(rng.integers(0, 9))).astype(np.uint8)) for _ in range(n)])


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", ["url", "bytes", "binary", "dna", "ladder", "7", "24", "31", "32", "33", "200"])
def test_small_sets(kind, n):
    s = _set(kind, n)
    p, l = gpu_sort(s)
    assert_parity(s, p, l)
    q, m = gpu_sort(s, small_cutoff=64)
    assert np.array_equal(p, q) and np.array_equal(l, m)
    q, _ = gpu_sort(s, with_lcp=False)
    assert np.array_equal(p, q)


@pytest.mark.parametrize("cap", [1, 8, 31, 32, 33, 70])
def test_caps(cap):
    s = _set("200", 777)
    s.max_len = cap
    assert_parity(s, *gpu_sort(s))


@pytest.mark.parametrize("n", [33, 500, 4096])
@pytest.mark.parametrize("cap", [0, 20, 21, 84, 85, 500])
def test_dna_codes(n, cap):
    s = _set("dna", n)
    s.max_len = cap
    assert_parity(s, *gpu_sort(s, dna=True))


def test_offsets_past_2_to_the_32():
    import torch

    import paper_1808_00963_gb300 as ss
    far = 1 << 32
    chars = torch.zeros(far + (1 << 20), dtype=torch.uint8, device="cuda")
    s = _set("33", 600)
    host = torch.from_numpy(s.chars)
    chars[:host.numel()] = host.cuda()
    chars[far:far + host.numel()] = host.cuda()
    offs = torch.from_numpy(s.offsets.view(np.int64).copy())
    offs[::2] += far
    p, l = ss.sort(chars, offs.cuda())
    assert_parity(s, p.cpu().numpy().view(np.uint32), l.cpu().numpy().view(np.uint32))


def test_exact_workspace():
    import torch

    import paper_1808_00963_gb300 as ss
    s = _set("url", 3000)
    chars, offsets = to_device(s)
    need = ss.workspace_size(s.n)
    buf = torch.empty(need, dtype=torch.uint8, device="cuda")
    p, l = ss.sort(chars, offsets, workspace=buf.data_ptr(), workspace_bytes=need)
    assert_parity(s, p.cpu().numpy().view(np.uint32), l.cpu().numpy().view(np.uint32))
    with pytest.raises(ss.SortError):
        ss.sort(chars, offsets, workspace=buf.data_ptr(), workspace_bytes=need - 256)
