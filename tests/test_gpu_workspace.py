"""A workspace made for n strings serves fewer strings too, also where fewer
strings need more of some of its parts (ranking by counting, smaller tiles,
more merge samples)."""
import pytest

import gen
import paper_1808_00963_gb300 as ss
from gpu_util import assert_parity, to_device


def test_sizes_do_not_shrink():
    lib = ss.load()
    ns = sorted({k * s + d for k in (1, 2, 3, 5, 7, 8, 9, 12) for s in (33, 1024, 4096, 8192, 350208, 420246)
                 for d in (-2, -1, 0, 1, 2, 1000)})
    for sizes in ([ss.workspace_size(n) for n in ns],
                  [ss.workspace_size(n, big_threshold=32768, small_cutoff=128) for n in ns],
                  [lib.ss_merge_workspace_size((ss.RunDesc * 2)(*[ss.RunDesc(8, 8, n // 2, 0)] * 2), 2, 0) for n in ns]):
        assert all(a <= b for a, b in zip(sizes, sizes[1:]))


@pytest.mark.gpu
@pytest.mark.parametrize("n, made_for", [(4096, 4097), (4000, 5000), (4096, 4096), (349_000, 352_000),
                                         (690_000, 710_000), (8192, 8193)])
def test_sort(n, made_for):
    import torch
    nbytes = ss.workspace_size(made_for)
    s = gen.random_set(n, n)
    chars, offsets = to_device(s)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    perm, lcp = ss.sort(chars, offsets, workspace=ws.data_ptr(), workspace_bytes=nbytes)
    assert_parity(s, perm.cpu().numpy().view("uint32"), lcp.cpu().numpy().view("uint32"))
