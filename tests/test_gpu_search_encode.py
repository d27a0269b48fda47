"""Search encoders at the edges of their vector loads and groups of 32 images.

Image arrays that start off the 16-byte boundary of the 8-pixel loads (scalar loads then), every
packed resolution, haystacks that end inside, at and past a group of 32, and pixel values up to
65,535 (deltas past every narrow class).  All results equal the int64 oracle's.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rici():
    import torch

    import paper_2007_02306_gb300 as p
    from paper_2007_02306_gb300 import build

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    p.load_library()
    return p


def place(a, offset):
    """The images on the GPU, `offset` elements past a 256-byte boundary."""
    import torch

    flat = torch.zeros(a.size + offset, dtype=torch.int16, device="cuda")
    flat[offset:] = torch.from_numpy(np.ascontiguousarray(a).view(np.int16).reshape(-1)).cuda()
    return flat[offset:].view(a.shape).view(torch.uint16)


@pytest.mark.parametrize("N,H", [(8, 31), (16, 33), (32, 64), (64, 95), (128, 40)])
@pytest.mark.parametrize("offset", [0, 1, 4])
@pytest.mark.parametrize("mode", [1, 3, 4, 6])
def test_alignment_and_group_edges(rici, oracle_mod, N, H, offset, mode):
    import torch

    rng = np.random.default_rng(N + H)
    nd, hay, m = synth.images.needle_haystack_set(rng, 19, H, N, tail_image_fraction=0.3,
                                                  tail_row_fraction=0.2)
    hay[1, 2, 3:] = 65535
    nd[2, N - 1, ::2] = 65535
    hay[H - 1] = rng.integers(0, 65536, size=(N, N))
    ref = oracle_mod.crss_search(nd, hay, m)
    # work counters keep even small calls on the form under test
    cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
    got = rici.crss_search(place(nd, offset), place(hay, offset + 1 if offset else 0),
                           torch.from_numpy(m.astype(np.int64)).cuda(), mode=mode, counters=cnt)
    assert rici.sync_status() == 0
    for k in ("rank", "true_distance", "top1"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
