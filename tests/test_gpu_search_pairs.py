"""Distances of single pairs, by both forms of the warp's loop: 8 pixels per lane (resolutions of whole
passes, 16-byte aligned images) and 1 (any other resolution or alignment), where each is used: true
distances, the distance matrix, the exact top-1 past 2^32 - 1, in one scene and in two, one of them
unaligned.  Equal to the int64 oracle.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KEYS = ("rank", "true_distance", "top1")


@pytest.fixture(scope="module")
def rici():
    import torch

    import paper_2007_02306_gb300 as p
    from paper_2007_02306_gb300 import build

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    p.load_library()
    return p


def dev(a, off=0):
    """The array on the device, off bytes past a 16-byte boundary."""
    import torch

    a = np.ascontiguousarray(a)
    if a.dtype != np.uint16:
        return torch.from_numpy(a).cuda()
    b = torch.zeros(a.size + 8, dtype=torch.int16, device="cuda")
    assert b.data_ptr() % 16 == 0
    t = b[off // 2:off // 2 + a.size]
    t.copy_(torch.from_numpy(a.view(np.int16).reshape(-1)))
    return t.view(a.shape).view(torch.uint16)


def images(N, Q=70, H=90):
    """Half of the images small steps, half 16-bit noise; needles partly near some image."""
    rng = np.random.default_rng(N)
    hay = rng.integers(0, 9, size=(H, N, N)).astype(np.uint16)
    hay[::2] = rng.integers(0, 65536, size=hay[::2].shape)
    nd = rng.integers(0, 65536, size=(Q, N, N)).astype(np.uint16)
    nd[::3] = hay[rng.integers(0, H, size=len(nd[::3]))] ^ 1
    return nd, hay, rng.integers(0, H, size=Q)


@pytest.mark.parametrize("N", [2, 8, 16, 24, 32, 33, 64, 100, 128])
@pytest.mark.parametrize("off", [(0, 0), (2, 0), (0, 14), (8, 6)])
def test_one_scene(rici, oracle_mod, N, off):
    import torch

    nd, hay, m = images(N)
    ref = oracle_mod.crss_search(nd, hay, m, return_distances=True)
    for mode in (0, 2, 3):
        for counters in (None, torch.zeros(4, dtype=torch.int64, device="cuda")):
            got = rici.crss_search(dev(nd, off[0]), dev(hay, off[1]), dev(m), mode=mode, counters=counters,
                                   return_distances=True)
            assert rici.sync_status() == 0
            for k in KEYS + ("distances",):
                assert np.array_equal(got[k].cpu().numpy(), ref[k]), (mode, k)


@pytest.mark.parametrize("N", [8, 16, 64])
def test_two_scenes(rici, oracle_mod, N):
    nd, hay, m = images(N)
    scenes = [dict(needles=dev(nd, o), haystack=dev(hay, o), true_match=dev(m)) for o in (0, 4)]
    ref = oracle_mod.crss_search(nd, hay, m)
    for got in rici.crss_search_batch(scenes, N):
        for k in KEYS:
            assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
    assert rici.sync_status() == 0
