"""Whole small searches in one launch (the forms that leave the choice to the library).

Sizes at and just past the rule's limits, every resolution class, unaligned images, equal
distances, bad true-match indices and the distance matrix; equal to the int64 oracle's results and
to the int64 kernel's.
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


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("Q,H,N", [(1, 1, 2), (3, 7, 12), (5, 9, 8), (40, 40, 64), (9, 64, 64),
                                   (9, 65, 64), (7, 16, 128), (7, 17, 128), (256, 256, 32),
                                   (200, 257, 32), (30, 257, 16), (100, 200, 33)])
@pytest.mark.parametrize("mode", [0, 6])
def test_sizes(rici, oracle_mod, Q, H, N, mode):
    rng = np.random.default_rng(Q + H + N)
    nd, hay, m = synth.images.needle_haystack_set(rng, Q, H, N, tail_image_fraction=0.2)
    nd[0], hay[0] = 0, 0
    nd[-1, 0, N // 2:] = 65535
    hay[H // 2:] = hay[: H - H // 2]  # equal distances: best rank, smallest index
    ref = oracle_mod.crss_search(nd, hay, m, return_distances=True)
    got = rici.crss_search(dev(nd), dev(hay), dev(m.astype(np.int64)), mode=mode,
                           return_distances=True)
    assert rici.sync_status() == 0
    for k in ("rank", "true_distance", "top1", "distances"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k


@pytest.mark.parametrize("offset", [1, 8])
def test_unaligned_and_identity_match(rici, oracle_mod, offset):
    import torch

    rng = np.random.default_rng(3)
    _, hay, _ = synth.images.needle_haystack_set(rng, 1, 60, 32)
    nd = hay[:50]
    flat = torch.zeros(hay.size + offset, dtype=torch.int16, device="cuda")
    flat[offset:] = torch.from_numpy(hay.view(np.int16).reshape(-1)).cuda()
    h = flat[offset:].view(hay.shape).view(torch.uint16)
    got = rici.crss_search(h[:50], h)
    assert rici.sync_status() == 0
    ref = oracle_mod.crss_search(nd, hay, np.arange(50))
    for k in ("rank", "true_distance", "top1"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k


def test_bad_match_is_reported(rici):
    rng = np.random.default_rng(5)
    nd, hay, m = synth.images.needle_haystack_set(rng, 6, 20, 16)
    m = m.astype(np.int64)
    m[2], m[4] = -1, 20
    got = rici.crss_search(dev(nd), dev(hay), dev(m))
    assert rici.sync_status() == 2
    slow = rici.crss_search(dev(nd), dev(hay), dev(m), mode=2)
    assert rici.sync_status() == 2
    for k in ("rank", "true_distance", "top1"):
        a, b = got[k].cpu().numpy(), slow[k].cpu().numpy()
        assert np.array_equal(a, b), k
        assert a[2] == -1 and a[4] == -1
