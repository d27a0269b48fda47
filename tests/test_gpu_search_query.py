"""Searches with few needles, whose haystack operands are built inside the GEMM kernel.

Needle and haystack counts around the tiles of 128, every resolution (rows shorter, equal to and
longer than the 64-pixel chunks), images of every class on both sides, a bad true-match index, and a
haystack off the 16-byte boundary (the general path); equal to the int64 oracle's results.
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


def dataset(Q, H, N, seed):
    rng = np.random.default_rng(seed)
    pool = max(Q, H)
    nd, hay, m = synth.images.needle_haystack_set(rng, Q, pool, N, tail_image_fraction=0.1,
                                                  tail_row_fraction=0.1)
    hay = hay[:H].copy()
    m = m % H
    hay[0, 1, N // 2:] += 46
    hay[H // 2, 2, 1:] += 128
    hay[H - 1, N - 1, ::2] = 65535
    nd[Q - 1, 0, 1::2] = 40000
    return nd, hay, m.astype(np.int64)


def same(got, ref):
    for k in ("rank", "true_distance", "top1"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k


@pytest.mark.parametrize("Q,H", [(1, 1), (3, 127), (100, 128), (128, 129), (129, 700), (256, 255),
                                 (512, 260), (513, 130)])
@pytest.mark.parametrize("N", [8, 16, 32, 64, 128])
def test_sizes(rici, oracle_mod, Q, H, N):
    nd, hay, m = dataset(Q, H, N, Q + H + N)
    got = rici.crss_search(dev(nd), dev(hay), dev(m), mode=rici.SEARCH_TENSOR)
    assert rici.sync_status() == 0
    same(got, oracle_mod.crss_search(nd, hay, m))


def test_many_tiles_per_block(rici, oracle_mod):
    """More haystack tiles than SMs: every stage, buffer and phase of the ring wraps."""
    N, H = 16, 152 * 128 * 3 + 77
    nd, hay, m = dataset(20, H, N, 9)
    got = rici.crss_search(dev(nd), dev(hay), dev(m))
    assert rici.sync_status() == 0
    same(got, oracle_mod.crss_search(nd, hay, m))


@pytest.mark.parametrize("offset", [1, 8])
def test_alignment_and_bad_match(rici, oracle_mod, offset):
    import torch

    nd, hay, m = dataset(30, 200, 32, 2)
    flat = torch.zeros(hay.size + offset, dtype=torch.int16, device="cuda")
    flat[offset:] = torch.from_numpy(hay.view(np.int16).reshape(-1)).cuda()
    ref = oracle_mod.crss_search(nd, hay, m)
    bad = m.copy()
    bad[5] = 200
    got = rici.crss_search(dev(nd), flat[offset:].view(hay.shape).view(torch.uint16), dev(bad),
                           mode=rici.SEARCH_TENSOR)
    assert rici.sync_status() == 2
    keep = np.arange(30) != 5
    for k in ("rank", "true_distance", "top1"):
        g = got[k].cpu().numpy()
        assert np.array_equal(g[keep], ref[k][keep]), k
        assert g[5] == -1
