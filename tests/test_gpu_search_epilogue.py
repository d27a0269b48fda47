"""Tensor-core searches where many images tie for the smallest distance.

Images drawn from a few different ones, so that the smallest distance occurs in many columns of a
tile, in several tiles and in several blocks: the smallest image index has to win, and only smaller
distances may count.  Column counts around the groups of 32 and the tiles of 128 and 256; equal to
the int64 oracle's results.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Q,H", [(1, 31), (40, 33), (128, 256), (130, 257), (520, 1000), (600, 5000)])
@pytest.mark.parametrize("N", [8, 16, 64])
@pytest.mark.parametrize("kinds", [1, 3, 40])
def test_ties(oracle_mod, Q, H, N, kinds):
    import torch

    import paper_2007_02306_gb300 as rici

    if N == 64 and H > 1000:
        H = 700
    rng = np.random.default_rng(Q + H + N + kinds)
    base = rng.integers(0, 12, (kinds, N, N)).astype(np.uint16)
    hay = base[rng.integers(0, kinds, H)]
    nd = base[rng.integers(0, kinds, Q)].copy()
    nd[::3, 1, 2] += 1
    m = rng.integers(0, H, Q).astype(np.int64)
    ref = oracle_mod.crss_search(nd, hay, m)
    got = rici.crss_search(*(torch.from_numpy(a).cuda() for a in (nd, hay, m)), mode=rici.SEARCH_TENSOR)
    assert rici.sync_status() == 0
    for k in ("rank", "true_distance", "top1"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k


@pytest.mark.parametrize("N", [8, 16])
@pytest.mark.parametrize("H", [(1 << 17) - 1, 1 << 17])
@pytest.mark.parametrize("mode", [3, 6])
def test_second_gemm_of_small_images(N, H, mode):
    """Either side of 2^26 pairs, where images with wider deltas move from the CUDA cores to a second
    GEMM; equal to the int64 form."""
    import torch

    import paper_2007_02306_gb300 as rici

    Q = 512
    g = torch.Generator().manual_seed(N + H)
    hay = torch.randint(0, 12, (H, N, N), generator=g).to(torch.int32)
    hay[::9, 1, N // 2:] += 60     # the split-square class
    hay[5::4001, 2, 3] += 500      # outside int8
    nd = hay[torch.randperm(H, generator=g)[:Q]].clone()
    nd[::2, 0, 1] += 3
    m = torch.randint(0, H, (Q,), generator=g)
    nd, hay = nd.to(torch.uint16).cuda(), hay.to(torch.uint16).cuda()
    a = rici.crss_search(nd, hay, m.cuda(), mode=mode)
    b = rici.crss_search(nd, hay, m.cuda(), mode=rici.SEARCH_EXACT_SLOW)
    assert rici.sync_status() == 0
    for k in ("rank", "true_distance", "top1"):
        assert torch.equal(a[k], b[k]), k
