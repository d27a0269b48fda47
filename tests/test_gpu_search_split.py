"""Tensor-core search of haystack images with deltas past the fp16 operands' square limit.

Deltas of 46..127 put an image in the split-square class; it is ranked by a second GEMM while the
partial-sum bound holds and there is room for its row, else by the CUDA-core kernel.  All results
equal the int64 oracle's.
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


def check(rici, oracle_mod, nd, hay, m, mode):
    import torch

    ref = oracle_mod.crss_search(nd, hay, m)
    cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (nd, hay, m.astype(np.int64))]
    got = rici.crss_search(*dev, mode=mode, counters=cnt)
    assert rici.sync_status() == 0
    for k in ("rank", "true_distance", "top1"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
    return cnt.cpu().numpy()


@pytest.mark.parametrize("N", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("H", [5, 300])
@pytest.mark.parametrize("mode", [3, 6])
def test_wide_deltas(rici, oracle_mod, N, H, mode):
    rng = np.random.default_rng(N)
    nd, hay, m = synth.images.needle_haystack_set(rng, min(H, 140), H, N)
    nd, hay = nd.astype(np.int64), hay.astype(np.int64)
    # every class: a step of 45, 46, 100, 127, 128 or 300 somewhere in most images (with 300 images
    # more rows than are kept for the split class), in some needles too
    for ims in (hay, nd):
        for i in range(len(ims)):
            step = (0, 45, 46, 100, 100, 127, 127, 128, 300)[rng.integers(9)]
            ims[i, rng.integers(N), rng.integers(1, N):] += step
    check(rici, oracle_mod, nd.astype(np.uint16), hay.astype(np.uint16), m, mode)


def test_no_room_left(rici, oracle_mod):
    """All images in the split class: the rows past the capacity run on the CUDA cores."""
    N, H = 16, 700
    rng = np.random.default_rng(4)
    nd, hay, m = synth.images.needle_haystack_set(rng, 50, H, N)
    hay = hay.astype(np.int64)
    hay[np.arange(H), rng.integers(0, N, H), N - 1] += 90
    cnt = check(rici, oracle_mod, nd, hay.astype(np.uint16), m, 3)
    assert cnt[0] > 0, "some pairs on the CUDA-core kernel"
    assert cnt[1] == 0, "no pair on the int64 kernel"


@pytest.mark.parametrize("n", [345, 346, 347])
def test_exact_at_the_partial_sum_bound(rici, oracle_mod, n):
    """n deltas of +127 against -127: partial sums up to n (127^2 + 254 * 127), just below 2^24 for
    n = 346 and outside the class for 347."""
    N = 64

    def stairs(step, count):
        im = np.zeros((N, N), np.int64)
        d = np.zeros(N * N, np.int64)
        at = np.arange(N * N).reshape(N, N)[:, 1::2].reshape(-1)[:count]
        d[at] = step
        back = at + 1
        back = back[(back % N) != 0]
        im += np.cumsum(d.reshape(N, N), axis=1)
        return im, at

    up, _ = stairs(127, n)
    down, at = stairs(127, n)
    down = down.max(axis=1, keepdims=True) - down  # deltas -127 at the same positions
    assert up.max() <= 65535 and down.min() >= 0
    nd = np.stack([down, up, np.zeros((N, N), np.int64)]).astype(np.uint16)
    hay = np.stack([up, down, np.zeros((N, N), np.int64), up]).astype(np.uint16)
    cnt = check(rici, oracle_mod, nd, hay, np.array([1, 3, 2]), 3)
    assert (cnt[0] > 0) == (n > 346)
