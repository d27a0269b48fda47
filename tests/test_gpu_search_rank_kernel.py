"""The tensor-core kernel of large searches (more than 512 needles: operands in memory) at the bounds of
its class and at ragged tiles, and haystack images of the split-square class past their capacity.

Smaller needle sets take the kernel that builds the haystack's operands itself; each check counts its
launches or its pairs by kernel to be where it wants to be.  Equal to the int64 oracle.
"""
import numpy as np
import pytest

import synth

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


def search(rici, nd, hay, m, mode=3):
    """Results, (dense pair rows, int64 pairs) and the launches of a call."""
    import torch

    cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (nd, hay, np.asarray(m, np.int64))]
    before = rici.binding.kernel_launches()
    got = rici.crss_search(*dev, mode=mode, counters=cnt)
    launches = rici.binding.kernel_launches() - before
    assert rici.sync_status() == 0
    return {k: got[k].cpu().numpy() for k in KEYS}, cnt.cpu().numpy(), launches


def check(rici, oracle_mod, nd, hay, m):
    ref = oracle_mod.crss_search(nd, hay, m)
    got, cnt, launches = search(rici, nd, hay, m)
    for k in KEYS:
        assert np.array_equal(got[k], ref[k]), k
    return cnt, launches


def test_which_kernel(rici, oracle_mod):
    nd, hay, m = synth.images.needle_haystack_set(np.random.default_rng(1), 513, 600, 64)
    _, few = check(rici, oracle_mod, nd[:512], hay, m[:512])
    _, many = check(rici, oracle_mod, nd, hay, m)
    assert many == few + 1  # the haystack's encode


def test_class_at_its_partial_sum_bound(rici, oracle_mod):
    """n deltas of +45 against -127: partial sums just below 2^24 for n = 1,246, outside the class for
    1,247 (130 times over)."""
    N = 64

    def image(n, step, base):
        img = np.zeros((N, N), np.int64)
        flat = np.zeros(N * (N - 1), np.int64)
        flat[:n] = step
        img[:, 1:] = flat.reshape(N, N - 1)
        return (base + np.cumsum(img, axis=1)).astype(np.uint16)

    noise = synth.images.rici_like_images(np.random.default_rng(14), 6, N)
    zero = np.zeros((N, N), np.uint16)
    for n, dense in ((1246, False), (1247, True)):
        hay = np.stack([image(n, 45, 0), image(n, 45, 0), zero, *noise])
        nd = np.tile(np.stack([image(n, -127, 127 * 63), zero, noise[0], image(n, -127, 127 * 63)]), (130, 1, 1))
        cnt, _ = check(rici, oracle_mod, nd, hay, np.tile([0, 2, 3, 1], 130))
        assert (cnt[0] > 0) == dense and cnt[1] == 0


@pytest.mark.parametrize("Q,H", [(513, 1), (600, 129), (641, 257), (1000, 3000)])
@pytest.mark.parametrize("N", [8, 32, 64])
def test_ragged_tiles(rici, oracle_mod, Q, H, N):
    _, hay, _ = synth.images.needle_haystack_set(np.random.default_rng(11), 1, H, N)
    rng = np.random.default_rng(H)
    m = rng.integers(0, H, size=Q)
    nd = hay[m].astype(np.int64)
    nd[::2, rng.integers(N), N // 2:] += 2
    check(rici, oracle_mod, nd.astype(np.uint16), hay, m)


@pytest.mark.parametrize("N", [32, 64])
@pytest.mark.parametrize("Q", [50, 600])
def test_split_rows_past_their_capacity(rici, oracle_mod, N, Q):
    """256 rows are kept for up to 700 images: all of 256 images on the second GEMM, and of 700 the rest
    on the CUDA cores (about 444 / 700 of the pair rows that all of them take there)."""
    H = 700
    rng = np.random.default_rng(4)
    nd, hay, m = synth.images.needle_haystack_set(rng, Q, H, N, tail_image_fraction=0.0)
    hay = hay.astype(np.int64)
    hay[np.arange(H), rng.integers(0, N, H), N - 1] += 90
    hay = hay.astype(np.uint16)
    cnt, _ = check(rici, oracle_mod, nd, hay[:256], m % 256)
    assert cnt[0] == 0 and cnt[1] == 0
    cnt, _ = check(rici, oracle_mod, nd, hay, m)
    _, all_dense, _ = search(rici, nd, hay, m, mode=1)
    assert 0.4 * all_dense[0] < cnt[0] < 0.9 * all_dense[0] and cnt[1] == 0
