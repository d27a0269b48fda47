"""The line between a search in one launch and the general sequence, by the work of either: calls to both
sides of it, for images that a warp reads 8 pixels at a time, unaligned ones and other resolutions.
Each takes the form that is faster there (its launches are counted) and equals the int64 oracle.
"""
import numpy as np
import pytest

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


def dev(a, off=0):
    import torch

    a = np.ascontiguousarray(a)
    if a.dtype != np.uint16:
        return torch.from_numpy(a).cuda()
    b = torch.zeros(a.size + off, dtype=torch.int16, device="cuda")
    b[off:].copy_(torch.from_numpy(a.view(np.int16).reshape(-1)))
    return b[off:].view(a.shape).view(torch.uint16)


@pytest.mark.parametrize("Q,H,N,off,small", [
    # 8 pixels per lane
    (4000, 4, 8, 0, True), (8000, 1, 8, 0, False), (4000, 16, 8, 0, False), (1000, 64, 8, 0, True),
    (4000, 4, 32, 0, True), (4000, 16, 32, 0, False), (256, 256, 32, 0, True), (65536, 1, 32, 0, False),
    (600, 16, 64, 0, True), (16000, 1, 64, 0, False), (4000, 1, 128, 0, True),
    # 1 pixel per lane
    (1, 64, 20, 0, True), (300, 17, 20, 0, True), (1000, 1, 24, 0, False), (1, 1, 33, 0, True),
    (256, 240, 33, 0, False), (1, 1, 48, 0, False), (1, 1, 100, 0, False), (4000, 1, 5, 0, False),
    (60, 64, 32, 1, True), (64, 256, 32, 1, False), (1, 17, 64, 1, False), (300, 128, 16, 1, True),
])
def test_each_side(rici, oracle_mod, Q, H, N, off, small):
    rng = np.random.default_rng(Q + H + N)
    hay = rng.integers(0, 9, size=(H, N, N)).astype(np.uint16)
    hay[H // 2:] = hay[: H - H // 2]
    m = rng.integers(0, H, size=Q)
    nd = hay[m]
    nd[::2, 0, N // 2:] += 3
    ref = oracle_mod.crss_search(nd, hay, m)
    q, h, t = dev(nd, off), dev(hay, off), dev(m)
    before = rici.binding.kernel_launches()
    got = rici.crss_search(q, h, t)
    assert rici.sync_status() == 0
    assert (rici.binding.kernel_launches() - before == 1) == small
    for k in ("rank", "true_distance", "top1"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
