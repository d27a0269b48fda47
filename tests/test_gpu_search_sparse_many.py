"""Sparse-needle and automatic search with many needles of every kind.

Sparse, empty, dense and wide needles together, haystacks that end inside and at a tile of 128 images,
every packed resolution, images outside int8; with and without work counters (a kernel of its own).
Equal to the int64 oracle's results.
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


@pytest.mark.parametrize("Q,H,N", [(1024, 31, 8), (1024, 33, 16), (1025, 128, 32), (1100, 129, 64),
                                   (7, 97, 64), (3000, 1500, 16), (1024, 40, 128)])
@pytest.mark.parametrize("mode", [4, 6])
def test_many_needles(rici, oracle_mod, Q, H, N, mode):
    import torch

    rng = np.random.default_rng(Q + H + N)
    pool = synth.images.rici_like_images(rng, max(Q, H), N, changes_per_row=0.4)
    synth.images.add_plateaus(rng, pool, 0.1, 0.1)
    m = rng.integers(0, H, Q)
    hay = pool[:H].copy()
    nd = hay[m].copy()
    nd[::5] = pool[rng.integers(0, len(pool), len(nd[::5]))]
    nd[1], nd[2] = 0, np.arange(N * N).reshape(N, N) % 7
    nd[3, 0, N // 2:] = 1000
    hay[H - 1, 1, 1:] = 65535
    ref = oracle_mod.crss_search(nd, hay, m)
    cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
    for counters in (None, cnt):  # the counting variant is a kernel of its own
        got = rici.crss_search(dev(nd), dev(hay), dev(m.astype(np.int64)), mode=mode,
                               counters=counters)
        assert rici.sync_status() == 0
        for k in ("rank", "true_distance", "top1"):
            assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
    c = cnt.cpu().numpy()
    assert c[3] >= c[0] >= 0
