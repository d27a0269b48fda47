"""Top-1 where distances reach 2^32 - 1, the limit of the packed minimum.

Images of uniform 16-bit noise lie 10^10 and more apart, so a needle without a near image gets its
top-1 from the exact minimum over its haystack: hundreds of such needles, more than the grid has
blocks, in one scene and in several; needles with a near image among them (their packed minimum is
exact); equal distances past the limit (the smaller index).  All equal to the int64 oracle.
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


def dev(*arrays):
    import torch

    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def noise(rng, Q, H, N):
    """Every third needle has a near image, which is not its true match; every fifth image is there twice."""
    nd = rng.integers(0, 65536, size=(Q, N, N)).astype(np.uint16)
    hay = rng.integers(0, 65536, size=(H, N, N)).astype(np.uint16)
    near = rng.integers(1, H, size=len(nd[::3]))
    hay[near] = nd[::3] ^ 1
    hay[1::5] = hay[(np.arange(1, H, 5) + 7) % H]
    return nd, hay, np.zeros(Q, np.int64)


@pytest.mark.parametrize("Q,H,N", [(300, 60, 33), (1500, 70, 8), (2600, 40, 16), (3, 300, 64)])
@pytest.mark.parametrize("mode", [0, 1, 2, 3, 4, 5, 6])
def test_past_the_packed_limit(rici, oracle_mod, Q, H, N, mode):
    import torch

    nd, hay, m = noise(np.random.default_rng(Q), Q, H, N)
    ref = oracle_mod.crss_search(nd, hay, m, return_distances=True)
    best = ref["distances"].min(axis=1)
    assert (best >= 2 ** 32).any() and (best < 2 ** 20).any()
    cnt = torch.zeros(4, dtype=torch.int64, device="cuda")  # (with counters: not the one-launch form)
    got = rici.crss_search(*dev(nd, hay, m), mode=mode, counters=cnt)
    assert rici.sync_status() == 0
    for k in KEYS:
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k


def test_several_scenes(rici, oracle_mod):
    scenes = [noise(np.random.default_rng(s), Q, H, 16) for s, (Q, H) in enumerate([(500, 30), (1, 9), (900, 50)])]
    got = rici.crss_search_batch([dict(zip(("needles", "haystack", "true_match"), dev(*s))) for s in scenes], 16)
    assert rici.sync_status() == 0
    for s, g in zip(scenes, got):
        ref = oracle_mod.crss_search(*s)
        for k in KEYS:
            assert np.array_equal(g[k].cpu().numpy(), ref[k]), k
