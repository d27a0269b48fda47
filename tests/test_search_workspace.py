"""Workspace of the tensor-core search: what an image of a large haystack takes, and results where the rows of
its split-square images and, after them, the int8 deltas of the images of neither class share one place.
"""
import numpy as np
import pytest

import synth


@pytest.mark.parametrize("mode", [0, 3])
@pytest.mark.parametrize("N", [8, 32, 64, 128])
def test_bytes_per_image(N, mode):
    """The fp16 operand row, the int8 deltas, and lists and flags of 32 bytes at most."""
    import paper_2007_02306_gb300 as p
    from paper_2007_02306_gb300 import build

    build.build()
    size = p.load_library().crss_search_workspace_size
    for H in (6144, 100_000, 2_500_000):
        per = (size(600, 2 * H, N, mode) - size(600, H, N, mode)) / H
        assert per <= 2 * N * N * 2 + N * N + 32


@pytest.mark.gpu
@pytest.mark.parametrize("Q", [300, 700])
@pytest.mark.parametrize("H", [1500, 6400, 9001])
def test_shared_place(oracle_mod, Q, H):
    import torch

    import paper_2007_02306_gb300 as p
    from paper_2007_02306_gb300 import build

    build.build()
    N = 32
    rng = np.random.default_rng(H)
    nd, hay, m = synth.images.needle_haystack_set(rng, Q, H, N)
    hay = hay.astype(np.int64)
    kind = rng.integers(0, 12, size=H)  # split-square, past its capacity at H = 1500; outside int8
    hay[kind <= 2, 5, N // 2:] += 100
    hay[kind == 3, 7, N // 2:] += 500
    hay = hay.astype(np.uint16)
    for i in range(0, H, 7):  # int8, but of neither tensor-core class (partial sums past 2^24)
        hay[i] = np.cumsum(rng.choice([-90, 90], size=(N, N)), axis=1) + 3000
    ref = oracle_mod.crss_search(nd, hay, m)
    cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
    got = p.crss_search(*(torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (nd, hay, m)), mode=3,
                        counters=cnt)
    assert p.sync_status() == 0
    assert cnt[0] > 0 and cnt[1] > 0
    for k in ("rank", "true_distance", "top1"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
