"""Generation where its FP32 and float-pair predicates are undecided most often.

Inputs that put vertices on layers, edges on circle radii, triangles flat between two layers or on
one, chords through the axis, and positions far from or close to zero, at the resolutions where
item and interval counts are smallest, odd and largest.  Every image equals the FP64 oracle's, and
the FP64 mode's, bit for bit (the definition has no tolerance).
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

R = 0.5


@pytest.fixture(scope="module")
def rici():
    import torch

    import paper_2007_02306_gb300 as p
    from paper_2007_02306_gb300 import build

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    p.load_library()
    return p


def _soup(kind, rng):
    """Vertices and triangles around the origin."""
    if kind == "grid":       # heights and distances on layers and radii exactly
        v = rng.integers(-40, 41, size=(500, 3)) / 128.0
        t = np.stack([rng.choice(500, 3, replace=False) for _ in range(1200)])
        return v, t
    if kind == "flat":       # triangles in planes of nearly one height, some on a layer
        n = 400
        c = rng.uniform(-0.4, 0.4, size=(n, 1, 3))
        d = rng.uniform(-0.1, 0.1, size=(n, 3, 3))
        d[:, :, 2] *= 10.0 ** rng.uniform(-9, -2, size=(n, 1))
        c[::2, :, 2] = rng.integers(-40, 41, size=(n - n // 2, 1)) / 128.0
        return (c + d).reshape(-1, 3), np.arange(3 * n).reshape(n, 3)
    if kind == "needle":     # slivers and chords past the axis, tiny and very long
        n = 400
        c = rng.uniform(-0.1, 0.1, size=(n, 1, 3))
        d = rng.normal(size=(n, 3, 3)) * 10.0 ** rng.uniform(-6, 2, size=(n, 1, 1))
        d[:, 2] = d[:, 1] + 1e-4 * d[:, 2]
        return (c + d).reshape(-1, 3), np.arange(3 * n).reshape(n, 3)
    s = synth.tiny_scene(4)
    return s.vertices.astype(np.float64), s.triangles


@pytest.mark.parametrize("N", [1, 2, 31, 64, 127, 128])
@pytest.mark.parametrize("kind,shift,scale", [("grid", 0.0, 1.0), ("flat", 0.0, 1.0),
                                              ("needle", 0.0, 1.0), ("needle", 0.0, 1e-8),
                                              ("mesh", 3000.0, 1.0), ("mesh", 0.0, 1e8)])
def test_undecided_items_stay_exact(rici, oracle_mod, N, kind, shift, scale):
    import torch

    rng = np.random.default_rng(17)
    v, t = _soup(kind, rng)
    ov = np.concatenate([np.zeros((3, 3)), rng.uniform(-0.2, 0.2, size=(5, 3)),
                         rng.integers(-8, 9, size=(4, 3)) / 128.0])
    on = np.concatenate([[(0, 0, 1), (0, 0, -2), (1, 0, 0)], rng.normal(size=(5, 3)),
                         [(0, 0, 1), (0, 0, 0), (0, 3, 0), (1, 1, 0)]])
    V = ((np.concatenate([v, ov]) + shift) * scale).astype(np.float32)
    Nr = np.concatenate([np.zeros_like(v), on]).astype(np.float32)
    o = np.arange(len(v), len(V))
    r = float(np.float32(R * scale))
    ref = oracle_mod.rici_fp64(V, Nr, t.astype(np.int32), o, r, N)
    args = [torch.from_numpy(np.ascontiguousarray(x)).cuda()
            for x in (V, Nr, t.astype(np.int32), o.astype(np.int32))]
    got = rici.rici_generate(*args, r, N)
    slow = rici.rici_generate(*args, r, N, mode=rici.GEN_FP64)
    assert rici.sync_status() == 0
    assert np.array_equal(got.cpu().numpy(), ref)
    assert np.array_equal(slow.cpu().numpy(), ref)
