"""Clutter measure: triangles on every path of its classification.

Triangles inside the support volume, across its end planes only, across its side only, across
both, beside, above and around it (the whole disk inside one triangle), slivers and triangles
without area, at very small and very large scales; compared with the FP64 oracle, each point's
areas to 1e-9 of its A_all (the bound of test_gpu_clutter.py: a triangle touching the volume may add
a sliver of 1e-15..1e-11 of R^2 on one side only).
"""
import numpy as np
import pytest

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


def triangles(kind, rng, n=400):
    c = rng.uniform(-0.7, 0.7, size=(n, 1, 3)) * R
    d = rng.uniform(-1, 1, size=(n, 3, 3)) * R
    if kind == "small":
        return c * 2 + 0.05 * d
    if kind == "planes":  # near the axis, through z = +-R/2 and past both
        return c * [[[0.5, 0.5, 0]]] + d * [[[0.2, 0.2, 3.0]]]
    if kind == "side":    # between the planes, through the cylinder's side
        return c * [[[2.0, 2.0, 0.5]]] + d * [[[0.5, 0.5, 0.1]]]
    if kind == "large":   # larger than the volume, some around the whole disk
        return c * [[[1.0, 1.0, 0.6]]] + d * [[[20.0, 20.0, 0.4]]]
    if kind == "huge":
        return c + d * 10.0 ** rng.uniform(0, 4, size=(n, 1, 1))
    # slivers, and every third without area
    t = c + d
    t[:, 2] = t[:, 1] + 1e-7 * d[:, 2]
    t[::3, 2] = t[::3, 1]
    return t


@pytest.mark.parametrize("kind", ["small", "planes", "side", "large", "huge", "slivers"])
@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e12])
def test_paths(rici, oracle_mod, kind, scale):
    import torch

    rng = np.random.default_rng(11)
    tri = triangles(kind, rng)
    n = len(tri)
    ov = np.concatenate([np.zeros((4, 3)), rng.uniform(-0.1, 0.1, size=(6, 3))])
    on = np.concatenate([[(0, 0, 1), (0, 0, -1), (0, 0, 0), (1, 2, 0)], rng.normal(size=(6, 3))])
    # a quarter disk's worth of plane, so that no point's A_all is zero
    quad = np.array([[(0, 0, 0), (R, 0, 0.01), (0, R, 0.02)]])
    V = np.concatenate([tri.reshape(-1, 3), quad.reshape(-1, 3), ov]) * scale
    V = V.astype(np.float32)
    Nr = np.concatenate([np.zeros((3 * n + 3, 3)), on]).astype(np.float32)
    t = np.arange(3 * n + 3).reshape(-1, 3).astype(np.int32)
    o = np.arange(3 * n + 3, len(V)).astype(np.int32)
    r, obj = float(np.float32(R * scale)), 3 * (n // 2)
    args = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (V, Nr, t, o)]
    ga, gb = rici.clutter_areas(*args, r, obj)
    assert rici.sync_status() == 0
    ra, rb = oracle_mod.clutter_areas(V, Nr, t, o, r, obj)
    assert (ra > 0).all()
    for got, ref in ((ga, ra), (gb, rb)):
        err = np.abs(got.cpu().numpy() - ref)
        assert (err <= 1e-9 * ra).all(), (err / ra).max()
