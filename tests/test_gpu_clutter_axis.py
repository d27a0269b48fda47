"""Clutter measure: triangles whose edges pass through the axis, with a corner of the clipped polygon on it.

An edge that meets the axis in an end plane leaves a corner there whose coordinates are rounding alone;
corners and edges on the axis between the planes, and grid triangles all around, against the
oracle to 1e-9 of each point's area (the bound of test_gpu_clutter.py).
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


def compare(rici, oracle_mod, tri, nrm, R, scale=1.0):
    import torch

    tri = np.asarray(tri, np.float64)
    n, k = len(tri), len(nrm)
    base = np.array([[(0.1, 0, 0.01), (0, 0.1, 0.02), (0.1, 0.1, 0.03)]]) * R  # no point's area is zero
    V = (np.concatenate([tri, base]).reshape(-1, 3) * scale).astype(np.float32)
    V = np.concatenate([V, np.zeros((k, 3), np.float32)])
    Nr = np.concatenate([np.zeros((3 * n + 3, 3)), nrm]).astype(np.float32)
    t = np.arange(3 * n + 3, dtype=np.int32).reshape(-1, 3)
    o = np.arange(3 * n + 3, len(V)).astype(np.int32)
    args = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (V, Nr, t, o)]
    r = float(np.float32(R * scale))
    a, _ = rici.clutter_areas(*args, r, 0)
    assert rici.sync_status() == 0
    ref, _ = oracle_mod.clutter_areas(V, Nr, t, o, r, 0)
    err = np.abs(a.cpu().numpy() - ref) / ref
    assert (err <= 1e-9).all(), (err.max(), int(err.argmax()))


UP = [(0, 0, 1), (0, 0, -1)]


@pytest.mark.parametrize("scale", [1.0, 0.3, 1e-12, 1e12])
def test_edges_that_meet_the_axis_in_an_end_plane(rici, oracle_mod, scale):
    rng = np.random.default_rng(1)
    d = rng.integers(-8, 9, size=(200, 2)) / 4.0
    h = rng.integers(1, 9, size=(200, 2)) / 4.0
    z = np.where(rng.random(200) < 0.5, 0.5, -0.5)
    # from (-f d, z - f h) to (g d, z + g h): through (0, 0, z)
    lo = np.c_[-d * h[:, :1], z - h[:, 0]]
    hi = np.c_[d * h[:, 1:], z + h[:, 1]]
    third = rng.integers(-8, 9, size=(200, 3)) / 4.0
    for i in range(0, 200, 10):  # few at a time: none hides behind the others' areas
        compare(rici, oracle_mod, np.stack([lo, hi, third], 1)[i:i + 10], UP, 1.0, scale)


def test_two_of_the_grid(rici, oracle_mod):
    compare(rici, oracle_mod, [[(0.5, 1.5, -3.0), (-0.5, -1.5, 2.0), (-1.0, -1.0, 0.5)]], UP, 1.0)
    compare(rici, oracle_mod, [[(4, 3, 5), (-4, -2, -5), (2, 2, -0.5)]], [(0, -1, 0), (0, 1, 0)], 1.0)


@pytest.mark.parametrize("seed", range(6))
def test_grid_triangles(rici, oracle_mod, seed):
    rng = np.random.default_rng(seed)
    tri = rng.integers(-8, 9, size=(300, 3, 3)) / 4.0
    tri[::3, 0, :2] = 0  # a corner on the axis
    nrm = [(0, 0, 1), (0, 0, -1), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0)]
    for i in range(0, 300, 30):
        compare(rici, oracle_mod, tri[i:i + 30], nrm, float(rng.choice([0.5, 0.75, 1.0, 1.5])))
