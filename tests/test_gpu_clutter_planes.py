"""Clutter measure: triangles that lie in an end plane of the support volume, which is closed.

Flat triangles at exactly |beta| = R/2 and one representable height to either side of it, inside the
cylinder, across its side and around the whole disk, triangles with an edge or a vertex in the plane,
and a box whose faces lie in both planes, for normals along each axis; compared with the FP64 oracle.
Heights and coordinates are exact in binary, so both sides decide the same predicates; areas differ by
FP64 rounding alone (a few operations per triangle: within 1e-13 of R^2 for these sizes).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

R = 0.5
H = 0.25


@pytest.fixture(scope="module")
def rici():
    import torch

    import paper_2007_02306_gb300 as p
    from paper_2007_02306_gb300 import build

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    p.load_library()
    return p


def triangles(kind, z):
    if kind == "inside":
        return [[(.125, 0, z), (0, .125, z), (.125, .125, z)], [(-.25, -.125, z), (.25, 0, z), (0, .25, z)]]
    if kind == "across":  # through the cylinder's side
        return [[(.25, 0, z), (1, 0, z), (.25, .5, z)]]
    if kind == "around":  # the whole disk
        return [[(-4, -4, z), (4, -4, z), (0, 4, z)]]
    if kind == "edge":    # the rest of the triangle within the volume, then past the plane
        return [[(.125, 0, z), (0, .125, z), (.125, .125, z / 2)],
                [(.125, 0, z), (0, .125, z), (.125, .125, z * 2)]]
    return [[(.125, 0, z), (0, .125, z / 2), (.125, .125, z / 2)],   # a vertex
            [(.125, 0, z), (0, .125, z * 2), (.125, .125, z * 2)]]


def check(rici, oracle_mod, tri, axis):
    """Areas around the origin, tri turned so that its z axis is the normal."""
    import torch

    tri = np.asarray(tri, np.float64)
    V = np.concatenate([np.roll(tri.reshape(-1, 3), axis + 1, axis=1), np.zeros((2, 3))]).astype(np.float32)
    N = np.zeros_like(V)
    N[-2, axis], N[-1, axis] = 1, -1
    t = np.arange(3 * len(tri), dtype=np.int32).reshape(-1, 3)
    o = np.array([len(V) - 2, len(V) - 1], np.int32)
    a, b = rici.clutter_areas(*(torch.from_numpy(x).cuda() for x in (V, N, t, o)), R, 3)
    assert rici.sync_status() == 0
    ra, rb = oracle_mod.clutter_areas(V, N, t, o, R, 3)
    for got, ref in ((a, ra), (b, rb)):
        assert (np.abs(got.cpu().numpy() - ref) <= 1e-13 * R * R).all(), (got.cpu().numpy(), ref)
    return ra


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("z", [H, -H])
@pytest.mark.parametrize("kind", ["inside", "across", "around", "edge", "vertex"])
def test_in_an_end_plane(rici, oracle_mod, kind, z, axis):
    for tri in triangles(kind, z):
        past = abs(tri[2][2]) > H  # only an edge or a vertex of it is in the volume
        assert ((check(rici, oracle_mod, [tri], axis) > 0) == (not past)).all()


@pytest.mark.parametrize("z", [H, -H])
def test_next_heights(rici, oracle_mod, z):
    inner, outer = (float(np.nextafter(np.float32(z), np.float32(x))) for x in (0, 4 * z))
    assert (check(rici, oracle_mod, triangles("inside", inner), 2) > 0).all()
    assert (check(rici, oracle_mod, triangles("inside", outer), 2) == 0).all()


def test_box_between_the_planes(rici, oracle_mod):
    c = [(x, y, z) for x in (-.125, .25) for y in (-.25, .125) for z in (-H, H)]
    quads = [(0, 1, 3, 2), (4, 5, 7, 6), (0, 1, 5, 4), (2, 3, 7, 6), (0, 2, 6, 4), (1, 3, 7, 5)]
    tri = [[c[q[i]] for i in k] for q in quads for k in ((0, 1, 2), (0, 2, 3))]
    a = check(rici, oracle_mod, tri, 2)
    assert np.allclose(a, 4 * .375 * .5 + 2 * .375 * .375, rtol=1e-15)
