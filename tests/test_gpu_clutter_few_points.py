"""Clutter measure of few oriented points in a large mesh: areas are prepared only where a point's walk
reaches.  Meshes of one and of many groups of 1,024 records (a ragged last one), points in and far
from the mesh, radii from a fraction of a triangle to several times the mesh, bad and non-finite
points among them.  Each point's areas equal the oracle's, and those of a call with so many points that
every area is prepared; the tolerances are those of FP64 sums of the same terms in another order.
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


def mesh(n, rng):
    """n triangles of a ball, every 50th ten times the size, in blobs, and their vertices' normals."""
    c = rng.normal(size=(n, 1, 3)) * 0.3 + rng.choice([-1.0, 1.0], size=(n, 1, 3))
    t = c + 0.02 * rng.normal(size=(n, 3, 3)) * np.where(np.arange(n) % 50 == 0, 10.0, 1.0)[:, None, None]
    v = t.reshape(-1, 3).astype(np.float32)
    v[-3:] = [(50, 0, 0), (50, 0.01, 0), (50, 0, 0.01)]  # a triangle and its points far away
    return v, rng.normal(size=v.shape).astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(-1, 3)


@pytest.mark.parametrize("n", [700, 30001, (1 << 17) - 1, 131072 + 77])
@pytest.mark.parametrize("R", [0.004, 0.1, 1.0, 200.0])
def test_few_points(rici, oracle_mod, n, R):
    import torch

    rng = np.random.default_rng(n)
    v, nr, t = mesh(n, rng)
    pts = np.r_[rng.integers(0, 3 * n, 6), 3 * n - 1].astype(np.int32)
    obj = 3 * (n // 3)
    d = [torch.from_numpy(x).cuda() for x in (v, nr, t)]
    ra, rb = oracle_mod.clutter_areas(v, nr, t, pts, R, obj)
    many = np.r_[pts, rng.integers(0, 3 * n, 1025 - len(pts))].astype(np.int32)
    ma, mb = rici.clutter_areas(*d, torch.from_numpy(many).cuda(), R, obj)
    for k in (1, 3, len(pts)):
        a, b = rici.clutter_areas(*d, torch.from_numpy(pts[:k].copy()).cuda(), R, obj)
        for got, whole, ref in ((a, ma, ra), (b, mb, rb)):
            got = got.cpu().numpy()
            assert (np.abs(got - whole[:k].cpu().numpy()) <= 1e-12 * ra[:k]).all()
            assert (np.abs(got - ref[:k]) <= 1e-9 * ra[:k]).all()
    assert rici.sync_status() == 0


def test_points_without_a_place(rici):
    import torch

    v, nr, t = mesh(1 << 17, np.random.default_rng(1))
    v = np.concatenate([v, [[np.nan, 0, 0]]]).astype(np.float32)
    nr = np.concatenate([nr, [[0, 0, 1]]]).astype(np.float32)
    d = [torch.from_numpy(x).cuda() for x in (v, nr, t)]
    o = torch.tensor([len(v) - 1, len(v), -1, 5], dtype=torch.int32, device="cuda")
    a, b = rici.clutter_areas(*d, o, 0.5, 9000)
    assert rici.sync_status() == rici.binding.ERR_INDEX_OUT_OF_RANGE | rici.binding.ERR_NONFINITE_INPUT
    ra, rb = rici.clutter_areas(*d, o[3:].contiguous(), 0.5, 9000)
    assert rici.sync_status() == 0
    assert a[:3].isnan().all() and b[:3].isnan().all()
    assert abs(float(a[3]) - float(ra)) <= 1e-12 * float(ra) and float(ra) > 0
