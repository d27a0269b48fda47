"""Meshes on either side of the one-block preparation's limits.

No triangle, one, counts around a chunk of 32, a group of 1,024 and the largest mesh the one-block
preparation takes (8,192), with every triangle in one bin and spread over many; images equal the
FP64 oracle's.
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


@pytest.mark.parametrize("nt", [0, 1, 31, 32, 33, 1023, 1024, 1025, 4097, 8191, 8192, 8193])
@pytest.mark.parametrize("spread", [0.0, 1.0, 50.0])
def test_triangle_counts(rici, oracle_mod, nt, spread):
    import torch

    rng = np.random.default_rng(nt)
    c = rng.uniform(-0.2, 0.2, size=(max(nt, 1), 1, 3))
    if spread == 0.0:
        c[:] = 0.1  # every centre in one bin
    elif spread > 1.0:
        c[::7] *= spread  # most of the others in the first bins
    v = (c + rng.uniform(-0.05, 0.05, size=(max(nt, 1), 3, 3))).reshape(-1, 3)
    if spread == 0.0:
        v = np.tile(v[:3], (max(nt, 1), 1)) * np.repeat(rng.uniform(0.5, 1.0, max(nt, 1)), 3)[:, None]
    ov = rng.uniform(-0.1, 0.1, size=(5, 3))
    V = np.concatenate([v, ov]).astype(np.float32)
    Nr = rng.normal(size=V.shape).astype(np.float32)
    t = np.arange(3 * nt).reshape(nt, 3).astype(np.int32)
    o = np.arange(len(v), len(V)).astype(np.int32)
    ref = oracle_mod.rici_fp64(V, Nr, t, o, 0.3, 24)
    got = rici.rici_generate(*[torch.from_numpy(np.ascontiguousarray(x)).cuda()
                               for x in (V, Nr, t, o)], 0.3, 24)
    assert rici.sync_status() == 0
    assert np.array_equal(got.cpu().numpy(), ref)


def test_bad_triangles_are_reported(rici):
    import torch

    v = np.zeros((4, 3), np.float32)
    v[1, 0] = v[2, 1] = 0.1
    v[3] = np.nan
    n = np.ones((4, 3), np.float32)
    for tri, status in (((0, 1, 4), 2), ((0, 1, -1), 2), ((0, 1, 3), 4)):
        t = np.array([(0, 1, 2), tri], np.int32)
        rici.rici_generate(*[torch.from_numpy(x).cuda()
                             for x in (v, n, t, np.zeros(1, np.int32))], 0.3, 16)
        assert rici.sync_status() == status
