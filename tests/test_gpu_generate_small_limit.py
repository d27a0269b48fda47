"""The largest mesh that one block prepares and the smallest one past it: two launches and more, and images
and clutter areas equal to the oracle's.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt,one_block", [(5119, True), (5120, True), (5121, False), (8192, False)])
def test_limit(oracle_mod, nt, one_block):
    import torch

    import paper_2007_02306_gb300 as rici
    from paper_2007_02306_gb300 import build

    build.build()
    rng = np.random.default_rng(nt)
    v = (rng.uniform(-0.3, 0.3, size=(nt, 1, 3)) + rng.uniform(-0.05, 0.05, size=(nt, 3, 3))).reshape(-1, 3)
    V, Nr = v.astype(np.float32), rng.normal(size=v.shape).astype(np.float32)
    t = np.arange(3 * nt, dtype=np.int32).reshape(nt, 3)
    o = rng.integers(0, 3 * nt, 9).astype(np.int32)
    d = [torch.from_numpy(x).cuda() for x in (V, Nr, t, o)]
    before = rici.binding.kernel_launches()
    got = rici.rici_generate(*d, 0.2, 32)
    assert (rici.binding.kernel_launches() - before == 2) == one_block
    assert np.array_equal(got.cpu().numpy(), oracle_mod.rici_fp64(V, Nr, t, o, 0.2, 32))
    a, b = rici.clutter_areas(*d, 0.2, 3000)
    ra, rb = oracle_mod.clutter_areas(V, Nr, t, o, 0.2, 3000)
    for x, r in ((a, ra), (b, rb)):
        assert (np.abs(x.cpu().numpy() - r) <= 1e-9 * ra).all()
    assert rici.sync_status() == 0
