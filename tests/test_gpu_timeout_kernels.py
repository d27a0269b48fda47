"""Bounded waits of both tensor-core kernels: the one of few needles (which builds the haystack's operands
itself) and the one of more than 512, each with the first load of block 0 withheld.  The call must end
by itself and report the time-out, and searches by both kernels after it must be exact.
"""
import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Q,N", [(200, 64), (600, 64), (200, 8), (512, 128)])
def test_withheld_load(oracle_mod, Q, N):
    import torch

    import paper_2007_02306_gb300 as p
    from paper_2007_02306_gb300 import build

    build.build()
    p.load_library()
    nd, hay, m = synth.images.needle_haystack_set(np.random.default_rng(4), max(Q, 600), 1500, N)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    q, h, t = d(nd), d(hay), d(m)
    t0 = time.time()
    p.crss_search(q[:Q], h, t[:Q], mode=p.SEARCH_TENSOR | p.binding.SEARCH_TEST_WITHHOLD_LOAD)
    assert p.sync_status() & p.binding.ERR_TIMEOUT
    assert time.time() - t0 < 30.0
    ref = oracle_mod.crss_search(nd, hay, m)
    for n in (200, 600):
        r = p.crss_search(q[:n], h, t[:n], mode=p.SEARCH_TENSOR)
        assert p.sync_status() == 0
        for k in ("rank", "true_distance", "top1"):
            assert np.array_equal(r[k].cpu().numpy(), ref[k][:n]), k
