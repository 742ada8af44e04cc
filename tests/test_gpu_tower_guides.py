"""GPU checks of the lattice kernels' tower samplers, every guide size among them,
against the oracle's binary search: each threshold, each edge of a guide bucket of
12, 13 and 14 bits and of a search bound of 7 bits, with their neighbours, the ends
of the 32-bit range, the null region, and random words.  More vectors than the byte
guide can name (255), flat towers and steep ones, square and cubic.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_5026_gb300 import build, binding
    build.build()
    binding.load()
    return binding


@pytest.mark.parametrize("L,dim,r_max,xi", [
    (16, 2, 1, 1.0), (32, 2, 9, 1.5), (32, 2, 10, 1.5), (64, 2, 8, 0.85), (16, 2, 4, 0.5),
    (64, 2, 20, 10.0), (24, 2, 11, 40.0), (96, 2, 40, 6.0), (8, 3, 3, 0.5), (18, 3, 8, 2.0),
    (18, 3, 8, 30.0)])
def test_samplers_agree_with_the_oracle(B, L, dim, r_max, xi):
    p = dict(L=L, nu=0.5, W=1.0, xi=xi, r_max=r_max, T=0.05, E=0.0, seed=1, dim=dim)
    s = B.System([p], precision=B.CG_FP32)
    try:
        ch = oracle.Chain(L, nu=0.5, W=1.0, xi=xi, r_max=r_max, T=0.05, E=0.0, seed=1, dim=dim)
        C = np.cumsum(ch.vectors()[2].astype(np.uint64)).astype(np.int64)
        edges = [np.arange(1 << b, dtype=np.int64) << (32 - b) for b in (7, 14)]
        pts = np.concatenate([[0, 1, (1 << 32) - 1]] + [a + d for a in [C] + edges
                                                        for d in (-2, -1, 0, 1)])
        rnd = np.random.default_rng(3).integers(0, 1 << 32, size=1 << 18)
        x1 = np.concatenate([pts, rnd])
        x1 = x1[(x1 >= 0) & (x1 < (1 << 32))].astype(np.uint32)
        np.testing.assert_array_equal(B.cg_debug_tower(s.h, 0, x1), ch.tower(x1))
    finally:
        s.close()
