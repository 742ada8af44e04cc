"""GPU checks of two-electron hops on lattices that just fit the shared memory
of one CTA: they are taken, stay on one CTA, and run the serial chain.

A guide table finer than the room left for the kernel's static part would
push these lattices to a cluster, or out: 202 and 146 are no multiples of 4,
so no cluster takes them either.
"""
import numpy as np
import pytest

import oracle
from tests import physics_ref as ref

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


def _bits(a):
    return np.ascontiguousarray(a, dtype=np.float64).view(np.uint64)


BASE = dict(nu=0.5, W=1.0, xi=1.0, T=0.1, E=0.01, seed=17, replica=2)


@pytest.mark.parametrize("L,r_max", [(144, 5), (146, 7)])
def test_binary64_pairs_at_the_edge_of_one_cta(B, L, r_max):
    p = dict(BASE, L=L, r_max=r_max)
    s = B.System([p], precision=B.CG_FP64, pair_frac=0.3, pair_rmax=4)
    try:
        assert B.cg_group_shape(s.h, 0)["cluster"] == 1
        assert s.run(200, 1024) == B.CG_OK
        ch = oracle.Chain(L, nu=0.5, W=1.0, xi=1.0, r_max=r_max, T=0.1, E=0.01, seed=17,
                          replica=2, pair_frac=0.3, pair_rmax=4)
        ch.run(200, 1024)
        n, eps, _, cnt = s.state(0)
        on, oeps, _ = ch.state()
        np.testing.assert_array_equal(n, on)
        np.testing.assert_array_equal(_bits(eps), _bits(oeps))
        for f in ("rounds", "hops", "attempts", "P"):
            assert cnt[f] == ch.counters()[f], f
    finally:
        s.close()


@pytest.mark.parametrize("L,r_max,dim", [(202, 6, 2), (200, 9, 2), (30, 9, 3)])
def test_binary32_pairs_at_the_edge_of_one_cta(B, L, r_max, dim):
    # eps after a few hops: one binary32 rounding each of an energy below 8 per
    # update, 2 updates a hop at most
    hops = 100
    p = dict(BASE, L=L, r_max=r_max, dim=dim)
    s = B.System([p], precision=B.CG_FP32, pair_frac=0.3, pair_rmax=4)
    try:
        assert B.cg_group_shape(s.h, 0)["cluster"] == 1
        assert s.run(hops, 1024) == B.CG_OK
        n, eps, phi, cnt = s.state(0)
        assert cnt["hops"] == hops and n.sum() == n.size // 2
        exact = (ref.site_energies_fft3(n, phi, 0.5, L) if dim == 3
                 else ref.site_energies_fft(n, phi, 0.5, L))
        assert np.abs(eps - exact).max() <= (2 * hops + 1) * 2 * 2.0 ** -22
    finally:
        s.close()
