"""GPU checks of two-electron hops on one CTA for every side that is fixed at
compile time and for its neighbours read at run time, both clocks, against the
serial oracle: binary64 states and counters bit for bit.  Cubic 32 is built in
binary32 alone: it follows the hops of its own log, and its energies their
definition.
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


@pytest.mark.parametrize("clock", [0, 1], ids=["deterministic", "gaussian"])
@pytest.mark.parametrize("L", [32, 34, 48, 64, 96, 128])
def test_binary64_pairs_of_every_side(B, L, clock):
    p = dict(L=L, nu=0.5, W=1.0, xi=1.0, r_max=4, T=0.1, E=0.01, seed=23, replica=1)
    s = B.System([p], precision=B.CG_FP64, pair_frac=0.3, pair_rmax=4, time_mode=clock)
    try:
        assert B.cg_group_shape(s.h, 0)["cluster"] == 1
        ch = oracle.Chain(L, nu=0.5, W=1.0, xi=1.0, r_max=4, T=0.1, E=0.01, seed=23, replica=1,
                          pair_frac=0.3, pair_rmax=4)
        ch.set_time_mode(clock)
        for hops in (1, 250):
            assert s.run(hops, 1024) == B.CG_OK
            ch.run(hops, 1024)
        n, eps, _, cnt = s.state(0)
        on, oeps, _ = ch.state()
        np.testing.assert_array_equal(n, on)
        np.testing.assert_array_equal(_bits(eps), _bits(oeps))
        oc = ch.counters()
        for f in ("rounds", "hops", "attempts", "P"):
            assert cnt[f] == oc[f], f
        if clock:
            assert cnt["time"] == oc["time"]
    finally:
        s.close()


@pytest.mark.parametrize("L", [30, 32])
def test_binary32_cubic_pairs(B, L):
    hops = 600
    p = dict(L=L, nu=0.5, W=1.0, xi=1.0, r_max=3, T=0.1, E=0.01, seed=29, replica=3, dim=3)
    s = B.System([p], precision=B.CG_FP32, pair_frac=0.3, pair_rmax=3)
    try:
        n0 = s.state(0)[0].astype(np.int64)
        rc, log = s.run_logged(hops, 1024)
        assert rc == B.CG_OK
        g = log[0]
        assert (g["k"] != 0xFFFFFFFF).any()
        for e in g:
            for a, b in ((e["i"], e["j"]), (e["k"], e["l"])):
                if a != 0xFFFFFFFF:
                    assert n0[a] == 1 and n0[b] == 0
                    n0[a], n0[b] = 0, 1
        n, eps, phi, _ = s.state(0)
        np.testing.assert_array_equal(n0, n)
        # an update rounds a difference and an energy below 8, at most twice a hop
        exact = ref.site_energies_fft3(n, phi, 0.5, L)
        assert np.abs(eps - exact).max() <= (2 * hops + 1) * 2 * 2.0 ** -22
    finally:
        s.close()
