"""GPU checks of binary64 energies in fixed point on both sides of the bound they
are held up to, 6: the runs' own energies, taken from the oracle hop by hop, show
which side each is on.  Started as multiples of 2^-60 below 6 (where the kernel
holds them as integers) and staying there, or carried past 6 by a hop in the
middle of the run (where it goes back to binary64): single and two-electron
hops, square and cubic, bit for bit.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

HOPS, M = 460, 256


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


@pytest.mark.parametrize("L,dim,pair,shift,crosses", [
    (32, 2, 0.0, 2.0, False), (32, 2, 0.0, 4.6, True), (48, 2, 0.0, 3.5, False),
    (48, 2, 0.0, 4.2, True), (12, 3, 0.0, 3.5, False), (12, 3, 0.0, 4.2, True),
    (32, 2, 0.3, 2.0, False), (32, 2, 0.3, 4.6, True), (48, 2, 0.3, 3.9, False),
    (48, 2, 0.3, 4.5, True), (12, 3, 0.3, 3.5, False), (12, 3, 0.3, 4.2, True)])
def test_energies_about_the_bound(B, L, dim, pair, shift, crosses):
    kw = dict(pair_frac=pair, pair_rmax=3) if pair else {}
    p = dict(L=L, nu=0.5, W=1.0, xi=1.0, r_max=3, T=0.5, E=0.01, seed=11, replica=0, dim=dim)
    ch = oracle.Chain(L, nu=0.5, W=1.0, xi=1.0, r_max=3, T=0.5, E=0.01, seed=11, replica=0,
                      dim=dim, **kw)
    # a checkerboard, whose energies are small, with some sites raised
    q = np.arange(L ** dim)
    n = ((q % L + q // L % L + q // (L * L)) % 2).astype(np.uint8)
    phi = ch.state()[2].copy()
    phi[::37] += shift
    ch.set_state(n, phi)
    e = ch.state()[1]
    assert L ** dim >= 1024 and np.abs(e).max() < 6.0
    assert np.all(e * 2.0 ** 60 == np.rint(e * 2.0 ** 60))
    s = B.System([p], precision=B.CG_FP64, **kw)
    try:
        B.cg_write_state(s.h, 0, n, phi=phi)
        np.testing.assert_array_equal(_bits(s.state(0)[1]), _bits(e))
        assert s.run(HOPS, M) == B.CG_OK
        past, pairs = [], 0
        for _ in range(HOPS):
            _, log = ch.run(1, M, log=True)
            pairs += int(log["k"][0] != 0xFFFFFFFF)
            past.append(np.abs(ch.state()[1]).max() >= 6.0)
        assert any(past) == crosses and (pairs > 0) == (pair > 0)
        if crosses:
            assert 10 < past.index(True) < HOPS - 10
        g, eps, _, cnt = s.state(0)
        on, oeps, _ = ch.state()
        np.testing.assert_array_equal(g, on)
        np.testing.assert_array_equal(_bits(eps), _bits(oeps))
        for f in ("rounds", "hops", "attempts", "P"):
            assert cnt[f] == ch.counters()[f], f
    finally:
        s.close()
