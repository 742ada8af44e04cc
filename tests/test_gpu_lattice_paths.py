"""GPU checks of the one-CTA lattice kernel where its parts change over:

* hop lists longer than the byte guide holds (more than 255 vectors), guide
  tables of every size, and steep towers whose buckets need the search;
* binary64 energies in fixed point, back in binary64 in the middle of a run
  (an energy of 6 or more), and never in it (a W that is no binary fraction);
* batches of more replicas than SMs, where CTAs choose their replica;
* the per-pair transforms of every side they are built for, and the binary64
  refresh of a group in one launch.

Binary64 chains equal the oracle's bit for bit; binary32 energies after a
refresh are within 2e-5 of their definition, the bound of the transform
refresh's own tests (2e-7 for the binary64 refresh: one binary32 rounding of
values below 4).
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


def _chain(p, **kw):
    return oracle.Chain(p["L"], nu=p["nu"], W=p["W"], xi=p["xi"], r_max=p["r_max"], T=p["T"],
                        E=p["E"], seed=p["seed"], replica=p.get("replica", 0), **kw)


def _equal(s, k, ch):
    n, eps, _, cnt = s.state(k)
    on, oeps, _ = ch.state()
    np.testing.assert_array_equal(n, on)
    np.testing.assert_array_equal(_bits(eps), _bits(oeps))
    oc = ch.counters()
    for f in ("rounds", "hops", "attempts", "P"):
        assert cnt[f] == oc[f], f


BASE = dict(nu=0.5, W=1.0, xi=1.0, T=0.05, E=0.01, seed=11)


@pytest.mark.parametrize("threads", [0, 256, 384, 512, 1024])
@pytest.mark.parametrize("case", [
    dict(L=32, r_max=14, xi=3.0),              # 612 vectors
    dict(L=34, r_max=9, xi=1.5),               # 252 vectors, even L
    dict(L=24, r_max=11, xi=40.0),             # nearly flat tower
    dict(L=64, r_max=8, xi=0.85, T=0.02),      # steep: the rim's weights are a few units
    dict(L=144, r_max=5),                      # the largest sides of one CTA: the
    dict(L=146, r_max=4),                      # finest guide table, and the next one
], ids=lambda c: f"L{c['L']}_r{c['r_max']}_xi{c.get('xi', 1.0)}")
def test_chain_equals_the_oracle(B, case, threads):
    p = dict(BASE, **case)
    s = B.System([p], precision=B.CG_FP64, block_threads=threads)
    try:
        assert s.run(150, 512) == B.CG_OK
        ch = _chain(p)
        ch.run(150, 512)
        _equal(s, 0, ch)
    finally:
        s.close()


@pytest.mark.parametrize("L,dim", [(32, 2), (48, 2), (12, 3)])
@pytest.mark.parametrize("W,shift", [(1.0, 0.0), (2.0, 3.0), (0.7, 0.0), (1.0, 5.0), (2.0, 3.6), (2.0, 3.95)],
                         ids=["fixed", "fixed_past_4", "fine_phi", "never_fixed", "past_6_L48",
                              "past_6_L32"])
def test_fixed_point_energies(B, L, dim, W, shift):
    # shift: a pattern of site energies that brings some eps near or past 6, the
    # fixed form's bound; with 3.6 (L = 48) and 3.95 (L = 32) the run starts
    # below it and hops push single sites over
    p = dict(BASE, L=L, r_max=3, W=W, T=0.5)
    s = B.System([dict(p, dim=dim)], precision=B.CG_FP64)
    try:
        ch = _chain(p, dim=dim)
        n, _, phi, _ = s.state(0)
        if shift:
            phi = phi.copy()
            phi[:: 7] += shift - 2.0
            phi[3:: 11] += 2.0 if shift > 4 else 1.0
            B.cg_write_state(s.h, 0, n, phi=phi)
            ch.set_state(n, phi)
            eps = s.state(0)[1]
            np.testing.assert_array_equal(_bits(eps), _bits(ch.state()[1]))
        for hops in (1, 60, 400):
            assert s.run(hops, 256) == B.CG_OK
            ch.run(hops, 256)
            n1, e1, _, _ = s.state(0)
            on, oe, _ = ch.state()
            np.testing.assert_array_equal(n1, on)
            np.testing.assert_array_equal(_bits(e1), _bits(oe))
    finally:
        s.close()


@pytest.mark.parametrize("R", [153, 304, 611])
def test_batches_past_one_replica_per_sm(B, R):
    # every replica runs once, whichever CTA took it
    reps = [dict(BASE, L=16, r_max=3, T=0.02 + 0.0005 * (s % 100), seed=s, replica=s)
            for s in range(R)]
    s = B.System(reps, precision=B.CG_FP64)
    try:
        for _ in range(2):                     # the second launch orders by the first
            assert s.run(40, 256) == B.CG_OK
        for k in range(R):
            assert s.observables(k)["hops"] == 80
        for k in (0, 1, 151, 152, R // 2, R - 2, R - 1):
            ch = _chain(reps[k])
            ch.run(40, 256)
            ch.run(40, 256)
            _equal(s, k, ch)
    finally:
        s.close()


@pytest.mark.parametrize("L,dim", [(L, 2) for L in [24] + list(range(16, 161, 16))] +
                         [(L, 3) for L in (16, 24, 32, 48, 64)])
@pytest.mark.parametrize("R", [1, 4, 9])
def test_transform_refresh_of_a_pair(B, L, dim, R):
    # sides that are neither 2^m nor 3 2^m go by the transforms from 8 replicas on
    fast = L in (16, 24, 32, 48, 64, 96, 128)
    if fast == (R == 9):
        pytest.skip("not by the transforms" if R < 9 else "covered by 1 and 4")
    if fast and dim == 3 and L > 32 and R > 1:
        R = 2
    reps = [dict(BASE, L=L, r_max=3, seed=s, replica=s, nu=0.25, dim=dim) for s in range(R)]
    s = B.System(reps, precision=B.CG_FP32, refresh_kind=B.CG_REFRESH_AUTO)
    try:
        assert s.run(60, 512) == B.CG_OK
        before = [s.state(k)[1] for k in range(R)]
        B.cg_refresh(s.h)
        for k in range(R):
            n, eps, phi, _ = s.state(k)
            exact = (ref.site_energies_fft3(n, phi, 0.25, L) if dim == 3
                     else ref.site_energies_fft(n, phi, 0.25, L))
            assert np.abs(eps - exact).max() <= 2e-5
            o = s.observables(k)
            assert o["refreshes"] == 1
            # the change reported is the largest one: eps_new is a binary32
            # rounding (at most 2^-24 of itself) of the sum it compares
            assert (abs(o["max_eps_err_last_refresh"] - np.abs(before[k] - eps).max())
                    <= 1.05 * 2.0 ** -24 * np.abs(eps).max())
    finally:
        s.close()


@pytest.mark.parametrize("L,dim,R", [(18, 2, 7), (42, 2, 5), (10, 3, 3)])
def test_binary64_refresh_of_a_group(B, L, dim, R):
    reps = [dict(BASE, L=L, r_max=3, seed=s, replica=s, dim=dim) for s in range(R)]
    s = B.System(reps, precision=B.CG_FP32, refresh_kind=B.CG_REFRESH_FP64)
    try:
        assert s.run(60, 512) == B.CG_OK
        B.cg_refresh(s.h)
        for k in range(R):
            n, eps, phi, _ = s.state(k)
            exact = (ref.site_energies_fft3(n, phi, 0.5, L) if dim == 3
                     else ref.site_energies_fft(n, phi, 0.5, L))
            assert np.abs(eps - exact).max() <= 2.5e-7
            assert s.observables(k)["refreshes"] == 1
    finally:
        s.close()
