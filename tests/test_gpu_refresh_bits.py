"""GPU checks that the transform refresh adds phi and the correction of nu with
all of their bits: the largest change it reports follows a change of phi of
2^-38 and 2^-47 at that site, and of nu below binary32's last place, to 2^-49
(binary64 values near 1; what the transforms return is the same in both runs).
Values that binary32 cannot hold take the binary64 sum.
"""
import numpy as np
import pytest

from tests import physics_ref as ref

pytestmark = pytest.mark.gpu

SIDES = [(8, 2), (16, 2), (24, 2), (64, 2), (128, 2), (192, 2), (8, 3), (16, 3), (32, 3)]


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_5026_gb300 import build, binding
    build.build()
    binding.load()
    return binding


def _system(B, L, dim, nu=0.5, R=2):
    return B.System([dict(L=L, nu=nu, W=1.0, xi=1.0, r_max=2, T=0.05, E=0.0, seed=5 + k,
                          replica=k, dim=dim) for k in range(R)], precision=B.CG_FP32)


def _change(B, s, k, n, eps, phi):
    B.cg_write_state(s.h, k, n, eps=eps, phi=phi)
    B.cg_refresh(s.h)
    return s.observables(k)["max_eps_err_last_refresh"]


@pytest.mark.parametrize("L,dim", SIDES)
def test_change_follows_every_bit_of_phi(B, L, dim):
    s = _system(B, L, dim)
    try:
        for k in range(2):
            n, eps, phi, _ = s.state(k)
            site = phi.size // 3 + k
            old = eps.copy()
            old[site] = np.float32(eps[site] + 1.0)
            c0 = _change(B, s, k, n, old, phi)
            assert 0.9 < c0 < 1.1
            for step in (2.0 ** -38, 2.0 ** -47):
                moved = phi.copy()
                moved[site] += step
                c1 = _change(B, s, k, n, old, moved)
                assert abs((c0 - c1) - (moved[site] - phi[site])) <= 2.0 ** -49
    finally:
        s.close()


@pytest.mark.parametrize("L,dim", [(24, 2), (48, 2), (96, 2), (6, 3), (24, 3)])
def test_change_follows_nu_below_binary32(B, L, dim):
    # a third of the sites: nu is no binary32 number, and nu N an integer to 1e-10
    N = L ** dim
    step = 2.0 ** -(34 + int(np.log2(N)))
    out = []
    for nu in (1 / 3, 1 / 3 + step):
        assert np.float32(nu) == np.float32(1 / 3)
        s = _system(B, L, dim, nu=nu)
        try:
            n, eps, phi, _ = s.state(0)
            if not out:
                n0, phi0 = n, phi
                old = eps.copy()
                old[N // 3] = np.float32(eps[N // 3] + 1.0)
            out.append((nu, _change(B, s, 0, n0, old, phi0)))
        finally:
            s.close()
    f = np.minimum(np.arange(L), L - np.arange(L)).astype(np.float64)
    r2 = f[:, None] ** 2 + f[None, :] ** 2
    if dim == 3:
        r2 = f[:, None, None] ** 2 + r2[None]
    C0 = np.sum(1.0 / np.sqrt(r2[r2 > 0]))
    (nu0, c0), (nu1, c1) = out
    # eps = phi + sum (n - nu) / r falls, and the change from above grows, by (nu1 - nu0) C0
    assert abs((c1 - c0) - (nu1 - nu0) * C0) <= 2.0 ** -49


@pytest.mark.parametrize("L,dim", [(8, 2), (16, 2), (16, 3)])
def test_values_outside_the_split(B, L, dim):
    s = _system(B, L, dim)
    try:
        n, eps, phi, _ = s.state(0)
        B.cg_refresh(s.h)
        base = s.state(0)[1]
        for value in (0.0, -0.0, 1e-30, -3e-26, 1e25, -1e30, 1e200, np.inf, -np.inf, np.nan):
            p = phi.copy()
            p[7] = value
            B.cg_write_state(s.h, 0, n, eps=eps, phi=p)
            B.cg_refresh(s.h)
            got = s.state(0)[1].astype(np.float32)
            # the transform's part of site 7, known to binary32
            v = float(base[7]) - phi[7]
            with np.errstate(over="ignore"):
                want = np.float32(value + v)
            if abs(value) < 1e-20:
                assert abs(float(got[7]) - v) <= 2.0 ** -22
            else:
                np.testing.assert_array_equal(got[7], want)
            np.testing.assert_array_equal(np.delete(got, 7), np.delete(base.astype(np.float32), 7))
            c = s.observables(0)["max_eps_err_last_refresh"]
            if np.isnan(value):
                assert c < 1e-4
            elif abs(value) >= 1e25:
                assert c == abs(value)         # eps and the transform's part are lost in it
        # an energy from before that is no number is not counted, an infinite one is
        for value, inf in ((np.nan, False), (np.inf, True)):
            old = eps.copy()
            old[7] = value
            B.cg_write_state(s.h, 0, n, eps=old, phi=phi)
            B.cg_refresh(s.h)
            np.testing.assert_array_equal(s.state(0)[1], base)
            assert np.isinf(s.observables(0)["max_eps_err_last_refresh"]) == inf
    finally:
        s.close()
