"""GPU check that cg_workspace_bytes covers a batch whose replicas differ in
r_max and xi: hop tables are kept per (L, r_max, xi), the refresh's DFT(1/r)
and twiddles per (L, dimension).  The workspace passed is exactly the size
asked for, and the refresh of every replica gives its energies (2e-5, the
transform refresh's bound).
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("L,dim,R", [(112, 2, 9), (80, 2, 8), (64, 2, 3), (96, 2, 2), (16, 3, 3),
                                     (42, 2, 3)])
def test_workspace_of_several_hop_tables(B, L, dim, R):
    import torch
    reps = [dict(L=L, nu=0.5, W=1.0, xi=1.0 + 0.25 * (k % 3), r_max=3 + k % 2, T=0.05, E=0.0,
                 seed=k, replica=k, dim=dim) for k in range(R)]
    o = B.opts(precision=B.CG_FP32)
    nbytes = B.cg_workspace_bytes(reps, o)
    buf = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    base = (buf.data_ptr() + 255) & ~255
    h = B.cg_create_batch_ws(reps, o, base, nbytes)
    try:
        assert B.cg_run(h, 30, 512) == B.CG_OK
        B.cg_refresh(h)
        for k in range(R):
            n, eps, phi, _ = B.cg_read_state(h, k)
            exact = (ref.site_energies_fft3(n, phi, 0.5, L) if dim == 3
                     else ref.site_energies_fft(n, phi, 0.5, L))
            assert np.abs(eps - exact).max() <= 2e-5
    finally:
        B.cg_destroy(h)
