"""The 2D coupling iterations in one launch with flagged words (the default in 2D) against the
per-iteration kernels (lks_persistent_coupling mode 0): DOF history and final state, at box sizes
around the kernel's shapes (one CTA, partial warps, several cells per thread, FP64 and FP32), both
weight kernels, masked degrees of freedom, the closed form of large step rotations. The two forms sum
the same terms in another order: FP64 1e-12; FP32, over a few steps, 2e-5 of the largest value."""
from __future__ import annotations

import numpy as np
import pytest

from tests.problems import BC_PERIODIC, DOF_ROT, DOF_TX, DOF_TY, W_BILINEAR, body2d, perturbed_state

pytestmark = pytest.mark.gpu


def _cases():
    yield "one-point", body2d(nx=16, ny=14, nd=1, centre=(7.3, 6.8), nt=5, mass=5.0, inertia=5.0), 0.0, 0.003
    yield "small", body2d(nt=6), 0.4, 0.003
    yield "bilinear", body2d(nt=6, wk=W_BILINEAR, mask=DOF_TX), 0.0, 0.0
    yield "one-iteration", body2d(nt=5, n_itr=1), -0.9, 0.003
    yield "wrapped", body2d(nx=27, ny=22, nd=7, centre=(1.2, 20.7), nt=4, bc=(BC_PERIODIC,) * 3, n_itr=6), 1.3, 0.003
    yield "fast-spin", body2d(nx=30, ny=26, nd=7, centre=(12.2, 12.7), nt=4, mask=DOF_ROT, inertia=1e6), 0.1, 0.1
    yield "faster-spin", body2d(nx=30, ny=26, nd=7, centre=(12.2, 12.7), nt=4, mask=DOF_ROT, inertia=1e6), 0.1, -0.3
    yield "medium", body2d(nx=150, ny=131, nd=71, centre=(70.2, 65.1), nt=3, mask=DOF_TX | DOF_TY | DOF_ROT), 0.7, 1e-4
    yield "several-cells-per-thread", body2d(nx=460, ny=421, nd=270, centre=(212.2, 210.1), nt=2, n_itr=2), 0.5, 1e-5


CASES = list(_cases())


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("name,problem,theta,omega", CASES, ids=[c[0] for c in CASES])
def test_flag_exchange_matches_per_iteration_kernels(name, problem, theta, omega, precision):
    import torch
    from paper_2601_18272_gb300 import lks
    from paper_2601_18272_gb300.lks import Solver
    P, g = problem
    p0, u0, s0 = perturbed_state(P, ug=0.002, omega=omega)
    s0[6] = theta
    out = []
    for mode in (2, 0):
        S = Solver(P, precision=precision, ckpt_policy=0)
        try:
            lks.lks_persistent_coupling(S.handle, mode)
            S.set_initial_state(p0, u0, s0)
            J = S.forward(torch.tensor(g, dtype=torch.float64, device="cuda"))
            J2 = S.forward(torch.tensor(g, dtype=torch.float64, device="cuda"))
            assert J == J2  # a fixed order of summation
            out.append([S.dof_history(), *S.state()])
        finally:
            S.close()
    tol = 1e-12 if precision == 64 else 2e-5
    for a, b in zip(*out):
        np.testing.assert_allclose(a, b, rtol=0, atol=tol * np.abs(b).max())


def test_flag_exchange_timeout_is_reported():
    """With the test hook the first CTA publishes nothing: the waits run out after a second, the call
    returns LKS_ERR_TIMEOUT, and the next march gives the same result as before."""
    import torch
    from paper_2601_18272_gb300 import lks
    from paper_2601_18272_gb300.lks import LksError, Solver
    P, g = body2d(nt=3)
    S = Solver(P, precision=32, ckpt_policy=0)
    try:
        gam = torch.tensor(g, dtype=torch.float64, device="cuda")
        J = S.forward(gam)
        lks.lks_debug_sync_skip(S.handle, True)
        with pytest.raises(LksError, match="LKS_ERR_TIMEOUT"):
            S.forward(gam)
        lks.lks_debug_sync_skip(S.handle, False)
        assert S.forward(gam) == J
    finally:
        S.close()
