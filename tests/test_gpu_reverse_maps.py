"""The reverse of the coupling iterations by linear maps (the default for bodies about one rotation
axis) against the per-iteration kernels (lks_persistent_coupling mode 0) and the oracle.

Cases cover what its sums and windows depend on: both weight kernels, every axis in 3D, masked
degrees of freedom with a rotated and turning body, support edges on nodes, a body across the periodic
boundary, ball-shaped and non-square design domains, one iteration, odd box sizes, chunks of steps that
do not divide the segment, binomial single steps. FP64: the two forms differ by the order of the
same sums, at most a few hundred terms of 1e-16 each (1e-11 leaves the cancellation of opposing
forces); the oracle is held to the 1e-9 of the other parity tests. FP32: single precision sums, 2e-5.
"""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from tests.problems import (BC_PERIODIC, BC_PRESSURE, BC_WALL, DOF_ROT, DOF_TX, DOF_TY, DOF_TZ, W_BILINEAR, body2d,
                            body3d, perturbed_state)
from workloads import CKPT_BINOMIAL, CKPT_STORE_ALL, CKPT_UNIFORM

pytestmark = pytest.mark.gpu


def _turned(P, theta, **kw):
    p0, u0, s0 = perturbed_state(P, **kw)
    s0[6] = theta
    return p0, u0, s0


def _cases():
    yield "2d", body2d(nt=7), dict(), 0.4
    yield "2d-bilinear", body2d(nt=5, wk=W_BILINEAR), dict(), -1.1
    yield "2d-edges-on-nodes", body2d(nd=5, centre=(10.0, 8.0), nt=3, wk=W_BILINEAR), dict(ug=0.0, omega=0.0), 0.0
    yield "2d-translation-turned", body2d(nt=4, mask=DOF_TX), dict(), 0.7
    yield "2d-fixed", body2d(nt=3, mask=0), dict(), 0.2
    yield "2d-one-iteration", body2d(nt=4, n_itr=1), dict(), 2.5
    yield "2d-wrapped", body2d(nx=26, ny=21, centre=(11.3, 1.2), nt=4, n_itr=6,
                               bc=(BC_PERIODIC, BC_PERIODIC, BC_PERIODIC)), dict(), 0.3
    yield "2d-channel", body2d(nx=29, ny=27, nd=9, centre=(13.4, 13.1), nt=5,
                               bc=(BC_PRESSURE, BC_WALL, BC_PERIODIC)), dict(), 0.9
    P, g = body2d(nx=40, ny=36, nd=13, centre=(18.2, 17.6), nt=3)
    yield "2d-ball", (P.replace(design_radius=5.5), g), dict(), 0.6
    for ax in (0, 1, 2):
        yield f"3d-axis{ax}", body3d(nx=24, ny=18, nz=19, nd=5, centre=(10.3, 8.6, 8.2), rot_axis=ax, nt=3), dict(), 0.5
    yield "3d-translation", body3d(nx=18, ny=14, nz=13, centre=(8.3, 6.2, 5.9), nt=4,
                                   mask=DOF_TX | DOF_TY | DOF_TZ), dict(omega=0.0), 0.0
    P, g = body3d(nx=24, ny=20, nz=20, nd=7, centre=(10.0, 9.5, 9.0), rot_axis=2, nt=2, mask=DOF_TZ | DOF_ROT)
    yield "3d-ball", (P.replace(design_radius=3.0), g), dict(), -0.8


CASES = list(_cases())


def _sweep(P, g, state, precision, mode, **ckpt):
    import torch
    from paper_2601_18272_gb300 import lks
    from paper_2601_18272_gb300.lks import Solver
    S = Solver(P, precision=precision, **ckpt)
    try:
        lks.lks_persistent_coupling(S.handle, mode)
        S.set_initial_state(*state)
        gam = torch.tensor(g, dtype=torch.float64, device="cuda")
        J = S.forward(gam)
        S.adjoint(1.0)
        d = S.sensitivity(torch.empty_like(gam))
        torch.cuda.synchronize()
        lp, lu, ls = S.initial_adjoint()
        return J, [d.cpu().numpy(), lp, lu, ls]
    finally:
        S.close()


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("name,problem,pert,theta", CASES, ids=[c[0] for c in CASES])
def test_linear_maps_match_per_iteration_kernels_and_oracle(name, problem, pert, theta):
    P, g = problem
    state = _turned(P, theta, **pert)
    J2, new = _sweep(P, g, state, 64, 2, ckpt_policy=CKPT_STORE_ALL)
    J0, old = _sweep(P, g, state, 64, 0, ckpt_policy=CKPT_STORE_ALL)
    assert abs(J2 - J0) <= 1e-12 * max(abs(J0), 1e-3)
    for a, b in zip(new, old):
        assert _rel(a, b) < 1e-11
    ref = O.gradient(P, g, *state)
    assert _rel(new[0], ref["dJdgamma"]) < 1e-9
    _, new32 = _sweep(P, g, state, 32, 2, ckpt_policy=CKPT_UNIFORM, ckpt_every=3)
    for a, b in zip(new32, new):
        assert _rel(a, b) < 2e-4
    _, old32 = _sweep(P, g, state, 32, 0, ckpt_policy=CKPT_UNIFORM, ckpt_every=3)
    for a, b, x in zip(new32, old32, new):
        assert _rel(a, x) <= 2.0 * _rel(b, x) + 2e-5


@pytest.mark.parametrize("ckpt", [dict(ckpt_policy=CKPT_STORE_ALL), dict(ckpt_policy=CKPT_UNIFORM, ckpt_every=70),
                                  dict(ckpt_policy=CKPT_BINOMIAL, ckpt_every=3)], ids=["all", "uniform", "binomial"])
def test_chunks_of_steps(ckpt):
    """Segments longer than the slabs of one chunk (64 steps), with a remainder, and single steps."""
    P, g = body2d(nx=30, ny=24, nt=141, centre=(10.3, 12.2), n_itr=2)
    state = _turned(P, 0.3, ug=0.001, omega=0.001)
    _, new = _sweep(P, g, state, 64, 2, **ckpt)
    _, old = _sweep(P, g, state, 64, 0, **ckpt)
    for a, b in zip(new, old):
        assert _rel(a, b) < 1e-11
