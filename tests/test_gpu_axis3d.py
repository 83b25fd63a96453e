"""The 3D body kernels that treat columns of cells along the rotation axis together (the default about
one axis) against the per-iteration kernels (lks_persistent_coupling mode 0): DOF history, final state,
gradient and initial adjoint for each axis, odd box and design sizes (remainders of 8 planes, of 4, of
32 in-plane positions), both weight kernels, ball domains, a body across periodic boundaries, support
edges on nodes, one iteration, masked rotation with a turned body, more units than warps. The two forms
sum the same terms in another order: FP64 1e-11; FP32 over a few steps 2e-4 against FP64 and no more
than twice the per-iteration kernels' error."""
from __future__ import annotations

import numpy as np
import pytest

from tests.problems import (BC_INFLOW_OUTFLOW, BC_PERIODIC, BC_WALL, DOF_TX, DOF_TY, DOF_TZ, W_BILINEAR,
                            perturbed_state)
from tests.problems import body3d as _body3d
from workloads import CKPT_STORE_ALL, CKPT_UNIFORM, mass_properties

pytestmark = pytest.mark.gpu
PER = (BC_PERIODIC,) * 3


def body3d(nd, rot_axis, **kw):  # with the mass and inertia of its design, so that the coupling is stable
    P, g = _body3d(nd=nd, rot_axis=rot_axis, **kw)
    M, inertia = mass_properties(g, (nd,) * 3, 3, rot_axis)
    return P.replace(mass=M, inertia=inertia), g


def _cases():
    for ax in (0, 1, 2):
        yield f"axis{ax}", body3d(nx=31, ny=29, nz=27, nd=9, centre=(14.3, 13.6, 12.2), rot_axis=ax, nt=3), 0.5, 0.003, 0.0
    yield "bilinear", body3d(nx=25, ny=24, nz=23, nd=6, centre=(11.3, 11.6, 10.2), rot_axis=2, nt=3, wk=W_BILINEAR), 0.9, 0.002, 0.0
    yield "edges-on-nodes", body3d(nx=22, ny=20, nz=21, nd=5, centre=(10.0, 9.0, 10.0), rot_axis=1, nt=2, wk=W_BILINEAR,
                                   mask=DOF_TX | DOF_TZ), 0.0, 0.0, 0.0
    yield "translation", body3d(nx=23, ny=20, nz=19, nd=7, centre=(10.3, 9.2, 8.9), rot_axis=2, nt=4,
                                mask=DOF_TX | DOF_TY | DOF_TZ), 0.0, 0.0, 0.0
    yield "turned-masked", body3d(nx=24, ny=24, nz=19, nd=6, centre=(11.0, 11.5, 8.7), rot_axis=2, nt=3, n_itr=1,
                                  mask=DOF_TX), 0.785398, 0.004, 0.0
    yield "wrapped", body3d(nx=25, ny=22, nz=23, nd=6, centre=(0.7, 21.2, 22.6), rot_axis=0, nt=3, n_itr=4, bc=PER), 1.9, 0.003, 0.0
    yield "walls", body3d(nx=28, ny=30, nz=28, nd=8, centre=(13.3, 14.2, 13.1), rot_axis=2, nt=3,
                          bc=(BC_INFLOW_OUTFLOW, BC_WALL, BC_WALL)), 0.3, 0.002, 0.0
    yield "ball", body3d(nx=28, ny=27, nz=26, nd=11, centre=(12.6, 12.2, 12.9), rot_axis=1, nt=2), 0.4, 0.002, 4.0
    yield "large", body3d(nx=84, ny=79, nz=66, nd=41, centre=(40.3, 39.1, 32.6), rot_axis=2, nt=2, n_itr=2), 0.6, 1e-4, 0.0
    yield "large-axis0", body3d(nx=66, ny=84, nz=79, nd=39, centre=(32.6, 40.3, 39.1), rot_axis=0, nt=2, n_itr=2), 0.6, 1e-4, 0.0
    yield "large-ball", body3d(nx=84, ny=66, nz=79, nd=41, centre=(40.3, 32.6, 39.1), rot_axis=1, nt=2, n_itr=2), 0.6, 1e-4, 17.2


CASES = list(_cases())


def _run(P, g, state, precision, mode, **ckpt):
    import torch
    from paper_2601_18272_gb300 import lks
    from paper_2601_18272_gb300.lks import Solver
    S = Solver(P, precision=precision, **ckpt)
    try:
        lks.lks_persistent_coupling(S.handle, mode)
        S.set_initial_state(*state)
        gam = torch.tensor(g, dtype=torch.float64, device="cuda")
        J = S.forward(gam)
        assert S.forward(gam) == J
        out = [S.dof_history(), *S.state()]
        S.adjoint(1.0)
        out += [S.sensitivity(torch.empty_like(gam)).cpu().numpy(), *S.initial_adjoint()]
        return out
    finally:
        S.close()


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("name,problem,theta,omega,radius", CASES, ids=[c[0] for c in CASES])
def test_axis_columns_match_per_iteration_kernels(name, problem, theta, omega, radius):
    P, g = problem
    P = P.replace(design_radius=radius)
    state = perturbed_state(P, ug=0.002, omega=omega)
    state[2][6] = theta
    new = _run(P, g, state, 64, 2, ckpt_policy=CKPT_STORE_ALL)
    old = _run(P, g, state, 64, 0, ckpt_policy=CKPT_STORE_ALL)
    for a, b in zip(new, old):
        assert _rel(a, b) < 1e-11
    new32 = _run(P, g, state, 32, 2, ckpt_policy=CKPT_UNIFORM, ckpt_every=2)
    old32 = _run(P, g, state, 32, 0, ckpt_policy=CKPT_UNIFORM, ckpt_every=2)
    for a, b, x in zip(new32, old32, new):
        assert _rel(a, x) < 2e-4
        assert _rel(a, x) <= 2.0 * _rel(b, x) + 2e-5
