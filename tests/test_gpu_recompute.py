"""A checkpointed march recomputes its steps to the bit: with native checkpoints the adjoint of the initial
state is the same, bit for bit, whether every state was stored or the steps are recomputed (uniform
checkpoints with a remainder, binomial snapshots), and dJ/dgamma differs only by the order in which the
steps' FP64 terms are added (1e-12 of its largest value). 2D in every lane count of the coupling's
gather (FP32 boxes of one and of several passes, FP64), both kernels, one iteration, across a periodic
boundary, ball domains; 3D above and below the box size of the column form. Also when the form changes between the forward and its
adjoint: another coupling mode, and the words given back to a call that needs its own buffers."""
from __future__ import annotations

import numpy as np
import pytest

from tests.problems import BC_PERIODIC, DOF_TX, W_BILINEAR, body2d, perturbed_state
from tests.test_gpu_axis3d import body3d
from workloads import CKPT_BINOMIAL, CKPT_STORE_ALL, CKPT_UNIFORM

pytestmark = pytest.mark.gpu
PER = (BC_PERIODIC,) * 3


def _cases():
    yield "2d-32", body2d(nx=60, ny=40, nd=15, centre=(25.3, 20.2), nt=8), 32
    yield "2d-32-bilinear", body2d(nx=61, ny=43, nd=15, centre=(25.3, 20.2), nt=8, wk=W_BILINEAR), 32
    yield "2d-32-one-iteration", body2d(nx=60, ny=40, nd=14, centre=(25.3, 20.2), nt=8, n_itr=1), 32
    yield "2d-32-wrapped", body2d(nx=60, ny=41, nd=14, centre=(25.3, 1.2), nt=8, bc=PER), 32
    yield "2d-32-masked", body2d(nx=60, ny=40, nd=14, centre=(25.3, 20.2), nt=8, mask=DOF_TX), 32
    yield "2d-32-one-lane", body2d(nx=420, ny=320, nd=201, centre=(205.3, 160.2), nt=5), 32  # 93,636 cells
    yield "2d-64", body2d(nx=60, ny=40, nd=15, centre=(25.3, 20.2), nt=8), 64
    yield "3d-32-small", body3d(nx=36, ny=30, nz=30, nd=9, centre=(15.3, 14.2, 13.9), rot_axis=1, nt=5), 32
    for ax in (0, 1, 2):  # boxes of 46 x 46 x 34 cells and 32 x 32 x 24
        yield f"3d-32-axis{ax}", body3d(nx=64, ny=50, nz=52, nd=27, centre=(29.3, 24.2, 25.9), rot_axis=ax, nt=5), 32
        yield f"3d-64-axis{ax}", body3d(nx=48, ny=36, nz=38, nd=17, centre=(22.3, 18.2, 18.9), rot_axis=ax, nt=5), 64
    P, g = body3d(nx=64, ny=50, nz=52, nd=31, centre=(29.3, 24.2, 25.9), rot_axis=2, nt=4)
    yield "3d-32-ball", (P.replace(design_radius=14.2), g), 32
    P, g = body2d(nx=60, ny=40, nd=20, centre=(25.3, 20.2), nt=8)
    yield "2d-32-ball", (P.replace(design_radius=8.2), g), 32


CASES = list(_cases())


def _sweep(P, g, precision, modes=(2, 2), alks=False, **ckpt):
    import torch
    from paper_2601_18272_gb300 import lks
    from paper_2601_18272_gb300.lks import Solver
    state = perturbed_state(P, ug=0.003, omega=2e-4)
    state[2][6] = 0.3
    S = Solver(P, precision=precision, **ckpt)
    try:
        lks.lks_persistent_coupling(S.handle, modes[0])
        S.set_initial_state(*state)
        gam = torch.tensor(g, dtype=torch.float64, device="cuda")
        S.forward(gam)
        lks.lks_persistent_coupling(S.handle, modes[1])
        held = lks.lks_workspace_bytes(S.handle)
        (S.adjoint_alks if alks else S.adjoint)(1.0)
        d = S.sensitivity(torch.empty_like(gam)).cpu().numpy()
        adj = S.alks_adjoint() if alks else S.initial_adjoint()
        return d, adj, held, lks.lks_workspace_bytes(S.handle)
    finally:
        S.close()


def _same(a, b):
    for x, y in zip(a[1], b[1]):
        assert np.array_equal(x, y)
    assert np.abs(a[0] - b[0]).max() <= 1e-12 * np.abs(a[0]).max()


@pytest.mark.parametrize("name,problem,precision", CASES, ids=[c[0] for c in CASES])
@pytest.mark.parametrize("modes", [(2, 2), (0, 0), (2, 0), (0, 2)], ids=["auto", "launches", "auto-then-launches", "launches-then-auto"])
def test_recomputed_steps_are_the_forward_s(name, problem, precision, modes):
    P, g = problem
    ref = _sweep(P, g, precision, modes, ckpt_policy=CKPT_STORE_ALL)
    _same(ref, _sweep(P, g, precision, modes, ckpt_policy=CKPT_UNIFORM, ckpt_every=3))
    _same(ref, _sweep(P, g, precision, modes, ckpt_policy=CKPT_BINOMIAL, ckpt_every=1))


@pytest.mark.parametrize("name", ["2d-32", "3d-32-axis2"])
def test_words_given_back_between_forward_and_adjoint(name):
    P, g = next(c[1] for c in CASES if c[0] == name)
    ckpt = dict(ckpt_policy=CKPT_UNIFORM, ckpt_every=3)
    need = _sweep(P, g, 32, (0, 0), True, **ckpt)[3]  # workspace of the paper's adjoint without the words
    ref = _sweep(P, g, 32, (2, 2), True, **ckpt)
    tight = _sweep(P, g, 32, (2, 2), True, hbm_budget_bytes=need, **ckpt)
    assert tight[2] == ref[2] and tight[3] == need  # the forward held them, the adjoint took their room
    _same(ref, tight)
