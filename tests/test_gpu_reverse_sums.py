"""Sums of the reverse by linear maps where a thread adds several cells before its block does (FP32 pairs):
boxes of more cells than k_rev_const has threads (2D 93,636; 3D 209,088) and the planes of the column form, with
remainders of four planes. FP32 against FP64 of the same form: terms rounded to 2^-24 and added without further loss, a few hundred of
them to each value (2e-5 leaves room for opposing forces); per-iteration kernels (mode 0) within twice that."""
from __future__ import annotations

import numpy as np
import pytest

from tests.problems import body2d, perturbed_state
from tests.test_gpu_axis3d import _rel, _run, body3d
from workloads import CKPT_STORE_ALL

pytestmark = pytest.mark.gpu

CASES = [("2d", body2d(nx=420, ny=320, nd=201, centre=(205.3, 160.2), nt=3, n_itr=2)),
         ("3d", body3d(nx=84, ny=79, nz=66, nd=41, centre=(40.3, 39.1, 32.6), rot_axis=2, nt=2, n_itr=2)),
         ("3d-remainder", body3d(nx=50, ny=44, nz=42, nd=22, centre=(22.3, 20.1, 20.6), rot_axis=0, nt=2, n_itr=3))]


@pytest.mark.parametrize("name,problem", CASES, ids=[c[0] for c in CASES])
def test_sums_of_several_cells_a_thread(name, problem):
    P, g = problem
    state = perturbed_state(P, ug=0.002, omega=1e-4)
    state[2][6] = 0.6
    ref = _run(P, g, state, 64, 2, ckpt_policy=CKPT_STORE_ALL)
    new = _run(P, g, state, 32, 2, ckpt_policy=CKPT_STORE_ALL)
    old = _run(P, g, state, 32, 0, ckpt_policy=CKPT_STORE_ALL)
    for a, b in zip(new[3:], ref[3:]):  # dJ/dgamma and the adjoint of the initial state
        assert _rel(a, b) < 2e-5
    for a, b in zip(new[3:], old[3:]):
        assert _rel(a, b) < 4e-5
    assert np.isfinite(new[3]).all()
