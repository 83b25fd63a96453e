"""Memory of the reverse by linear maps: one set of a step's planes (10 N_itr + 19 values per box cell in 3D) where a
segment has one chunk (binomial schedules, segments of one step), two where chunks follow one another, and
never more than 16 GiB, beyond which the per-iteration kernels run. A budget that holds one set lets a
binomial sweep take the maps. The gradient does not depend on it: FP64 1e-11, as between the forms."""
from __future__ import annotations

import numpy as np
import pytest

from tests.problems import perturbed_state
from tests.test_gpu_axis3d import _rel, body3d
from workloads import CKPT_BINOMIAL, CKPT_UNIFORM

pytestmark = pytest.mark.gpu


def _grown(P, g, precision, state=None, **ckpt):
    """Workspace taken by the first adjoint, box cells, gradient."""
    import torch
    from paper_2601_18272_gb300 import lks
    from paper_2601_18272_gb300.lks import Solver
    S = Solver(P, precision=precision, **ckpt)
    try:
        if state is not None:
            S.set_initial_state(*state)
        gam = torch.tensor(g, dtype=torch.float64, device="cuda")
        S.forward(gam)
        before = lks.lks_workspace_bytes(S.handle)
        S.adjoint(1.0)
        d = S.sensitivity(torch.empty_like(gam)).cpu().numpy()
        box = lks.lks_support_sets(S.handle, S.dof_history()[0])[1] if P.ndx < 100 else None
        return lks.lks_workspace_bytes(S.handle) - before, box, d, before
    finally:
        S.close()


def test_one_set_where_no_chunk_follows_another():
    P, g = body3d(nx=60, ny=48, nz=48, nd=21, centre=(25.3, 23.2, 23.9), rot_axis=2, nt=4)
    state = perturbed_state(P, ug=0.002, omega=1e-4)
    one, box, d1, held = _grown(P, g, 64, state, ckpt_policy=CKPT_BINOMIAL, ckpt_every=1)
    planes = (10 * P.n_itr + 19) * int(np.prod(box)) * 8
    assert planes < one < 1.3 * planes  # and per-block sums, matrices
    single, _, _, _ = _grown(P, g, 64, state, ckpt_policy=CKPT_UNIFORM, ckpt_every=1)
    assert single == one
    two, _, d2, _ = _grown(P, g, 64, state, ckpt_policy=CKPT_UNIFORM, ckpt_every=4)
    assert 2 * planes < two < 2.6 * planes
    tight, _, d3, _ = _grown(P, g, 64, state, ckpt_policy=CKPT_BINOMIAL, ckpt_every=1, hbm_budget_bytes=held + one)
    assert tight == one
    for d in (d2, d3):
        assert _rel(d, d1) < 1e-11


def test_maps_beyond_the_limit_are_not_taken():
    P, g = body3d(nx=224, ny=216, nz=160, nd=144, centre=(111.6, 107.8, 79.7), rot_axis=2, nt=1, n_itr=64)
    P = P.replace(mass=20.0 * P.mass, inertia=20.0 * P.inertia)
    grown, _, d, _ = _grown(P, g, 32, ckpt_policy=CKPT_BINOMIAL, ckpt_every=1)
    assert grown == 0  # 6.8 million box cells by 659 values: 18 GB
    assert np.isfinite(d).all() and np.abs(d).max() > 0
