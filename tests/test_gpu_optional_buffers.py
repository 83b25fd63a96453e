"""The buffers that a handle can do without (the coupling sums' flagged words, the reverse's linear maps)
never take the room of a call that needs its own: with a budget that holds the paper's adjoint but
not both, it still runs after the exact one, its gradient is the same, and the next gradient runs on
the other forms. FP64: the forms sum the same terms in another order (1e-11, as between the forms)."""
from __future__ import annotations

import numpy as np
import pytest

from tests.problems import body2d, body3d, perturbed_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("problem", [body2d(nx=120, ny=96, nd=3, centre=(50.3, 48.2), nt=4),
                                     body3d(nx=40, ny=32, nz=32, nd=3, centre=(18.3, 16.2, 15.9), nt=3)],
                         ids=["2d", "3d"])
def test_paper_adjoint_after_the_exact_one_within_a_tight_budget(problem):
    import torch
    from paper_2601_18272_gb300 import lks
    from paper_2601_18272_gb300.lks import Solver
    P, g = problem
    state = perturbed_state(P)
    gam = torch.tensor(g, dtype=torch.float64, device="cuda")

    def sweeps(mode, budget):
        S = Solver(P, precision=64, ckpt_policy=0, hbm_budget_bytes=budget)
        try:
            lks.lks_persistent_coupling(S.handle, mode)
            S.set_initial_state(*state)
            out = []
            for adjoint in (S.adjoint, S.adjoint_alks, S.adjoint):
                out.append(np.array([S.forward(gam)]))
                adjoint(1.0)
                d = torch.empty_like(gam)
                S.sensitivity(d)
                out.append(d.cpu().numpy())
            return out, lks.lks_workspace_bytes(S.handle)
        finally:
            S.close()

    ref, need = sweeps(0, 0)  # no optional buffers: what the three calls cannot do without
    free, used = sweeps(2, 0)
    assert used > need
    tight, held = sweeps(2, need)
    assert held <= need
    for a, b, c in zip(ref, free, tight):
        for x in (b, c):
            np.testing.assert_allclose(x, a, rtol=0, atol=1e-11 * np.abs(a).max())
