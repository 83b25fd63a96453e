"""The tiled 2D predictor and transpose (small grids) against the oracle, where a tile can go wrong:
grids smaller than a tile, a last tile of one column or row, both tile shapes, every boundary kind; and
the strip form (large grids) against the tiled one on a problem whose disturbance does not reach the
edges of either grid, so that the results are the same up to rounding."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from tests.problems import BC_INFLOW_OUTFLOW, BC_PERIODIC, BC_PRESSURE, BC_WALL, body2d, perturbed_state

pytestmark = pytest.mark.gpu

PER, IO, PR, WA = BC_PERIODIC, BC_INFLOW_OUTFLOW, BC_PRESSURE, BC_WALL
GRIDS = [(17, 16, PER, PER), (25, 17, IO, PER), (33, 25, PR, WA), (24, 41, IO, WA), (31, 23, PER, WA), (40, 33, PR, PER),
         (257, 161, IO, WA), (225, 193, PR, WA), (256, 177, PER, PER)]


def _gradient(P, g, state, precision):
    import torch
    from paper_2601_18272_gb300.lks import Solver
    S = Solver(P, precision=precision, ckpt_policy=0)
    try:
        if state:
            S.set_initial_state(*state)
        gam = torch.tensor(g, dtype=torch.float64, device="cuda")
        J = S.forward(gam)
        p, u = S.state()
        S.adjoint(1.0)
        d = S.sensitivity(torch.empty_like(gam)).cpu().numpy()
        return J, d, S.dof_history(), p, u, *S.initial_adjoint()
    finally:
        S.close()


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("nx,ny,bx,by", GRIDS, ids=[f"{c[0]}x{c[1]}-{c[2]}{c[3]}" for c in GRIDS])
def test_tiles_match_oracle(nx, ny, bx, by):
    P, g = body2d(nx=nx, ny=ny, nd=4, centre=(nx / 2 + 0.2, ny / 2 - 0.3), nt=3, n_itr=2, bc=(bx, by, PER))
    P = P.replace(dp=1e-3 if bx == PR else 0.0)
    state = perturbed_state(P)
    ref = O.gradient(P, g, *state)
    po, uo, _, _ = O.forward(P, g, *state)
    _, d, _, p, u, lp, lu, _ = _gradient(P, g, state, 64)
    for a, b in ((d, ref["dJdgamma"]), (p, po), (u, uo)):
        assert _rel(a, np.asarray(b)) < 1e-11  # FP64 rounding over three steps
    _, d32, _, p32, u32, lp32, lu32, _ = _gradient(P, g, state, 32)
    for a, b in ((d32, d), (p32, p), (u32, u), (lp32, lp), (lu32, lu)):
        assert _rel(a, b) < 2e-4


def test_strips_match_tiles():
    kw = dict(nd=10, nt=5, n_itr=3, bc=(PER, PER, PER))
    P, g = body2d(nx=96, ny=80, centre=(48.3, 40.2), **kw)
    Q, _ = body2d(nx=3702, ny=2001, centre=(1848.3, 1000.2), **kw)  # strips of 14 rows
    a, b = _gradient(P, g, None, 32), _gradient(Q, g, None, 32)
    assert _rel(b[1], a[1]) < 2e-4
    np.testing.assert_allclose(b[2][:, 3:], a[2][:, 3:], rtol=0, atol=2e-5 * np.abs(a[2][:, 3:]).max())
    win = lambda f, n: f.reshape(-1, n[1], n[0])  # noqa: E731
    for q in (4, 6):  # u, dJ/du0 around the body
        x, y = win(a[q], (96, 80)), win(b[q], (3702, 2001))[:, 960:1040, 1800:1896]
        assert np.abs(y - x).max() < 2e-4 * np.abs(x).max()
