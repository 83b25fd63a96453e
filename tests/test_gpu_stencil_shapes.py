"""Shapes of 2D grids the other stencil tests leave out: grids narrower than the 32-column tile but with more cells than
the small tile takes, against the oracle with every boundary kind; and FP64 grids whose predictor runs on strips
while the transpose runs on tiles, against a small grid of tiles, on a problem whose disturbance does not
reach the edges of either (results the same up to rounding: 1e-11)."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from tests.problems import BC_INFLOW_OUTFLOW, BC_PERIODIC, BC_PRESSURE, BC_WALL, body2d, perturbed_state
from tests.test_gpu_stencil_tile import _gradient, _rel

pytestmark = pytest.mark.gpu

PER, IO, PR, WA = BC_PERIODIC, BC_INFLOW_OUTFLOW, BC_PRESSURE, BC_WALL


@pytest.mark.parametrize("nx,ny,bx,by", [(20, 2003, PER, PER), (26, 1600, IO, PER), (27, 1501, PR, WA), (2003, 20, PER, WA),
                                         (1501, 29, IO, WA)])
def test_narrow_grids(nx, ny, bx, by):
    P, g = body2d(nx=nx, ny=ny, nd=4, centre=(nx / 2 + 0.2, ny / 2 - 0.3), nt=2, n_itr=2, bc=(bx, by, PER))
    P = P.replace(dp=1e-3 if bx == PR else 0.0)
    state = perturbed_state(P)
    ref = O.gradient(P, g, *state)
    po, uo, _, _ = O.forward(P, g, *state)
    _, d, _, p, u, lp, lu, _ = _gradient(P, g, state, 64)
    for a, b in ((d, ref["dJdgamma"]), (p, po), (u, uo)):
        assert _rel(a, np.asarray(b)) < 1e-11  # FP64 rounding over two steps
    for a, b in zip(_gradient(P, g, state, 32)[3:7], (p, u, lp, lu)):
        assert _rel(a, b) < 2e-4


@pytest.mark.parametrize("nx,ny", [(3302, 1701), (4096, 2048)], ids=["strips-of-4", "strips-of-7"])
def test_fp64_strips_match_tiles(nx, ny):
    kw = dict(nd=10, nt=4, n_itr=2, bc=(PER, PER, PER))
    x0, y0 = nx // 2 - 48, ny // 2 - 40
    P, g = body2d(nx=96, ny=80, centre=(48.3, 40.2), **kw)
    Q, _ = body2d(nx=nx, ny=ny, centre=(x0 + 48.3, y0 + 40.2), **kw)
    a, b = _gradient(P, g, None, 64), _gradient(Q, g, None, 64)
    assert _rel(b[1], a[1]) < 1e-11
    for q in (3, 4, 5, 6):  # p, u, dJ/dp0, dJ/du0 around the body
        x = a[q].reshape(-1, 80, 96)
        y = b[q].reshape(-1, ny, nx)[:, y0:y0 + 80, x0:x0 + 96]
        assert np.abs(y - x).max() <= 1e-11 * np.abs(x).max()
