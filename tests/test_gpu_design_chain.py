"""The design chain's kernels at the edges of their branches against the oracle: radii below one, with
diagonal neighbours (R^2 not a square), a radius whose weight table does not fit and is computed per
pair, ball domains, 3D, odd sizes that leave partial blocks, more points than one pass of the volume's
cluster. FP64 sums of at most a few thousand weights in [0, 1]: 1e-12."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from tests.problems import body2d, body3d

pytestmark = pytest.mark.gpu

CASES = [("r0.7", 2, 11, dict(filter_radius=0.7)), ("r1.9", 2, 17, dict(filter_radius=1.9)),
         ("r3-exact", 2, 21, dict(filter_radius=3.0, proj_beta=4.0)), ("r4.5-cyclic", 2, 19, dict(filter_radius=4.5, cyclic_order=4)),
         ("r46-no-table", 2, 13, dict(filter_radius=46.0)), ("ball", 2, 23, dict(filter_radius=2.5, design_radius=8.2)),
         ("projection-only", 2, 9, dict(proj_beta=8.0)), ("cyclic-only", 2, 10, dict(cyclic_order=2)),
         ("one-point", 2, 1, dict(filter_radius=2.0)), ("large", 2, 190, dict(filter_radius=1.5)),
         ("3d", 3, 9, dict(filter_radius=2.3, proj_beta=3.0)), ("3d-ball", 3, 11, dict(filter_radius=1.8, design_radius=4.0))]


@pytest.mark.parametrize("name,dim,nd,kw", CASES, ids=[c[0] for c in CASES])
def test_constraint_and_gradient(name, dim, nd, kw):
    import torch
    from paper_2601_18272_gb300.lks import Solver
    n = 2 * nd + 24
    make = body2d if dim == 2 else body3d
    size = dict(nx=n, ny=n) if dim == 2 else dict(nx=n, ny=n, nz=n)
    P, g = make(nd=nd, centre=(n / 2.0,) * dim, nt=1, **size)
    P = P.replace(v_min=0.3, rot_axis=2, inertia=max(P.inertia, 1.0), **kw)
    Go, dGo = O.constraint(P, g)
    S = Solver(P, precision=64, ckpt_policy=0)
    try:
        gam = torch.tensor(g, dtype=torch.float64, device="cuda")
        dG = torch.full_like(gam, np.nan)
        G = S.constraint(gam, dG)
        assert S.constraint(gam) == G
    finally:
        S.close()
    assert abs(G - Go) <= 1e-12 * max(1.0, abs(Go))
    np.testing.assert_allclose(dG.cpu().numpy(), dGo, rtol=0, atol=1e-12 * np.abs(dGo).max())
