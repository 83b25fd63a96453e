"""The 3D column kernels themselves (coupling and recompute take them above 10,000 box cells in FP64, 40,000 in FP32;
the boxes here have 60,000 to 90,000) where they can go wrong: the bilinear window, a body across every
periodic boundary, also along the rotation axis, walls, one iteration, a masked turned body, support edges
on nodes, a solid body about each axis, ball domains. Against the per-iteration kernels (mode 0), as in
test_gpu_axis3d.py and with its bounds. The "couple" launches show that the one-launch form ran."""
from __future__ import annotations

import pytest

from tests.problems import (BC_INFLOW_OUTFLOW, BC_PERIODIC, BC_WALL, DOF_TX, DOF_TZ, W_BILINEAR, perturbed_state)
from tests.test_gpu_axis3d import _rel, _run, body3d
from workloads import CKPT_STORE_ALL, CKPT_UNIFORM

pytestmark = pytest.mark.gpu
PER, IO, WA = BC_PERIODIC, BC_INFLOW_OUTFLOW, BC_WALL


def _case(name, ax, theta, radius=0.0, n=(64, 51, 53), centre=(30.3, 25.2, 26.9), **kw):
    kw.setdefault("nd", 27)
    P, g = body3d(nx=n[0], ny=n[1], nz=n[2], centre=centre, rot_axis=ax, nt=2, **kw)
    return name, P.replace(design_radius=radius), g, theta


CASES = [_case(f"solid-axis{ax}", ax, 0.6) for ax in (0, 1, 2)]
CASES += [_case(f"bilinear-axis{ax}", ax, 0.9, wk=W_BILINEAR, nd=29) for ax in (0, 1, 2)]
CASES += [_case(f"wrapped-axis{ax}", ax, 1.9, bc=(PER,) * 3, centre=(0.7, 50.2, 52.6)) for ax in (0, 1, 2)]
CASES += [
    _case("walls", 2, 0.3, bc=(IO, WA, WA), n=(64, 61, 63), centre=(30.3, 30.2, 31.4)),
    _case("walls-along-axis", 1, 0.3, bc=(IO, WA, PER), n=(64, 46, 53), centre=(30.3, 22.8, 26.9)),
    _case("one-iteration", 0, 0.785398, n_itr=1),
    _case("turned-masked", 2, 0.785398, mask=DOF_TX | DOF_TZ),
    _case("edges-on-nodes", 1, 0.0, wk=W_BILINEAR, nd=29, centre=(30.0, 25.0, 27.0)),
    _case("edges-on-nodes-cosine", 2, 0.0, centre=(30.0, 25.0, 27.0)),
    _case("quarter-turn", 0, 1.5707963267948966, nd=28, centre=(30.5, 25.5, 26.5)),
    _case("ball", 1, 0.4, radius=17.3, nd=37, n=(64, 53, 53)),
    _case("small-ball", 2, -2.4, radius=16.0, nd=45, n=(64, 53, 53)),
    _case("many-iterations", 1, 0.2, n_itr=7),
]


@pytest.mark.parametrize("name,P,g,theta", CASES, ids=[c[0] for c in CASES])
def test_column_kernels_match_per_iteration_kernels(name, P, g, theta):
    edges = name.startswith(("edges", "quarter"))
    state = perturbed_state(P, ug=0.0 if edges else 0.002, omega=0.0 if edges else 2e-4)
    state[2][6] = theta
    new = _run(P, g, state, 64, 2, ckpt_policy=CKPT_STORE_ALL)
    old = _run(P, g, state, 64, 0, ckpt_policy=CKPT_STORE_ALL)
    for a, b in zip(new, old):
        assert _rel(a, b) < 1e-11
    new32 = _run(P, g, state, 32, 2, ckpt_policy=CKPT_UNIFORM, ckpt_every=1)
    old32 = _run(P, g, state, 32, 0, ckpt_policy=CKPT_UNIFORM, ckpt_every=1)
    for a, b, x in zip(new32, old32, new):
        assert _rel(a, x) < 2e-4
        assert _rel(a, x) <= 2.0 * _rel(b, x) + 2e-5


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("name", ["solid-axis1", "bilinear-axis0", "ball"])
def test_these_boxes_take_the_column_kernels(name, precision):
    import torch
    from paper_2601_18272_gb300 import lks
    from paper_2601_18272_gb300.lks import Solver
    _, P, g, _ = next(c for c in CASES if c[0] == name)
    S = Solver(P, precision=precision, ckpt_policy=CKPT_STORE_ALL)
    try:
        gam = torch.tensor(g, dtype=torch.float64, device="cuda")
        for mode, launches in ((2, P.n_steps), (0, P.n_steps * P.n_itr + 1)):
            lks.lks_persistent_coupling(S.handle, mode)
            lks.lks_set_kernel_timing(S.handle, True)
            S.forward(gam)
            n = lks.lks_kernel_time(S.handle, "couple")[1]
            assert n == launches if mode == 2 else n >= launches
    finally:
        S.close()
