"""Ball-shaped design domains about one rotation axis whose radius is well below the half extent of the
design grid: the body box is sized to the ball, so a group of design points along the axis reaches past
the box where only some of its points belong to the domain. The gradient of the default kernels against
the per-iteration ones (lks_persistent_coupling mode 0) in both precisions, and against the oracle at the
smallest size. The forms sum the same terms in another order: FP64 1e-11, FP32 2e-4 against FP64 and no
more than twice the per-iteration kernels' error (the bounds of test_gpu_axis3d.py); every design point
of the domain whose FP64 sensitivity is not zero has one in FP32 too."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from tests.problems import body3d as _body3d
from tests.problems import perturbed_state
from tests.test_gpu_axis3d import _rel, _run
from workloads import CKPT_STORE_ALL, CKPT_UNIFORM, mass_properties

pytestmark = pytest.mark.gpu


def _cases():
    # nd, radius, fraction of x^G, rotation axis
    for nd, radius, frac in ((16, 5.0, 0.0), (16, 5.0, 0.6), (24, 7.0, 0.3), (27, 10.0, 0.1), (31, 10.0, 0.7)):
        for ax in (0, 1, 2):
            yield nd, radius, frac, ax
    yield 48, 20.0, 0.4, 2


CASES = list(_cases())


@pytest.mark.parametrize("nd,radius,frac,ax", CASES, ids=[f"{n}-r{r:g}-{f:g}-axis{a}" for n, r, f, a in CASES])
def test_small_ball_in_a_large_design_grid(nd, radius, frac, ax):
    n = 2 * int(radius) + 9
    P, g = _body3d(nx=n + 7, ny=n + 1, nz=n + 2, nd=nd, centre=(n // 2 + 3 + frac, n // 2 + frac, n // 2 + frac),
                   rot_axis=ax, nt=2, n_itr=2)
    M, inertia = mass_properties(g, (nd,) * 3, 3, ax)
    P = P.replace(mass=M, inertia=inertia, design_radius=radius)
    state = perturbed_state(P, ug=0.002, omega=0.001)
    state[2][6] = 0.4
    new = _run(P, g, state, 64, 2, ckpt_policy=CKPT_STORE_ALL)
    old = _run(P, g, state, 64, 0, ckpt_policy=CKPT_STORE_ALL)
    for a, b in zip(new, old):
        assert _rel(a, b) < 1e-11
    if nd == 16:
        assert _rel(new[3], O.gradient(P, g, *state)["dJdgamma"]) < 1e-9
    new32 = _run(P, g, state, 32, 2, ckpt_policy=CKPT_UNIFORM, ckpt_every=2)
    old32 = _run(P, g, state, 32, 0, ckpt_policy=CKPT_UNIFORM, ckpt_every=2)
    assert np.array_equal(new32[3] != 0.0, old32[3] != 0.0)
    for a, b, x in zip(new32, old32, new):
        assert _rel(a, x) < 2e-4
        assert _rel(a, x) <= 2.0 * _rel(b, x) + 2e-5
