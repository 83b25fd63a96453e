"""lks_support_sets reports the gather of the coupling form that runs: the index sets of
test_gpu_index_sets.py for the per-iteration kernels (mode 0), for the column form (3D boxes above its size
limit, every axis, both weight kernels, a ball domain, periodic boundaries) and for FP32 handles (2D with one and
with two lanes per cell, 3D) at positions whose support edges lie further from every node than FP32 rounding,
all against the oracle as integers. Where edges lie on nodes only up to rounding (Pythagorean rotations), FP32
sets differ between the forms: the 2D default's are compared with its own test, restated in numpy."""
from __future__ import annotations

import math

import numpy as np
import pytest

from oracle import oracle as O
from tests.problems import BC_INFLOW_OUTFLOW, BC_PERIODIC, BC_WALL, W_BILINEAR, body2d, body3d, perturbed_state
from tests.test_gpu_index_sets import _box_to_grid
from tests.test_oracle_index_sets import _cases as _small_cases

pytestmark = pytest.mark.gpu
PER = (BC_PERIODIC,) * 3


def _state(P, theta):
    _, _, s = perturbed_state(P)
    s[6] = theta
    return s


def _large():
    """3D boxes of more than 10,000 (FP64) cells; the first three also above 40,000 (FP32)."""
    for ax in (0, 1, 2):
        P, _ = body3d(nx=64, ny=50, nz=52, nd=27, centre=(29.3, 24.2, 25.9), rot_axis=ax)
        yield f"3d-axis{ax}", P, 0.41 + ax
    P, _ = body3d(nx=48, ny=36, nz=38, nd=17, centre=(22.3, 18.2, 18.9), rot_axis=1, wk=W_BILINEAR)
    yield "3d-bilinear", P, -0.7
    P, _ = body3d(nx=48, ny=36, nz=38, nd=17, centre=(1.3, 35.2, 0.9), rot_axis=2, bc=PER)
    yield "3d-wrapped", P, 1.3
    P, _ = body3d(nx=48, ny=46, nz=48, nd=17, centre=(22.0, 23.0, 24.0), rot_axis=0, bc=(BC_INFLOW_OUTFLOW, BC_WALL, BC_WALL))
    yield "3d-edges-on-nodes", P, 0.0
    P, _ = body3d(nx=64, ny=50, nz=52, nd=31, centre=(29.3, 24.2, 25.9), rot_axis=1)
    yield "3d-ball", P.replace(design_radius=12.4), 0.9


CASES = [(n, P, s, 64) for n, P, s in _small_cases()] + [(n, P, _state(P, th), 64) for n, P, th in _large()]
for _n, _P, _th in list(_large())[:3]:
    CASES.append((_n + "-32", _P, _state(_P, _th), 32))
for _n, _kw, _th in (("2d-two-lanes-32", dict(nx=60, ny=40, nd=15, centre=(25.3, 20.2)), 0.8),
                     ("2d-bilinear-32", dict(nx=60, ny=40, nd=15, centre=(25.3, 20.2), wk=W_BILINEAR), -2.1),
                     ("2d-one-lane-32", dict(nx=420, ny=320, nd=201, centre=(205.3, 160.3)),
                      math.atan2(4, 3))):  # coordinates are multiples of 0.2 off 0.3
    _P, _ = body2d(**_kw)
    CASES.append((_n, _P, _state(_P, _th), 32))


def _edge_distance(P, s):
    """Least distance of a design point's world coordinate to one where its set of nodes changes."""
    a = P.rot_axis
    b, c = (a + 1) % 3, (a + 2) % 3
    nd = (P.ndx, P.ndy, P.ndz)
    r = [np.arange(nd[e]) - (nd[e] - 1) / 2.0 for e in range(3)]
    x = {b: s[b] + math.cos(s[6]) * r[b][:, None] - math.sin(s[6]) * r[c][None, :],
         c: s[c] + math.sin(s[6]) * r[b][:, None] + math.cos(s[6]) * r[c][None, :]}
    if P.dim == 3:
        x[a] = s[a] + r[a]
    return min(np.abs(v - np.rint(v)).min() for v in x.values())


def _sets(P, s, precision, mode):
    from paper_2601_18272_gb300 import lks
    from paper_2601_18272_gb300.lks import Solver
    S = Solver(P, precision=precision, ckpt_policy=0)
    try:
        lks.lks_persistent_coupling(S.handle, mode)
        return lks.lks_support_sets(S.handle, s)
    finally:
        S.close()


@pytest.mark.parametrize("mode", [0, 2], ids=["launches", "auto"])
@pytest.mark.parametrize("name,P,s,precision", CASES, ids=[c[0] for c in CASES])
def test_index_sets_of_each_form(name, P, s, precision, mode):
    # offsets of up to 285 (27 in 3D) in FP32, each with a few roundings of 2^-24 of that
    assert precision == 64 or _edge_distance(P, s) > (1e-3 if P.ndx > 100 else 3e-5)
    lo, B, gpu = _sets(P, s, precision, mode)
    ref = O.support_sets(P, s)
    node = _box_to_grid(P, lo, B)
    inside = node >= 0
    assert np.array_equal(gpu[inside], ref[node[inside]])
    assert np.all(gpu[~inside, 0] == 0) and ref[:, 0].sum() > 0


def _fma(a, b, c):
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(np.float32)


@pytest.mark.parametrize("p,q,nd,centre", [(5, 12, 9, (25.0, 20.0)), (3, 4, 15, (25.2, 20.4)), (4, 3, 15, (25.0, 20.0)),
                                           (4, 3, 16, (25.5, 20.0))])
def test_sets_at_ties_are_those_of_the_2d_default(p, q, nd, centre):
    f = np.float32
    P, _ = body2d(nx=60, ny=40, nd=nd, centre=centre, bc=PER)
    s = _state(P, math.atan2(q, p))
    lo, B, gpu = _sets(P, s, 32, 2)
    cs, sn, xic = f(math.cos(s[6])), f(math.sin(s[6])), f((nd - 1) / 2)
    xi = np.floor(s[:2])
    xf = (s[:2] - xi).astype(f)
    jy, jx = np.mgrid[0:B[1], 0:B[0]]
    dx = (lo[0] + jx - xi[0]).astype(f) - xf[0]
    dy = (lo[1] + jy - xi[1]).astype(f) - xf[1]
    ix, iy = np.arange(nd, dtype=f)[:, None], np.arange(nd, dtype=f)[None, :]
    ex = ix - (_fma(cs, dx, sn * dy) + xic)[..., None, None]
    ey = iy - (_fma(cs, dy, -sn * dx) + xic)[..., None, None]
    ex, ey = np.broadcast_arrays(ex, ey)
    w = f(1.57079632679)  # offsets are compared as the cosines' arguments
    cw, nw = w * cs, w * sn
    ok = (np.abs(_fma(cw, ex, -nw * ey)) < f(3.14159265359)) & (np.abs(_fma(nw, ex, cw * ey)) < f(3.14159265359))
    m = (np.arange(nd)[:, None] + nd * np.arange(nd)[None, :]) * np.ones(ok.shape, dtype=np.int64)
    ref = np.stack([ok.sum((2, 3)), np.where(ok, m, nd * nd).min((2, 3)), np.where(ok, m, -1).max((2, 3)),
                    (m * ok).sum((2, 3)), (m * m * ok).sum((2, 3))], -1).reshape(-1, 5)
    ref[ref[:, 0] == 0, 1] = -1
    assert np.array_equal(gpu, ref)
