"""The filter's vote over a warp where lanes have no point of their own: a last warp of one point or of one less than a
warp, warps inside, across and outside a ball domain, warps whose discs are whole beside others that are cut.
FP64 sums of at most a few hundred weights in [0, 1]: 1e-12."""
from __future__ import annotations

import pytest

from tests import test_gpu_design_chain as chain

pytestmark = pytest.mark.gpu

CASES = [("last-warp-one-point", 2, 33, dict(filter_radius=1.0)), ("last-warp-short", 2, 31, dict(filter_radius=2.0, proj_beta=2.0)),
         ("whole-and-cut", 2, 129, dict(filter_radius=3.0)), ("ball", 2, 97, dict(filter_radius=2.0, design_radius=20.3)),
         ("small-ball", 2, 65, dict(filter_radius=1.5, design_radius=1.2)),
         ("3d-ball", 3, 13, dict(filter_radius=2.0, design_radius=3.1)), ("3d-ragged", 3, 7, dict(filter_radius=1.8))]


@pytest.mark.parametrize("name,dim,nd,kw", CASES, ids=[c[0] for c in CASES])
def test_votes_of_ragged_warps(name, dim, nd, kw):
    chain.test_constraint_and_gradient(name, dim, nd, kw)
