"""Leaf maps and solves of the plane elimination at its dispatch edges: one
leaf over four warps (up to 304 leaves), one leaf per warp (up to 1216), two
leaves per warp in CTAs of four warps (beyond; leaf counts that are no
multiple of eight), more than 16 segments; leaves of one plane, of one cell per
plane, of even and odd plane counts, with truncated leaves at both ends.

The maps against the oracle's dense local problem: both sides' errors are
below about (planes) x u x cond, 16 x 1.1e-16 x 1e3 = 2e-12 for these fields
(cond of a leaf below 1e3), so 1e-11 bounds their difference.  The solves are
refined on both sides: 1e-10 as in the other parity tests.
"""
import numpy as np
import pytest

import inputs
from conftest import gpu_solve, rel
from oracle.geometry import Decomposition
from oracle.local import LeafProblem
from oracle.mrcm import solve_mrcm

from test_gpu_parity import _oracle_seg_key

pytestmark = pytest.mark.gpu

# nx, ny, sub, seg
GRIDS = [(20, 23, (6, 9), (2, 3)),
         (33, 16, (16, 1), (4, 1)),       # one plane per leaf
         (16, 45, (1, 15), (1, 5)),       # one cell per plane
         (40, 34, (16, 16), (1, 1)),      # up to 64 segments
         (122, 83, (6, 4), (2, 2)),       # 441 leaves
         (124, 154, (3, 5), (1, 5)),      # 1302 leaves
         (560, 561, (16, 16), (4, 4)),    # 1260 leaves, the last row one plane each
         (499, 500, (5, 10), (5, 5))]     # 5000 leaves


def _problem(nx, ny, sub, seg):
    return inputs.darcy_problem(nx, ny, sigma2=1.0, corr=0.1, seed=nx + ny, bc="quarter_five_spot", sub=sub, seg=seg)


@pytest.mark.parametrize("nx,ny,sub,seg", GRIDS)
def test_leaf_maps_at_the_dispatch_edges(mrcm_lib, nx, ny, sub, seg):
    prob = _problem(nx, ny, sub, seg)
    solver = gpu_solve(prob, want_iface=False)["solver"]
    ctx = solver.ctx
    dec = Decomposition(prob)
    n = len(dec.leaves)
    for leaf in sorted({0, 1, n // 3, n // 2, n // 2 + 1, n - 2, n - 1}):
        lp = LeafProblem(dec, leaf)
        R_o, _ = lp.robin_to_flux()
        R_g = mrcm_lib.mrcm_node_operator(ctx, leaf)
        okey = {_oracle_seg_key(dec, t): k for k, t in enumerate(lp.segs)}
        perm = []
        for t in mrcm_lib.mrcm_node_segments(ctx, leaf):
            si = mrcm_lib.mrcm_segment_info(ctx, t)
            perm.append(okey[(si["axis"], si["line"], si["lo"])])
        assert rel(R_g, R_o[np.ix_(perm, perm)]) < 1e-11, leaf


@pytest.mark.parametrize("nx,ny,sub,seg", GRIDS[:-2])
def test_solves_at_the_dispatch_edges(mrcm_lib, nx, ny, sub, seg):
    prob = _problem(nx, ny, sub, seg)
    g, o = gpu_solve(prob, want_iface=False, refine=3), solve_mrcm(prob, refine=3)
    for key in ("p", "Fx", "Fy"):
        assert rel(g[key], o[key]) < 1e-10, key
