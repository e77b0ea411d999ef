"""Leaves at the line between the two eliminations (cell by cell for small and
narrow leaves, plane by plane otherwise; chosen by shape, segments and number):
one or two grids on either side of each branch of the rule, truncated leaves
among them, with leaf counts that are no multiple of the leaves per CTA (4 or 2
cell by cell, 4 or 8 plane by plane), FP64 and FP32 leaves.

Maps against the oracle's dense local problem: both sides' errors are below
(rows of the elimination) x u x cond, 256 x 1.1e-16 x 1e2 = 3e-12 in FP64 (K with
sigma^2 = 1: cond of a leaf below 1e2 over its diagonal), 1e-11 as in the other
leaf tests; in FP32 with errors that add as roots 16 x 6e-8 x 1e2 = 1e-4.
Solves: refinement takes its residuals from kernels of its own,
so a wrong particular problem or pressure does not converge; after the steps
given the solution has the FP64 one's 1e-9.
"""
import numpy as np
import pytest

import inputs
from conftest import rel
from oracle.geometry import Decomposition
from oracle.local import LeafProblem

from test_gpu_parity import _oracle_seg_key

pytestmark = pytest.mark.gpu

# nx, ny, sub, seg
GRIDS = [(67, 90, (4, 4), (4, 4)),            # cells: 391 leaves, last column 3 wide
         (41, 83, (2, 16), (1, 4)),           # cells, 12 segments
         (33, 70, (1, 16), (1, 16)),          # cells, one cell a row
         (39, 50, (2, 8), (1, 1)),            # cells, 20 segments
         (45, 70, (3, 8), (1, 1)),            # planes, 22 segments
         (43, 61, (4, 4), (1, 1)),            # planes: as many segments as cells
         (405, 395, (8, 8), (8, 8)),          # cells: 2550 leaves
         (330, 395, (8, 8), (8, 8)),          # planes: 2100 leaves
         (405, 397, (8, 8), (2, 2)),          # planes: 16 segments
         (985, 971, (16, 16), (16, 16)),      # cells: 3782 leaves of 16 x 16
         (940, 971, (16, 16), (16, 16)),      # planes: 3599 leaves, one per warp
         (1105, 1149, (16, 16), (4, 4)),      # planes: 5040 leaves, two per warp (8 * 630)
         (1121, 1137, (16, 16), (4, 4)),      # 71 x 72 = 5112
         (1137, 1121, (16, 16), (8, 8)),      # 72 x 71, one row of cells at the top
         (1153, 1105, (16, 16), (4, 4))]      # 73 x 70 = 5110 = 8 * 638 + 6, one column at the right


def _build(mr, torch, nx, ny, sub, seg, fp32):
    prob = inputs.darcy_problem(nx, ny, K=np.exp(np.random.default_rng(nx + ny).standard_normal((ny, nx))),
                                bc="left_right", sub=sub, seg=seg)
    s = mr.Solver(torch.from_numpy(prob.K).cuda(), prob.Lx, prob.Ly, prob.sub, prob.seg, prob.alpha, prob.bc_type,
                  precision=mr.binding.MRCM_MIXED if fp32 else mr.binding.MRCM_FP64)
    if fp32:
        mr.mrcm_set_mixed_leaves(s.ctx, 1)
    s.build_basis()
    return s, prob


def _sample(n):
    return sorted({0, 1, n // 3, n // 2, n // 2 + 1, n - 7, n - 3, n - 2, n - 1})


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("nx,ny,sub,seg", GRIDS)
def test_leaf_maps_on_both_sides_of_the_rule(mrcm_lib, nx, ny, sub, seg, fp32):
    import torch
    import paper_2009_07965_gb300 as mr
    s, prob = _build(mr, torch, nx, ny, sub, seg, fp32)
    dec = Decomposition(prob)
    for leaf in _sample(len(dec.leaves)):
        lp = LeafProblem(dec, leaf)
        R_o, _ = lp.robin_to_flux()
        okey = {_oracle_seg_key(dec, t): k for k, t in enumerate(lp.segs)}
        perm = []
        for t in mr.mrcm_node_segments(s.ctx, leaf):
            si = mr.mrcm_segment_info(s.ctx, t)
            perm.append(okey[(si["axis"], si["line"], si["lo"])])
        assert rel(mr.mrcm_node_operator(s.ctx, leaf), R_o[np.ix_(perm, perm)]) < (1e-4 if fp32 else 1e-11), leaf
    s.close()


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("nx,ny,sub,seg", GRIDS)
def test_solves_on_both_sides_of_the_rule(mrcm_lib, nx, ny, sub, seg, fp32):
    import torch
    import paper_2009_07965_gb300 as mr
    out = []
    for mixed, steps in ((fp32, 14 if fp32 else 1), (False, 3)):
        s, prob = _build(mr, torch, nx, ny, sub, seg, mixed)
        mr.mrcm_set_refinement(s.ctx, steps)
        q = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
        q[ny // 2, nx // 3] = 0.5
        s.solve(q, torch.from_numpy(prob.bc_val).cuda())
        torch.cuda.synchronize()
        res = mr.mrcm_residual_history(s.ctx)
        assert res[-1] < 1e-4 * res[0] or res[-1] < 1e-11, res
        out.append([t.cpu().numpy() for t in (s.p, s.Fx, s.Fy)])
        s.close()
    for a, b in zip(*out):
        assert rel(a, b) < 1e-9


@pytest.mark.parametrize("nx,ny,sub,seg", [(67, 90, (4, 4), (4, 4)), (41, 83, (2, 16), (2, 4)),
                                           (405, 395, (8, 8), (8, 8)), (70, 60, (8, 8), (4, 4))])
def test_leaf_fields_of_both_forms(mrcm_lib, nx, ny, sub, seg):
    # column s of A^-1 B, in single precision on output
    import torch
    import paper_2009_07965_gb300 as mr
    s, prob = _build(mr, torch, nx, ny, sub, seg, False)
    dec = Decomposition(prob)
    leaves = _sample(len(dec.leaves))
    ids = torch.tensor(leaves, dtype=torch.int32, device="cuda")
    psi = torch.zeros(len(leaves), 256, 16, dtype=torch.float32, device="cuda")
    mr.binding.mrcm_leaf_fields(s.ctx, ids, psi)
    psi = psi.cpu().numpy()
    for k, leaf in enumerate(leaves):
        lp = LeafProblem(dec, leaf)
        okey = {_oracle_seg_key(dec, t): i for i, t in enumerate(lp.segs)}
        X = np.linalg.solve(lp.A, lp.B)
        for j, t in enumerate(mr.mrcm_node_segments(s.ctx, leaf)):
            si = mr.mrcm_segment_info(s.ctx, t)
            x = X[:, okey[(si["axis"], si["line"], si["lo"])]]
            assert np.max(np.abs(psi[k, :lp.n, j] - x)) <= 1e-6 * np.max(np.abs(x)), (leaf, j)
    s.close()
