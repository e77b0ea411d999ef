"""3D blocks whose x-y planes have one, two or four cells, four to a warp in the
solve: against the 3D oracle (rel-L2 <= 1e-10 as in the other 3D parity tests),
with one to eight planes a block, patches of every aspect, and block counts that
leave the last warp and the last CTA part empty (a CTA takes 16 blocks)."""
import pytest

import inputs
from conftest import rel

from test_gpu_3d import _solve

pytestmark = pytest.mark.gpu

# n, sub, seg
CASES = [((6, 5, 7), (3, 5, 7), (1, 1, 1)),        # 210 blocks, one plane
         ((8, 8, 6), (4, 4, 6), (2, 2, 1)),        # 96 blocks of one plane of four cells
         ((6, 6, 10), (3, 3, 5), (1, 1, 5)),       # 72 blocks of one column
         ((10, 6, 8), (5, 6, 4), (1, 2, 2)),       # planes of two cells
         ((12, 6, 8), (12, 3, 4), (4, 1, 4)),      # planes of four cells in a row
         ((12, 8, 16), (4, 4, 8), (2, 2, 8)),      # eight planes
         ((8, 12, 9), (8, 4, 9), (1, 4, 3))]


@pytest.mark.parametrize("n,sub,seg", CASES, ids=lambda c: "x".join(map(str, c)))
@pytest.mark.parametrize("bc", ["left_right", "quarter_five_spot"])
def test_narrow_blocks_match_the_oracle(n, sub, seg, bc, mrcm_lib):
    import torch
    from oracle.mrcm3d import solve_mrcm3d
    prob = inputs.darcy_problem_3d(*n, sigma2=2.0, corr=(0.3, 0.3, 0.2), seed=sum(n), bc=bc, sub=sub, seg=seg,
                                   alpha=1.5, L=(1.0, 0.8, 0.6))
    if bc == "left_right":
        prob.q[n[2] // 2, n[1] // 3, n[0] // 2] = 0.3
    g, o = _solve(prob, torch, refine=2), solve_mrcm3d(prob)
    for key in ("p", "Fx", "Fy", "Fz"):
        assert rel(g[key], o[key]) < 1e-10, key
