"""The up sweep's wide form (eight outputs to eight lanes; heights with 2g >= 16
and enough outputs) against its narrow form: a batch of 48 problems has heights
of about 2000 merges and takes the wide form there, each problem on its own has
heights of at most 48 merges and takes the narrow one everywhere.

One-face segments and truncated leaves put m on and off multiples of eight and
2g on and off multiples of sixteen.  No refinement.  The two differ in rounding
only (order of sums, form of the interface inverses): each is good to about
2g u times the condition of the interface matrices, 300 x 1.1e-16 x 1e3 = 3e-11.
"""
import pytest

import inputs
from conftest import gpu_solve, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,seg", [(147, 131, (1, 1)), (150, 144, (2, 2))])
def test_wide_up_sweep_matches_single_contexts(mrcm_lib, nx, ny, seg):
    import torch
    import paper_2009_07965_gb300 as mr
    probs = [inputs.darcy_problem(nx, ny + 2 * (k % 2), sigma2=1.0, corr=0.1, seed=k % 4, bc="left_right", seg=seg)
             for k in range(48)]
    b = mr.BatchSolver([torch.from_numpy(p.K).cuda() for p in probs], [(p.Lx, p.Ly) for p in probs],
                       [p.bc_type for p in probs], sub=probs[0].sub, seg=seg, alpha=1.0)
    mr.mrcm_set_refinement(b.ctx, 0)
    b.build_basis()
    b.solve([torch.from_numpy(p.q).cuda() for p in probs], [torch.from_numpy(p.bc_val).cuda() for p in probs])
    torch.cuda.synchronize()
    outs = [[t.cpu().numpy() for t in o] for o in b.split()]
    b.close()
    for k in (0, 1, 2, 3, 47):
        s = gpu_solve(probs[k], want_iface=False, refine=0)
        for x, key in zip(outs[k], ("p", "Fx", "Fy")):
            assert rel(x, s[key]) < 3e-11, (k, key)
        s["solver"].close()
