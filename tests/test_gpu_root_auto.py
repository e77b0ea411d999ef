"""Which roots MRCM_ROOT_AUTO factors: a single FP64 root system of 1024 <= 2g <
1408.  Read off the phase the root's flops are booked under, and the solution
of the chosen form bit for bit.  One-face segments on n x n cells: 2g = 2 n."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def _root(mr, torch, n, count=1, mixed=False, form=None):
    K = np.exp(np.random.default_rng(n).standard_normal((n, n)))
    p = inputs.darcy_problem(n, n, K=K, bc="left_right", seg=(1, 1))
    prec = mr.binding.MRCM_MIXED if mixed else mr.binding.MRCM_FP64
    Kd, q, bc = (torch.from_numpy(x).cuda() for x in (p.K, p.q, p.bc_val))
    if count > 1:
        s = mr.BatchSolver([Kd] * count, [(p.Lx, p.Ly)] * count, [p.bc_type] * count, sub=p.sub, seg=p.seg, alpha=1.0,
                           precision=prec)
    else:
        s = mr.Solver(Kd, p.Lx, p.Ly, p.sub, p.seg, p.alpha, p.bc_type, precision=prec)
    if form is not None:
        mr.mrcm_set_root_form(s.ctx, form)
    mr.mrcm_set_refinement(s.ctx, 0)
    s.build_basis()
    s.solve([q] * count, [bc] * count) if count > 1 else s.solve(q, bc)
    torch.cuda.synchronize()
    assert mr.mrcm_query(s.ctx, "MAX_GAMMA") == 2 * n
    out = mr.mrcm_phase_flops(s.ctx)["root_factor"] > 0, s.p.cpu().numpy().copy()
    s.close()
    return out


@pytest.mark.parametrize("n,count,mixed,factored", [(496, 1, False, False), (512, 1, False, True),
                                                    (688, 1, False, True), (704, 1, False, False),
                                                    (512, 2, False, False), (512, 1, True, False)])
def test_auto_root_form(mrcm_lib, n, count, mixed, factored):
    import torch
    import paper_2009_07965_gb300 as mr
    fac, p = _root(mr, torch, n, count, mixed)
    assert fac == factored
    form = mr.binding.MRCM_ROOT_FACTOR if factored else mr.binding.MRCM_ROOT_INVERSE
    assert np.array_equal(p, _root(mr, torch, n, count, mixed, form)[1])
