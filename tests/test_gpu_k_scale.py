"""Scaling K by a power of two scales every quantity of the method exactly: no
result may depend on it, far out in FP64 as little as near the ends of the FP32
range in the mixed form.  Single passes: the same computation at both scales,
up to what FP32 subnormals round at the far end (entries 2^-24 of the largest
and less: 1e-6 of the result).
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def _solver(mr, torch, K, seg, alpha=1.0, mixed=False):
    ny, nx = K.shape
    prob = inputs.darcy_problem(nx, ny, K=K, bc="left_right", seg=(seg, seg), alpha=alpha)
    s = mr.Solver(torch.from_numpy(prob.K).cuda(), prob.Lx, prob.Ly, prob.sub, prob.seg, prob.alpha, prob.bc_type,
                  precision=mr.binding.MRCM_MIXED if mixed else mr.binding.MRCM_FP64)
    mr.mrcm_set_refinement(s.ctx, 0)
    s.build_basis()
    return s, prob


@pytest.mark.parametrize("mixed,power", [(False, 300), (False, -300), (True, 110), (True, -90)])
def test_scaling_k_by_a_power_of_two_changes_nothing(mrcm_lib, mixed, power):
    import torch
    import paper_2009_07965_gb300 as mr
    K = np.exp(np.random.default_rng(4).standard_normal((96, 140)))
    out = []
    for f in (1.0, 2.0 ** power):
        s, prob = _solver(mr, torch, K * f, 1, mixed=mixed)
        p, Fx, Fy = s.solve(torch.from_numpy(prob.q).cuda(), torch.from_numpy(prob.bc_val).cuda())
        torch.cuda.synchronize()
        out.append([t.cpu().numpy() / g for t, g in ((p, 1.0), (Fx, f), (Fy, f))])
        s.close()
    for a, b in zip(*out):
        assert np.linalg.norm(a - b) <= (1e-6 if mixed else 1e-13) * np.linalg.norm(a)
