"""The bounded waits of the block sweeps, made to run out with a limit of zero
polls: the tile waits of the phase-per-launch sweep (64 systems or more per
height) and the grid barriers of the cooperative one.  The build returns
MRCM_ERR_TIMEOUT, and with the default limit back the same context builds the
same bits again.

140 x 140 cells with one-face segments: 2g = 280 at the root, 140 or so below.
64 problems have 64 systems or more at every height above 2g = 64, so that
nothing but the tile waits can run out; a row pair past 256 rows has a piece
of a single tile, whose wait follows its issue at once.  8 problems have
8 * 280^2 >= 540000 at the root: the cooperative sweep.
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def _batch(count, precision):
    import torch
    import paper_2009_07965_gb300 as mr
    probs = [inputs.darcy_problem(140, 140, sigma2=2.0, corr=0.1, seed=k % 3, bc="left_right", seg=(1, 1))
             for k in range(count)]
    b = mr.BatchSolver([torch.from_numpy(p.K).cuda() for p in probs], [(p.Lx, p.Ly) for p in probs],
                       [p.bc_type for p in probs], sub=probs[0].sub, seg=(1, 1), alpha=1.0,
                       precision=mr.binding.MRCM_FP64 if precision == "fp64" else mr.binding.MRCM_MIXED)
    mr.mrcm_set_refinement(b.ctx, 0)
    return b, ([torch.from_numpy(p.q).cuda() for p in probs], [torch.from_numpy(p.bc_val).cuda() for p in probs])


def _results(mr, b, data):
    """Node information; maps of the three heights below the root and the pressures."""
    import torch
    nodes = mr.mrcm_query(b.ctx, "NODES")
    info = [mr.mrcm_node_info(b.ctx, v) for v in range(nodes)]
    top = max(i["height"] for i in info)
    maps = [mr.mrcm_node_operator(b.ctx, v) for h in range(top - 3, top)
            for v in [u for u in range(nodes) if info[u]["height"] == h][:3]]
    b.solve(*data)
    torch.cuda.synchronize()
    return info, maps + [b.p.cpu().numpy().copy()]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("count", [64, 8])
def test_sweep_waits_run_out_and_the_context_recovers(mrcm_lib, count, precision):
    import paper_2009_07965_gb300 as mr
    from paper_2009_07965_gb300 import MrcmError
    b, data = _batch(count, precision)
    b.build_basis()
    info, ref = _results(mr, b, data)
    wide = {}
    for i in info:
        if i["height"] > 0 and i["g"] > 32:
            wide.setdefault(i["height"], []).append(2 * i["g"])
    if count == 64:
        assert all(len(w) >= 64 and len(w) * max(w) ** 2 >= 1 << 20 for w in wide.values())
        assert any(256 < max(w) <= 288 for w in wide.values())
    assert any(len(w) * max(w) ** 2 >= 540000 for w in wide.values())
    mr.mrcm_set_wait_limit(b.ctx, 0)
    with pytest.raises(MrcmError) as e:
        b.build_basis()
    assert e.value.code == -8                    # MRCM_ERR_TIMEOUT
    mr.mrcm_set_wait_limit(b.ctx, -1)
    b.build_basis()
    _, again = _results(mr, b, data)
    b.close()
    assert len(ref) >= 3
    for x, y in zip(ref, again):
        assert np.array_equal(x, y)


def test_tuned_launch_shapes_keep_the_bits_of_the_block_sweep(mrcm_lib):
    import paper_2009_07965_gb300 as mr
    b, data = _batch(8, "fp64")
    b.build_basis()
    _, ref = _results(mr, b, data)
    mr.mrcm_autotune(b.ctx, 1)
    _, tuned = _results(mr, b, data)        # as the last candidate left them
    b.build_basis()
    _, again = _results(mr, b, data)
    b.close()
    for x, y, z in zip(ref, tuned, again):
        assert np.array_equal(x, y) and np.array_equal(x, z)
