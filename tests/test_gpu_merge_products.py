"""The merged maps of blocked merges (2g > 32), whose products X = -W C and
R = R_oo + C^T X run as split products on the tensor cores, against the same
merge formed on the host from the children's maps; the last test does so on
levels large enough for the block sweep (count (2g)^2 >= 540000) and the
strips.

The sizes put 2g, m and the two children's shares of m on and off the edges
of the 64 x 32 product tiles and of the 64-entry chunks of k, odd ones among
them.  FP64: the host's own partial-pivot LU and products are good to about
2g u times the condition of the interface matrix (below 1e3 for these
fields), so 2g u 1e3 < 256 * 1.1e-16 * 1e3 = 3e-11 bounds both sides'
errors; the maps of the mixed form carry FP32 merges, 2g 2^-24 1e3 / 10 per
merge with the same reasoning, below 1.5e-3 at 2g = 256 (the FP32 LU-free
elimination of the quasi-definite form stays far inside it).
"""
import numpy as np
import pytest

import inputs
from conftest import rel

pytestmark = pytest.mark.gpu

# nx, ny, seg, alpha
GRIDS = [(96, 512, 1, 1.0),        # 2g up to 192, chunks of 64 and 32
         (80, 330, 1, 0.5),        # truncated leaves: odd g and m
         (333, 70, 2, 2.0),
         (272, 272, 4, 1.0)]       # 2g = 68 and 72: one entry row past a tile


def _merge_on_host(mr, ctx, prob, node):
    info = mr.mrcm_node_info(ctx, node)
    s1, s2 = (mr.mrcm_node_segments(ctx, info[c]) for c in ("c1", "c2"))
    R1, R2 = (mr.mrcm_node_operator(ctx, info[c]) for c in ("c1", "c2"))
    pos2 = {t: k for k, t in enumerate(s2)}
    gam = [t for t in s1 if t in pos2]
    g1, g2 = [k for k, t in enumerate(s1) if t in pos2], [pos2[t] for t in gam]
    gs = set(gam)
    o1, o2 = ([k for k, t in enumerate(s) if t not in gs] for s in (s1, s2))
    D = []
    for t in gam:
        si = mr.mrcm_segment_info(ctx, t)
        e = np.arange(si["lo"], si["lo"] + si["len"])
        ka, kb = ((prob.K[e, si["line"] - 1], prob.K[e, si["line"]]) if si["axis"] == 0 else
                  (prob.K[si["line"] - 1, e], prob.K[si["line"], e]))
        D.append(np.mean(2 * ka * kb / (ka + kb)) / (2 * prob.alpha))
    g = len(gam)
    M = np.block([[R1[np.ix_(g1, g1)] + np.diag(D), -np.diag(D)], [-np.diag(D), R2[np.ix_(g2, g2)] + np.diag(D)]])
    C = np.zeros((2 * g, len(o1) + len(o2)))
    C[:g, :len(o1)] = R1[np.ix_(g1, o1)]
    C[g:, len(o1):] = R2[np.ix_(g2, o2)]
    R = -C.T @ np.linalg.solve(M, C)
    R[:len(o1), :len(o1)] += R1[np.ix_(o1, o1)]
    R[len(o1):, len(o1):] += R2[np.ix_(o2, o2)]
    return R


@pytest.mark.parametrize("precision,tol", [("fp64", 3e-11), ("mixed", 1.5e-3)])
@pytest.mark.parametrize("nx,ny,seg,alpha", GRIDS)
def test_blocked_merges_match_the_host(mrcm_lib, nx, ny, seg, alpha, precision, tol):
    import torch
    import paper_2009_07965_gb300 as mr
    prob = inputs.darcy_problem(nx, ny, sigma2=2.0, corr=0.1, seed=nx, bc="left_right", seg=(seg, seg), alpha=alpha)
    s = mr.Solver(torch.from_numpy(prob.K).cuda(), prob.Lx, prob.Ly, prob.sub, prob.seg, prob.alpha, prob.bc_type,
                  precision=mr.binding.MRCM_FP64 if precision == "fp64" else mr.binding.MRCM_MIXED)
    s.build_basis()
    seen = {}
    for v in range(mr.mrcm_query(s.ctx, "LEAVES"), mr.mrcm_query(s.ctx, "NODES")):
        i = mr.mrcm_node_info(s.ctx, v)
        if i["g"] > 16 and i["m"] > 0:
            seen.setdefault((i["g"], i["m"]), v)      # one node of every shape
    assert len(seen) >= 3
    for shape, v in seen.items():
        e = rel(mr.mrcm_node_operator(s.ctx, v), _merge_on_host(mr, s.ctx, prob, v))
        assert e <= tol, (shape, e)
    s.close()


@pytest.mark.parametrize("precision,tol", [("fp64", 3e-11), ("mixed", 1.5e-3)])
def test_block_sweep_levels_match_the_host(mrcm_lib, precision, tol):
    # 40 problems of 170 x 147 cells, one-face segments: 2g = 294 at the root's
    # children's level, 170 and 148 below (a last block of 38, 42 or 20 rows)
    import torch
    import paper_2009_07965_gb300 as mr
    probs = [inputs.darcy_problem(170, 147 + 3 * (k % 2), sigma2=2.0, corr=0.1, seed=90 + k, bc="left_right",
                                  seg=(1, 1)) for k in range(40)]
    b = mr.BatchSolver([torch.from_numpy(p.K).cuda() for p in probs], [(p.Lx, p.Ly) for p in probs],
                       [p.bc_type for p in probs], sub=probs[0].sub, seg=(1, 1), alpha=1.0,
                       precision=mr.binding.MRCM_FP64 if precision == "fp64" else mr.binding.MRCM_MIXED)
    b.build_basis()
    count, first = {}, {}
    nodes = mr.mrcm_query(b.ctx, "NODES")
    owner = [-1] * nodes
    roots = [v for v in range(nodes) if mr.mrcm_node_info(b.ctx, v)["parent"] < 0]
    for k, r in enumerate(roots):
        stack = [r]
        while stack:
            v = stack.pop()
            owner[v] = k
            i = mr.mrcm_node_info(b.ctx, v)
            stack += [c for c in (i["c1"], i["c2"]) if c >= 0]
    for v in range(mr.mrcm_query(b.ctx, "LEAVES"), nodes):
        i = mr.mrcm_node_info(b.ctx, v)
        if i["m"] > 0 and i["g"] > 32:
            count[i["height"]] = count.get(i["height"], 0) + 1
            first.setdefault((i["height"], i["g"], i["m"]), v)
    blocked = {s: v for s, v in first.items() if count[s[0]] * (2 * s[1]) ** 2 >= 540000}
    assert len(blocked) >= 3 and any(2 * s[1] % 64 for s in blocked)
    for s, v in blocked.items():
        e = rel(mr.mrcm_node_operator(b.ctx, v), _merge_on_host(mr, b.ctx, probs[owner[v]], v))
        assert e <= tol, (s, e)
    b.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny,seg", [(170, 147, 1), (145, 150, 1), (276, 140, 2)])
def test_phase_sweep_gives_the_bits_of_the_cooperative_one(mrcm_lib, nx, ny, seg, precision):
    # 33 problems have 66 systems at the height of two merges per problem (one
    # launch per phase, tcgen05), 30 have 60 (cooperative, mma.sync); the digit
    # products are exact in both, so every map agrees bit for bit.  2g = 148 to
    # 170, 130 and 136: last blocks of 2, 8, 20 and 42 rows, one and two row pairs
    import torch
    import paper_2009_07965_gb300 as mr
    probs = [inputs.darcy_problem(nx, ny, sigma2=2.0, corr=0.1, seed=k % 5, bc="left_right", seg=(seg, seg))
             for k in range(33)]
    maps = []
    for n in (33, 30):
        b = mr.BatchSolver([torch.from_numpy(p.K).cuda() for p in probs[:n]], [(p.Lx, p.Ly) for p in probs[:n]],
                           [p.bc_type for p in probs[:n]], sub=probs[0].sub, seg=(seg, seg), alpha=1.0,
                           precision=mr.binding.MRCM_FP64 if precision == "fp64" else mr.binding.MRCM_MIXED)
        b.build_basis()
        nodes = mr.mrcm_query(b.ctx, "NODES")
        info = [mr.mrcm_node_info(b.ctx, v) for v in range(nodes)]
        top = max(i["height"] for i in info)
        maps.append([mr.mrcm_node_operator(b.ctx, v) for h in range(top, 0, -1)
                     for v in [u for u in range(nodes) if info[u]["height"] == h][:2] if info[v]["m"] > 0])
        b.close()
    assert len(maps[0]) == len(maps[1]) > 4
    for x, y in zip(*maps):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny,seg", [(170, 147, 1), (163, 150, 1)])
def test_strips_give_the_bits_of_the_tiles(mrcm_lib, nx, ny, seg, precision):
    # 40 problems have heights wide enough for the strips of X and R
    # (2g <= 128), 6 problems take the tiles; g, m and the children's
    # shares of m on and off the edges of the 64 x 32 tiles and of
    # the 16-entry steps of k.  One chunk of k: exact digit products in both
    import torch
    import paper_2009_07965_gb300 as mr
    probs = [inputs.darcy_problem(nx, ny, sigma2=2.0, corr=0.1, seed=k % 5, bc="left_right", seg=(seg, seg))
             for k in range(40)]
    maps, n_small = [], 6
    for n in (40, n_small):
        b = mr.BatchSolver([torch.from_numpy(p.K).cuda() for p in probs[:n]], [(p.Lx, p.Ly) for p in probs[:n]],
                           [p.bc_type for p in probs[:n]], sub=probs[0].sub, seg=(seg, seg), alpha=1.0,
                           precision=mr.binding.MRCM_FP64 if precision == "fp64" else mr.binding.MRCM_MIXED)
        b.build_basis()
        nodes = mr.mrcm_query(b.ctx, "NODES")
        info = [mr.mrcm_node_info(b.ctx, v) for v in range(nodes)]
        heights = {}
        for v, i in enumerate(info):
            if i["height"] > 0:
                heights.setdefault(i["height"], []).append(v)
        out = []
        for h in sorted(heights):
            width = max(2 * info[v]["g"] for v in heights[h])
            # the same inverses in both: up to 2g = 64, or enough work for the block sweep in the small batch
            if 32 < width <= 64 or 64 < width <= 128 and len(heights[h]) * n_small / n * width ** 2 >= 540000:
                out += [((h, v - heights[h][0]), mr.mrcm_node_operator(b.ctx, v)) for v in heights[h][:6]]
        maps.append(out)
        b.close()
    assert len(maps[0]) == len(maps[1]) >= 12
    for (k0, x), (k1, y) in zip(*maps):
        assert k0 == k1 and np.array_equal(x, y), k0
