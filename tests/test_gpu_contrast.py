"""Merged maps of fields of high contrast, where the rows of the products'
operands are graded: the node maps of blocked merges (2g > 32) against the same
merge in extended precision from the library's own maps of the children.

The error of entry (i, j) is taken over (R_ii R_jj)^1/2.  Rounding errors of
sums of 2g terms grow as (2g)^1/2 u, and the elimination has its condition:
both are in the error of the host's plain FP64 merge of the same node (scaled
symmetrically, partial pivoting).  So a map may be 4 max(host error, (2g)^1/2 u)
away from the extended-precision one, the host's error being the largest over
the nodes of the grid with that 2g or more (one node's may be small by luck);
FP32 merges 8 (2g)^1/2 2^-24.
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _channels(ny, nx, decades, seed):
    """Winding two-cell channels of 10^decades times the background."""
    r = np.random.default_rng(seed)
    K = np.exp(0.5 * r.standard_normal((ny, nx)))
    chan = np.zeros((ny, nx), bool)
    for _ in range(max(nx, ny) // 12):
        if r.random() < 0.5:
            j = int(r.integers(ny))
            for i in range(nx):
                j = min(max(j + int(r.integers(-1, 2)), 0), ny - 1)
                chan[j:j + 2, i] = True
        else:
            i = int(r.integers(nx))
            for j in range(ny):
                i = min(max(i + int(r.integers(-1, 2)), 0), nx - 1)
                chan[j, i:i + 2] = True
    return np.where(chan, 10.0 ** decades, 1.0) * K


def _random(ny, nx, decades, seed):
    return 10.0 ** (decades * np.random.default_rng(seed).random((ny, nx)))


def _solve(M, C):
    """M^-1 C in M's precision: symmetric scaling, Gauss-Jordan with partial pivoting."""
    s = 1 / np.sqrt(np.abs(np.diag(M)))
    A = np.concatenate([M * s[:, None] * s[None, :], C * s[:, None]], 1)
    n = len(M)
    for k in range(n):
        p = k + int(np.argmax(np.abs(A[k:, k])))
        if p != k:
            A[[k, p]] = A[[p, k]]
        A[k, k:] /= A[k, k]
        f = A[:, k].copy()
        f[k] = 0
        A[:, k:] -= np.outer(f, A[k, k:])
    return A[:, n:] * s[:, None]


def _merge(mr, ctx, K, alpha, node, dtype):
    info = mr.mrcm_node_info(ctx, node)
    s1, s2 = (mr.mrcm_node_segments(ctx, info[c]) for c in ("c1", "c2"))
    R1, R2 = (mr.mrcm_node_operator(ctx, info[c]).astype(dtype) for c in ("c1", "c2"))
    pos2 = {t: k for k, t in enumerate(s2)}
    gam = [t for t in s1 if t in pos2]
    gs = set(gam)
    g1, g2 = [k for k, t in enumerate(s1) if t in pos2], [pos2[t] for t in gam]
    o1, o2 = ([k for k, t in enumerate(s) if t not in gs] for s in (s1, s2))
    D = []
    for t in gam:
        si = mr.mrcm_segment_info(ctx, t)
        e = np.arange(si["lo"], si["lo"] + si["len"])
        ka, kb = ((K[e, si["line"] - 1], K[e, si["line"]]) if si["axis"] == 0 else
                  (K[si["line"] - 1, e], K[si["line"], e]))
        D.append(np.mean(2 * ka * kb / (ka + kb)) / (2 * alpha))
    d, g = np.diag(np.array(D)).astype(dtype), len(gam)
    M = np.block([[R1[np.ix_(g1, g1)] + d, -d], [-d, R2[np.ix_(g2, g2)] + d]])
    C = np.zeros((2 * g, len(o1) + len(o2)), dtype=dtype)
    C[:g, :len(o1)] = R1[np.ix_(g1, o1)]
    C[g:, len(o1):] = R2[np.ix_(g2, o2)]
    X = _solve(M, C)
    R = np.zeros((C.shape[1],) * 2, dtype=dtype)
    R[:len(o1), :len(o1)] = R1[np.ix_(o1, o1)]
    R[len(o1):, len(o1):] = R2[np.ix_(o2, o2)]
    for k in range(2 * g):
        R -= np.outer(C[k], X[k])
    return R


def _err(R, ref):
    d = np.sqrt(np.abs(np.diag(ref)))
    return float(np.max(np.abs(R - ref) / np.outer(d, d)))


def _solver(mr, torch, K, seg, alpha=1.0, mixed=False, refine=0):
    ny, nx = K.shape
    prob = inputs.darcy_problem(nx, ny, K=K, bc="left_right", seg=(seg, seg), alpha=alpha)
    s = mr.Solver(torch.from_numpy(prob.K).cuda(), prob.Lx, prob.Ly, prob.sub, prob.seg, prob.alpha, prob.bc_type,
                  precision=mr.binding.MRCM_MIXED if mixed else mr.binding.MRCM_FP64)
    mr.mrcm_set_refinement(s.ctx, refine)
    s.build_basis()
    return s, prob


def _nodes(mr, s):
    seen = {}
    for v in range(mr.mrcm_query(s.ctx, "LEAVES"), mr.mrcm_query(s.ctx, "NODES")):
        i = mr.mrcm_node_info(s.ctx, v)
        if i["g"] > 16 and i["m"] > 0:
            seen.setdefault((i["height"], i["g"]), []).append(v)
    return {k: [v[0], v[len(v) // 2], v[-1]] for k, v in seen.items()}


@pytest.mark.parametrize("kind,decades,alpha", [("channels", 5, 1.0), ("channels", 8, 1.0), ("channels", 11, 1.0),
                                                ("channels", 11, 10.0), ("random", 2, 1.0), ("random", 2, 100.0),
                                                ("random", 8, 1.0), ("random", 11, 1.0)])
def test_maps_of_high_contrast_fields_keep_fp64_accuracy(mrcm_lib, kind, decades, alpha):
    import torch
    import paper_2009_07965_gb300 as mr
    K = (_channels if kind == "channels" else _random)(140, 96, decades, 8)
    s, prob = _solver(mr, torch, K, 1, alpha)
    got, host = [], []
    for (h, g), vs in sorted(_nodes(mr, s).items()):
        for v in dict.fromkeys(vs):
            ref = _merge(mr, s.ctx, K, alpha, v, LD)
            host.append((2 * g, _err(_merge(mr, s.ctx, K, alpha, v, np.float64), ref)))
            got.append((2 * g, h, _err(mr.mrcm_node_operator(s.ctx, v), ref)))
    s.close()
    assert len(got) >= 6
    for g2, h, e in got:
        worst = max(x for w, x in host if w >= g2)
        assert e <= 4 * max(worst, np.sqrt(g2) * 2.0 ** -53), (g2, h, e, worst)


@pytest.mark.parametrize("seg", [1, 2])
def test_fp32_merges_keep_24_bits(mrcm_lib, seg):
    import torch
    import paper_2009_07965_gb300 as mr
    K = np.exp(np.random.default_rng(3).standard_normal((150, 200)))
    s, prob = _solver(mr, torch, K, seg, mixed=True)
    mr.mrcm_set_mixed_split(s.ctx, 1 << 20)              # every merge in FP32
    s.build_basis()
    n = 0
    for (h, g), vs in sorted(_nodes(mr, s).items()):
        e = _err(mr.mrcm_node_operator(s.ctx, vs[0]), _merge(mr, s.ctx, K, 1.0, vs[0], np.float64))
        assert e <= 8 * np.sqrt(2 * g) * 2.0 ** -24, (h, g, e)
        n += 1
    s.close()
    assert n >= 3
