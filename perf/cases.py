"""Workloads of the Recursive MRCM library as its users run them.

A case is a plain dict.  "kind" picks the call sequence:

  step       a new permeability on a kept context: set_permeability,
             build_basis, solve (Monte-Carlo and time-lapse loops, and the
             first solve on any field);
  solve      new sources and boundary data on a built basis (well schedules);
  batch      the step on a batched context of independent problems;
  surrogate  one training step of the learned basis network.

2D problems have 16 x 16 leaves and quarter-five-spot ("qfs": no flow on any
side, a source and a sink) or left-right ("lr": p = 1 / 0 on x, no flow on y)
data; 3D boxes have 16^3 leaves, 4^3-cell blocks and left-right data.  K is
log-normal with exponential covariance.  "refine" is the number of
refinement steps, -1 the library's default; the mixed form refines until its
result is as good as the FP64 form's (its default stops at 1e-8).
"""
import math

import numpy as np
import torch

import paper_2009_07965_gb300 as mr
from paper_2009_07965_gb300 import binding as B
from paper_2009_07965_gb300.surrogate import LAYERS, BasisSurrogate


def _flat(name, nx, ny, **kw):
    c = dict(name=name, kind="step", nx=nx, ny=ny, nz=0, sigma2=3.0, corr=0.05, bc="qfs", seg=4, alpha=1.0,
             mixed=False, refine=-1, tune=False, stream=True)
    c.update(kw)
    return c


def _box(name, nx, ny, nz, **kw):
    c = dict(name=name, kind="step", nx=nx, ny=ny, nz=nz, sigma2=2.0, corr=0.2, bc="lr", seg=4, alpha=1.0,
             mixed=False, refine=-1, tune=False, stream=True)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest useful problem, on the default stream (no graphs): launches and latency
        _flat("square64", 64, 64, sigma2=1.0, corr=0.1, bc="lr", stream=False),
        # a ragged grid with two-face segments: truncated leaves, twice the interface unknowns
        _flat("ragged333x517_seg2", 333, 517, sigma2=2.0, corr=0.1, bc="lr", seg=2, alpha=2.0),
        # one realisation of an ordinary size, with the default refinement
        _flat("square1024", 1024, 1024, sigma2=4.0),
        # the next well schedule on the same field, one-sided fluxes wanted
        _flat("solve1024", 1024, 1024, sigma2=4.0, kind="solve"),
        # the flagship field, the paper's single pass, launch shapes tuned once
        _flat("square4096", 4096, 4096, corr=0.02, refine=0, tune=True),
        # the same field in the mixed form
        _flat("square4096_mixed", 4096, 4096, corr=0.02, mixed=True, refine=4, tune=True),
        # the mixed form on an ordinary ragged grid
        _flat("ragged1500x700_mixed", 1500, 700, corr=0.05, bc="lr", mixed=True, refine=4),
        # an ensemble of fields of different sizes in one context
        dict(name="ensemble24", kind="batch", count=24, nmin=250, nmax=1000, corr=0.05, alpha=1.0, refine=-1),
        # a small box
        _box("box64x64x32", 64, 64, 32),
        # an ordinary box in FP64
        _box("box128x128x64", 128, 128, 64),
        # the largest box, in the mixed form
        _box("box256x256x64_mixed", 256, 256, 64, mixed=True, refine=3),
        # training the learned basis: BF16 convolutions forward and backward, Adam
        dict(name="surrogate_train256", kind="surrogate", count=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.random()
    sigma2, alpha = round(rng.uniform(1.0, 4.0), 2), rng.choice([0.5, 1.0, 1.0, 2.0])
    bc = rng.choice(["qfs", "lr"])
    if pick < 0.45:
        nx, ny = _log_int(rng, 48, 2600), _log_int(rng, 48, 2600)
        seg = rng.choice([4, 4, 4, 8]) if nx * ny > 600000 else rng.choice([4, 4, 2, 8])
        c = _flat("", nx, ny, sigma2=sigma2, corr=round(rng.uniform(0.02, 0.1), 3), bc=bc, alpha=alpha, seg=seg,
                  refine=rng.choice([-1, -1, 0]), stream=rng.random() < 0.8)
        if rng.random() < 0.3:
            c["kind"] = "solve"
    elif pick < 0.6:
        c = _flat("", _log_int(rng, 200, 3000), _log_int(rng, 200, 3000), sigma2=sigma2,
                  corr=round(rng.uniform(0.02, 0.1), 3), bc=bc, mixed=True, refine=5)
    elif pick < 0.72:
        c = dict(kind="batch", count=_log_int(rng, 3, 32), nmin=_log_int(rng, 60, 400), corr=0.05, alpha=alpha,
                 refine=rng.choice([-1, 0]))
        c["nmax"] = c["nmin"] + rng.randint(10, 600)
    elif pick < 0.95:
        n = [16 * _log_int(rng, 1, 9) for _ in range(3)]
        n[0] += 16 * (max(n) == 16)
        mixed = rng.random() < 0.4
        c = _box("", *n, sigma2=sigma2, bc=rng.choice(["lr", "lr", "qfs"]), alpha=alpha, mixed=mixed,
                 refine=4 if mixed else -1)
    else:
        c = dict(kind="surrogate", count=_log_int(rng, 32, 512))
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs
def _field(n, h, corr, sigma2, seed):
    """exp(sigma xi) on an array of n cells (array order), xi a Gaussian field
    with covariance exp(-|r / corr|) by circulant embedding."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    pad = []
    for nd, hd, cd in zip(n, h, corr):
        p = nd + int(math.ceil(6.0 * cd / hd))
        pad.append((p + 63) // 64 * 64)
    r2 = torch.zeros((), dtype=torch.float64, device="cuda")
    for d, (p, hd, cd) in enumerate(zip(pad, h, corr)):
        i = torch.arange(p, dtype=torch.float64, device="cuda")
        x = torch.minimum(i, p - i) * (hd / cd)
        r2 = r2 + (x * x).reshape([-1 if k == d else 1 for k in range(len(n))])
    lam = torch.fft.fftn(torch.exp(-torch.sqrt(r2))).real.clamp_min(0.0) / math.prod(pad)
    z = torch.complex(torch.randn(pad, generator=g, dtype=torch.float64, device="cuda"),
                      torch.randn(pad, generator=g, dtype=torch.float64, device="cuda"))
    xi = torch.fft.fftn(z.mul_(torch.sqrt(lam))).real[tuple(slice(0, nd) for nd in n)]
    return torch.exp(math.sqrt(sigma2) * xi).contiguous()


def _shape(case):
    return ((case["nz"],) if case["nz"] else ()) + (case["ny"], case["nx"])


def _extent(case):
    """(Lx, Ly[, Lz]): unit length along x, square / cubic cells."""
    return tuple(k / case["nx"] for k in reversed(_shape(case)))


def _bc_type(case):
    nd = len(_shape(case))
    return (1, 1) + (0,) * (2 * nd - 2) if case["bc"] == "lr" else (0,) * (2 * nd)


def _problem(case, seed):
    """K, q, bc_val of one problem (CUDA, float64)."""
    n, L = _shape(case), _extent(case)
    nd = len(n)
    h = [L[nd - 1 - a] / n[a] for a in range(nd)]
    corr = [case["corr"]] * nd
    if nd == 3:
        corr[0] = case["corr"] / 4           # shorter in depth
    K = _field(n, h, corr, case["sigma2"], seed)
    q = torch.zeros(n, dtype=torch.float64, device="cuda")
    nb = sum(2 * K.numel() // k for k in n)
    bcv = torch.zeros(nb, dtype=torch.float64, device="cuda")
    rng = np.random.default_rng(seed)
    if case["bc"] == "lr":
        side = K.numel() // case["nx"]
        bcv[:side] = 1.0 + float(rng.uniform(0.0, 0.1))
    else:
        q.view(-1)[0], q.view(-1)[-1] = 1.0, -1.0
    if case["kind"] == "solve":
        # a schedule of balanced wells at random cells
        at = rng.choice(K.numel(), 16, replace=False)
        q.view(-1)[torch.from_numpy(at).cuda()] += torch.tensor([0.5, -0.5] * 8, dtype=torch.float64, device="cuda")
    return K, q, bcv


def _members(case):
    """Sizes and variances of a batch's problems: the ensemble is part of the
    plan, so it depends on the case alone."""
    rng = np.random.default_rng(4000)
    out = []
    for _ in range(case["count"]):
        nx, ny = (int(x) for x in rng.integers(case["nmin"], case["nmax"] + 1, 2))
        out.append((nx, ny, float(rng.uniform(1.0, 4.0))))
    return out


def _member(case, k, seed):
    nx, ny, s2 = _members(case)[k]
    K = _field((ny, nx), (1.0 / ny, 1.0 / nx), (case["corr"],) * 2, s2, 1000 * seed + k)
    q = torch.zeros_like(K)
    bcv = torch.zeros(2 * (nx + ny), dtype=torch.float64, device="cuda")
    bcv[:ny] = 1.0
    return K, q, bcv


def _training_data(case, seed):
    """Patches (bf16, 18 x 18 x 16 channels) of a log-normal field and fields
    in [0, 1] that fall off from the segment they belong to."""
    cnt = case["count"]
    side = int(math.ceil(math.sqrt(cnt)))
    n = 16 * side + 2
    lk = torch.log(_field((n, n), (1.0 / 1024,) * 2, (0.05,) * 2, 4.0, seed)).float()
    pt = lk.unfold(0, 18, 16).unfold(1, 18, 16).reshape(-1, 18, 18)[:cnt]
    pt = 0.5 * (pt - pt[:, 1:-1, 1:-1].mean(dim=(1, 2), keepdim=True))
    x = torch.zeros(cnt, 18, 18, 16, dtype=torch.bfloat16, device="cuda")
    x[..., 0] = pt.bfloat16()
    t = torch.arange(16, device="cuda", dtype=torch.float32)
    mid = 4 * torch.arange(4, device="cuda", dtype=torch.float32) + 1.5
    cx = torch.cat([torch.full_like(mid, -0.5), torch.full_like(mid, 15.5), mid, mid])
    cy = torch.cat([mid, mid, torch.full_like(mid, -0.5), torch.full_like(mid, 15.5)])
    dist = torch.sqrt((t[None, :, None] - cx) ** 2 + (t[:, None, None] - cy) ** 2)
    target = torch.exp(-0.25 * dist) * torch.sigmoid(pt[:, 1:-1, 1:-1, None])
    return x, target.contiguous()


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "surrogate":
        x, target = _training_data(case, seed)
        return dict(kind=kind, net=BasisSurrogate("cuda", seed=seed), x=x, target=target)
    stream = torch.cuda.Stream() if case.get("stream", True) else torch.cuda.default_stream()
    if kind == "batch":
        probs = [_member(case, k, seed) for k in range(case["count"])]
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            s = mr.BatchSolver([p[0] for p in probs], [(1.0, 1.0)] * len(probs), [(1, 1, 0, 0)] * len(probs),
                               alpha=case["alpha"], stream=stream)
        if case["refine"] >= 0:
            mr.mrcm_set_refinement(s.ctx, case["refine"])
        torch.cuda.synchronize()
        return dict(kind=kind, solver=s, stream=stream, K=[p[0] for p in probs], q=[p[1] for p in probs],
                    bc=[p[2] for p in probs])
    K, q, bcv = _problem(case, seed)
    torch.cuda.synchronize()
    prec = B.MRCM_MIXED if case["mixed"] else B.MRCM_FP64
    with torch.cuda.stream(stream):
        if case["nz"]:
            s = mr.Solver3D(K, L=_extent(case), seg=(case["seg"],) * 3, alpha=case["alpha"], bc_type=_bc_type(case),
                            stream=stream, precision=prec)
        else:
            s = mr.Solver(K, *_extent(case), seg=(case["seg"],) * 2, alpha=case["alpha"], bc_type=_bc_type(case),
                          stream=stream, precision=prec)
        if case["refine"] >= 0:
            mr.mrcm_set_refinement(s.ctx, case["refine"])
        if case["tune"] or kind == "solve":
            s.build_basis()
        if case["tune"]:
            mr.mrcm_autotune(s.ctx, 3)
    torch.cuda.synchronize()
    return dict(kind=kind, solver=s, stream=stream, K=K, q=q, bc=bcv)


def run(state):
    if state["kind"] == "surrogate":
        net = state["net"]
        loss = net.train_step(state["x"], state["target"])
        # Adam's running means carry the step's gradients
        return dict(loss=loss, mw=net.mw, mb=net.mb)
    s = state["solver"]
    with torch.cuda.stream(state["stream"]):
        if state["kind"] == "solve":
            out = s.solve(state["q"], state["bc"], want_iface=True)
            return list(out) + [s.iface]
        s.set_permeability(state["K"])
        s.build_basis()
        out = s.solve(state["q"], state["bc"])
        # a batch: p, Fx, Fy of every problem, packed problem after problem
        return [s.p, s.Fx, s.Fy] if state["kind"] == "batch" else list(out)


def work(case):
    """K, sources and boundary values in, pressures and face fluxes out;
    the flops of a direct method (banded Cholesky leaves, LU merges) and two
    passes over its local factors."""
    if case["kind"] == "surrogate":
        macs = 256 * 9 * sum(cin * cout for cin, cout, _, _ in LAYERS)
        inner = 256 * 9 * sum(cin * cout for cin, cout, _, _ in LAYERS[1:])
        return {"bytes": case["count"] * (18 * 18 * 16 * 2 + 256 * 16 * 4), "flops": 2 * case["count"] * (2 * macs + inner)}
    if case["kind"] == "batch":
        total = {"bytes": 0, "flops": 0}
        for nx, ny, _ in _members(case):
            one = _one(nx, ny, 0, (1.0, 1.0), 4, (1, 1, 0, 0))
            for k in total:
                total[k] += one[k]
        return total
    w = _one(case["nx"], case["ny"], case["nz"], _extent(case), case["seg"], _bc_type(case))
    if case["kind"] == "solve":
        cells = case["nx"] * case["ny"]
        passes = 1 + (1 if case["refine"] < 0 else case["refine"])
        return {"bytes": 8 * cells * (1 + 3 + 4), "flops": passes * 4 * cells * (16 + 16)}
    return w


def _one(nx, ny, nz, L, seg, bc):
    n = (nx, ny, nz) if nz else (nx, ny)
    cells = math.prod(n)
    flops = mr.mrcm_plan_query(n, L, (16,) * len(n), (seg,) * len(n), bc, "MODEL_BUILD_FLOPS")
    return {"bytes": 8 * cells * (2 + 1 + len(n)), "flops": flops + 4 * cells * (16 + 16)}


# ---------------------------------------------------------------- 64 bits, without the library
def _along(x, dim, lo, hi):
    return x.narrow(dim, lo, hi - lo)


def _exact_darcy(K, q, bcv, bc_type, L, sub, seg, alpha):
    """The discrete MRCM solution by dense linear algebra: every leaf's local
    Robin problem by Cholesky, one dense interface system over all segments
    (scaled by the Robin couplings, refined), then the final local solves.
    Arrays in array order; sub, seg, L, bc_type in x, y, z order."""
    nd, n, dev = K.dim(), list(K.shape), K.device
    f64 = dict(dtype=torch.float64, device=dev)
    h = [L[nd - 1 - a] / n[a] for a in range(nd)]
    sub, seg = list(reversed(sub)), list(reversed(seg))
    cell = math.prod(h)
    nl = [-(-n[a] // sub[a]) for a in range(nd)]
    diag, rhs = torch.zeros(n, **f64), q.clone()
    down = {}                              # coupling to the lower neighbour inside the leaf
    rho = {}                               # (axis, up): Robin coefficient and segment per cell
    D, beta, nseg, faces, off = [], [], 0, {}, 0
    sides = {}
    for d in range(nd):
        a = nd - 1 - d
        shp = [n[k] for k in range(nd) if k != a]
        for up in (0, 1):
            m = math.prod(shp)
            sides[(a, up)] = bcv[off:off + m].reshape(shp)
            off += m
    for a in range(nd):
        d = nd - 1 - a
        area = cell / h[a]
        r = h[a] / (2.0 * K)
        lo, hi = _along(K, a, 0, n[a] - 1), _along(K, a, 1, n[a])
        ra, rb = _along(r, a, 0, n[a] - 1), _along(r, a, 1, n[a])
        T = area / (ra + rb)
        skel = (torch.arange(1, n[a], device=dev) % sub[a] == 0)
        where = skel.nonzero().reshape(-1)
        cl, cu = T.clone(), T.clone()
        sid = torch.full(T.shape, -1, dtype=torch.int64, device=dev)
        if where.numel():
            idx = torch.arange(where.numel(), device=dev).reshape([-1 if k == a else 1 for k in range(nd)])
            for k in range(nd):
                if k != a:
                    c = torch.arange(n[k], device=dev) // seg[k]
                    idx = idx * (-(-n[k] // seg[k])) + c.reshape([-1 if j == k else 1 for j in range(nd)])
            count = int(idx.max()) + 1
            hm = (2.0 * lo * hi / (lo + hi)).index_select(a, where)
            flat = idx.reshape(-1)
            num = torch.zeros(count, **f64).index_add_(0, flat, torch.ones(flat.numel(), **f64))
            keff = torch.zeros(count, **f64).index_add_(0, flat, hm.reshape(-1)) / num
            size = num * area
            bt = alpha * (size if nd == 2 else torch.sqrt(size)) / keff
            bf = bt[idx]
            cl.index_copy_(a, where, area / (ra.index_select(a, where) + bf))
            cu.index_copy_(a, where, area / (rb.index_select(a, where) + bf))
            sid.index_copy_(a, where, idx + nseg)
            D.append(size / (2.0 * bt))
            beta.append(bt)
            nseg += count
        _along(diag, a, 0, n[a] - 1).add_(cl)
        _along(diag, a, 1, n[a]).add_(cu)
        t = torch.zeros(n, **f64)
        _along(t, a, 1, n[a]).copy_(torch.where(sid < 0, T, torch.zeros_like(T)))
        down[a] = t
        for up in (0, 1):
            rr, ss = torch.zeros(n, **f64), torch.full(n, -1, dtype=torch.int64, device=dev)
            w = (0, n[a] - 1) if up else (1, n[a])
            _along(rr, a, *w).copy_(torch.where(sid >= 0, cl if up else cu, torch.zeros_like(T)))
            _along(ss, a, *w).copy_(sid)
            rho[(a, up)] = (rr, ss)
            at, g = (n[a] - 1 if up else 0), sides[(a, up)]
            if bc_type[2 * d + up]:
                tau = 2.0 * K.select(a, at) * area / h[a]
                diag.select(a, at).add_(tau)
                rhs.select(a, at).add_(tau * g)
            else:
                rhs.select(a, at).sub_(area * g)
        faces[a] = (T, cl, cu, sid, area)

    def leaves(x, fill):
        padded = torch.full([nl[k] * sub[k] for k in range(nd)], fill, dtype=x.dtype, device=dev)
        padded[tuple(slice(0, k) for k in n)] = x
        order = [v for k in range(nd) for v in (nl[k], sub[k])]
        perm = [2 * k for k in range(nd)] + [2 * k + 1 for k in range(nd)]
        return padded.reshape(order).permute(perm).reshape(math.prod(nl), -1)

    nleaf, nc = math.prod(nl), math.prod(sub)
    strides = [math.prod(sub[k + 1:]) for k in range(nd)]
    ldiag, lrhs = leaves(diag, 1.0), leaves(rhs, 0.0)
    ldown = {a: leaves(down[a], 0.0) for a in range(nd)}
    lrob = [(leaves(rho[k][0], 0.0), leaves(rho[k][1], -1), k[1]) for k in rho]
    D = torch.cat(D) if D else torch.zeros(0, **f64)
    sq = torch.sqrt(D).repeat_interleave(2)
    G = torch.zeros(2 * nseg, 2 * nseg, **f64)
    g0 = torch.zeros(2 * nseg, **f64)
    pieces = []
    ar = torch.arange(nc, device=dev)
    chunk = max(1, (1 << 27) // (nc * nc))
    for l0 in range(0, nleaf, chunk):
        sl = slice(l0, min(nleaf, l0 + chunk))
        m = sl.stop - sl.start
        A = torch.diag_embed(ldiag[sl])
        for a in range(nd):
            cells = ar[(ar // strides[a]) % sub[a] > 0]
            A[:, cells, cells - strides[a]] = -ldown[a][sl][:, cells]
            A[:, cells - strides[a], cells] = -ldown[a][sl][:, cells]
        # the unknown 2 t + side of every Robin face, made dense per leaf
        unk = torch.cat([torch.where(s[sl] >= 0, 2 * s[sl] + (0 if up else 1), -1) for _, s, up in lrob], 1)
        val = torch.cat([r[sl] for r, _, _ in lrob], 1)
        cel = ar.repeat(len(lrob)).expand(m, -1)
        kept = []
        for i in range(m):
            kept.append(torch.unique(unk[i][unk[i] >= 0]))
        ms = max([1] + [k.numel() for k in kept])
        Bm = torch.zeros(m, nc, ms, **f64)
        for i in range(m):
            ok = unk[i] >= 0
            col = torch.searchsorted(kept[i], unk[i][ok])
            Bm[i].index_put_((cel[i][ok], col), val[i][ok], accumulate=True)
        C = torch.linalg.cholesky(A)
        del A
        Z = torch.linalg.solve_triangular(C, torch.cat([Bm, lrhs[sl][:, :, None]], 2), upper=False)
        R = Z[:, :, :ms].mT @ Z[:, :, :ms] - torch.diag_embed(Bm.sum(1))
        rb = (Z[:, :, :ms].mT @ Z[:, :, ms:])[:, :, 0]
        for i in range(m):
            u = kept[i]
            k = u.numel()
            G[u[:, None], u[None, :]] = R[i, :k, :k] / (sq[u][:, None] * sq[u][None, :])
            g0[u] = -rb[i, :k] / sq[u]
        pieces.append((sl, C, Z, kept, ms))
    if nseg:
        e = torch.arange(nseg, device=dev) * 2
        G[e, e] += 1.0
        G[e + 1, e + 1] += 1.0
        G[e, e + 1] -= 1.0
        G[e + 1, e] -= 1.0
        closed = not any(bc_type)
        if closed:
            v = sq / torch.linalg.norm(sq)
            G -= v[:, None] * v[None, :]
        LU, piv = torch.linalg.lu_factor(G)
        x = torch.linalg.lu_solve(LU, piv, g0[:, None])
        for _ in range(2):
            x = x + torch.linalg.lu_solve(LU, piv, g0[:, None] - G @ x)
        lam = x[:, 0] / sq
        del LU, G
    p_l = torch.zeros(nleaf, nc, **f64)
    for sl, C, Z, kept, ms in pieces:
        y = Z[:, :, ms].clone()
        for i, u in enumerate(kept):
            if u.numel():
                y[i] += Z[i, :, :u.numel()] @ lam[u]
        p_l[sl] = torch.linalg.solve_triangular(C.mT, y[:, :, None], upper=True)[:, :, 0]
    del pieces
    p = p_l.reshape(nl + sub).permute([v for k in range(nd) for v in (k, nd + k)])
    p = p.reshape([nl[k] * sub[k] for k in range(nd)])[tuple(slice(0, k) for k in n)].contiguous()
    shift = p.mean() if not any(bc_type) else 0.0
    p = p - shift
    out, one_sided = [p], []
    for d in range(nd):
        a = nd - 1 - d
        T, cl, cu, sid, area = faces[a]
        shp = list(n)
        shp[a] += 1
        F, Fa, Fb = (torch.zeros(shp, **f64) for _ in range(3))
        pa, pb = _along(p, a, 0, n[a] - 1), _along(p, a, 1, n[a])
        inner = T * (pa - pb)
        fa, fb = inner, inner
        if nseg:
            on = sid >= 0
            s = sid.clamp_min(0)
            fa = torch.where(on, cl * (pa - (lam[2 * s] - shift)), inner)
            fb = torch.where(on, -cu * (pb - (lam[2 * s + 1] - shift)), inner)
        for o, f in ((F, 0.5 * (fa + fb)), (Fa, fa), (Fb, fb)):
            _along(o, a, 1, n[a]).copy_(f)
            for up in (0, 1):
                at, g, sg = (n[a] if up else 0), sides[(a, up)], (1.0 if up else -1.0)
                pc, Kc = p.select(a, n[a] - 1 if up else 0), K.select(a, n[a] - 1 if up else 0)
                o.select(a, at).copy_(sg * (2.0 * Kc * area / h[a] * (pc - g) if bc_type[2 * d + up] else area * g))
        out.append(F)
        one_sided += [Fa.reshape(-1), Fb.reshape(-1)]
    return out, torch.cat(one_sided)


def _unknowns(n, seg):
    """Robin unknowns of a 2D grid with 16 x 16 leaves, or of a 3D one."""
    total = 0
    for a in range(len(n)):
        t = -(-n[a] // 16) - 1
        for k in range(len(n)):
            if k != a:
                t *= -(-n[k] // seg)
        total += 2 * t
    return total


def _exact_training(case, seed):
    """Loss and (1 - beta1) x gradients of one step, without the roundings to
    bf16 inside the network."""
    x, target = _training_data(case, seed)
    net = BasisSurrogate("cuda", seed=seed)          # the initial weights only
    w = [t.double().requires_grad_() for t in net.wbf]
    b = [t.double().requires_grad_() for t in net.b]
    y = x.double().permute(0, 3, 1, 2)
    for wi, bi, (_, _, pad, relu) in zip(w, b, LAYERS):
        y = torch.nn.functional.conv2d(y, wi.permute(0, 3, 1, 2), bi, padding=pad)
        y = torch.relu(y) if relu else y
    loss = 0.5 * ((y.permute(0, 2, 3, 1) - target.double()) ** 2).sum() / case["count"]
    g = torch.autograd.grad(loss, w + b)
    return dict(loss=float(loss), mw=[0.1 * t for t in g[:len(w)]], mb=[0.1 * t for t in g[len(w):]])


def exact(case, seed):
    if case["kind"] == "surrogate":
        return _exact_training(case, seed)
    if case["kind"] == "batch":
        if sum(_unknowns((ny, nx), 4) ** 3 for nx, ny, _ in _members(case)) > 24000 ** 3:
            return None
        out = []
        for k in range(case["count"]):
            K, q, bcv = _member(case, k, seed)
            one, _ = _exact_darcy(K, q, bcv, (1, 1, 0, 0), (1.0, 1.0), (16, 16), (4, 4), case["alpha"])
            out.append([t.reshape(-1) for t in one])
        return [torch.cat(t) for t in zip(*out)]
    n = _shape(case)
    if _unknowns(n, case["seg"]) > 24000 or math.prod(n) > (1 << 20):
        return None
    K, q, bcv = _problem(case, seed)
    nd = len(n)
    out, one_sided = _exact_darcy(K, q, bcv, _bc_type(case), _extent(case), (16,) * nd, (case["seg"],) * nd,
                                  case["alpha"])
    return out + [one_sided] if case["kind"] == "solve" else out
