// The 3D path: Robin and face coefficients, refinement residuals and the
// face fluxes.
//
// arXiv 2009.07965 runs its experiments in 3D (Section 5.1): box subdomains,
// rectangular interfaces cut into patches of H-bar (Section 4).  The Robin
// coefficient of a segment t is Eq. (robin.beta) with K_eff from Eq.
// (permeff): Keff_t = mean over the faces of t of 2 K_a K_b / (K_a + K_b),
// beta_t = alpha Hbar_t / Keff_t with Hbar_t = sqrt(|t|) (the patch side of
// a square patch), and the Robin coupling D_t = |t| / (2 beta_t).
//
// Leaves.  The grid is tiled by blocks of the patch shape (at most 64
// cells), so a patch between two subdomains is exactly the shared side of
// two blocks.  Inside a subdomain every face between two blocks is its own
// segment: with one unknown pair per fine face the Robin coupling reproduces
// the two-point flux exactly, whatever beta (the one-face-segment property of
// Eqs. 11.2-14.2), so merging the blocks of a subdomain solves its local
// Robin problems exactly -- a nested dissection of the subdomain by the same
// merges that couple subdomains.  The blocks' own local problems run in the
// leaf kernels (kernels_leaf.cu).
#include "leaf_geometry.cuh"

#include <algorithm>

namespace mrcm {
namespace {

__device__ __forceinline__ double hnorm3(const Grid3& G, int d) {
    return d == 0 ? G.hx : (d == 1 ? G.hy : G.hz);
}

// beta_t and D_t of every segment (faces: v outer along the second
// tangential axis, u inner along the first).
__global__ void seg_beta3_kernel(DevView v) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= v.nseg) return;
    const Grid3& G = v.g3;
    const int d = v.seg_axis[t], line = v.seg_line[t];
    const int lo1 = v.seg_lo[t], len1 = v.seg_len[t], lo2 = v.seg_lo2[t], len2 = v.seg_len2[t];
    const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
    double sum = 0.0;
    for (int w = lo2; w < lo2 + len2; ++w)
        for (int u = lo1; u < lo1 + len1; ++u) {
            int pos[3];
            pos[d] = line; pos[t1] = u; pos[t2] = w;
            const double kb = v.K[cell3(G, pos[0], pos[1], pos[2])];
            pos[d] = line - 1;
            const double ka = v.K[cell3(G, pos[0], pos[1], pos[2])];
            sum += 2.0 * ka * kb / (ka + kb);
        }
    const int nf = len1 * len2;
    const double keff = sum / nf;
    const double area = nf * area3(G, d);
    const double beta = v.alpha * sqrt(area) / keff;
    v.seg_beta[t] = beta;
    v.seg_D[t] = area / (2.0 * beta);
}

// Face coefficients seen from the lower (cL) and the upper (cU) cell:
// interior T = |e| / (r_a + r_b), skeleton rho = |e| / (r_c + beta_t),
// Dirichlet tau = 2 K_c |e| / h, Neumann 0 (r_c = h / (2 K_c)).
__global__ void face_coef3_kernel(DevView v) {
    const Grid3& G = v.g3;
    const long long total = v.nxface + v.nyface + v.nzface;
    for (long long f = blockIdx.x * (long long)blockDim.x + threadIdx.x; f < total;
         f += (long long)gridDim.x * blockDim.x) {
        int d, i, j, k;
        long long fl;
        double *cL, *cU;
        const int* fseg;
        if (f < v.nxface) {
            d = 0; fl = f; cL = v.cxL; cU = v.cxU; fseg = v.xface_seg;
            i = (int)(fl % (G.nx + 1)); const long long r = fl / (G.nx + 1); j = (int)(r % G.ny); k = (int)(r / G.ny);
        } else if (f < v.nxface + v.nyface) {
            d = 1; fl = f - v.nxface; cL = v.cyL; cU = v.cyU; fseg = v.yface_seg;
            i = (int)(fl % G.nx); const long long r = fl / G.nx; j = (int)(r % (G.ny + 1)); k = (int)(r / (G.ny + 1));
        } else {
            d = 2; fl = f - v.nxface - v.nyface; cL = v.czL; cU = v.czU; fseg = v.zface_seg;
            i = (int)(fl % G.nx); const long long r = fl / G.nx; j = (int)(r % G.ny); k = (int)(r / G.ny);
        }
        const int n_d = d == 0 ? G.nx : (d == 1 ? G.ny : G.nz);
        const int pos = d == 0 ? i : (d == 1 ? j : k);
        const double area = area3(G, d), hn = hnorm3(G, d);
        const long long cu = pos < n_d ? cell3(G, i, j, k) : -1;
        const long long cl = pos > 0 ? cell3(G, i - (d == 0), j - (d == 1), k - (d == 2)) : -1;
        double vl = 0.0, vu = 0.0;
        if (cl < 0) {
            if (G.bc[2 * d]) vu = 2.0 * v.K[cu] * area / hn;
        } else if (cu < 0) {
            if (G.bc[2 * d + 1]) vl = 2.0 * v.K[cl] * area / hn;
        } else {
            // quotients as products with a reciprocal within an ulp (rcp_nr)
            const double ra = hn * rcp_nr(2.0 * v.K[cl]), rb = hn * rcp_nr(2.0 * v.K[cu]);
            const int t = fseg[fl];
            if (t >= 0) {
                const double beta = v.seg_beta[t];
                vl = area * rcp_nr(ra + beta);
                vu = area * rcp_nr(rb + beta);
            } else {
                vl = vu = area * rcp_nr(ra + rb);
            }
        }
        cL[fl] = vl;
        cU[fl] = vu;
    }
}

__device__ __forceinline__ void block_max3(unsigned long long* slot, double x) {
    __shared__ double wmax[32];
    double a = fabs(x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x < 32) {
        double b = threadIdx.x < (blockDim.x >> 5) ? wmax[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
        // non-negative doubles order like their bit patterns
        if (threadIdx.x == 0 && b > 0.0) atomicMax(slot, (unsigned long long)__double_as_longlong(b));
    }
}

// Refinement residuals in FP64 of the discrete equations (Eqs. 11.2-14.2
// with lumped RT0) at the current state (p_hi + p_lo, the segments' Robin
// data lambda^a = P - beta U, lambda^b = P + beta U): cell balances
// E_c = sum of outward fluxes - q_c, rcell = -E_c.
__global__ void __launch_bounds__(256) residual3_cells_kernel(DevView v, const double* __restrict__ q,
                                                              const double* __restrict__ bc_val, int step) {
    const Grid3& G = v.g3;
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    double e = 0.0;
    if (c < v.ncell) {
        const int i = (int)(c % G.nx);
        const long long r = c / G.nx;
        const int j = (int)(r % G.ny), k = (int)(r / G.ny);
        const double pc = v.p_hi[c] + v.p_lo[c];
        double E = -q[c];
        for (int side = 0; side < 6; ++side) {
            const int d = side >> 1, up = side & 1;
            const int pos = d == 0 ? i : (d == 1 ? j : k);
            const int nd = d == 0 ? G.nx : (d == 1 ? G.ny : G.nz);
            long long f;
            const double* cf;
            const int* fs;
            if (d == 0) { f = xface3(G, i + up, j, k); cf = up ? v.cxL : v.cxU; fs = v.xface_seg; }
            else if (d == 1) { f = yface3(G, i, j + up, k); cf = up ? v.cyL : v.cyU; fs = v.yface_seg; }
            else { f = zface3(G, i, j, k + up); cf = up ? v.czL : v.czU; fs = v.zface_seg; }
            const double coef = cf[f];
            if (up ? pos == nd - 1 : pos == 0) {
                const double g = bc_value3(G, bc_val, side, i, j, k);
                E += G.bc[side] ? coef * (pc - g) : area3(G, d) * g;
                continue;
            }
            const int t = fs[f];
            if (t >= 0) {
                const double2 l = v.seg_lam_dd[2 * t + (up ? 0 : 1)];
                E += coef * (pc - (l.x + l.y));
            } else {
                const long long nb = c + (up ? 1 : -1) * (d == 0 ? 1LL : (d == 1 ? (long long)G.nx : (long long)G.nx * G.ny));
                E += coef * (pc - (v.p_hi[nb] + v.p_lo[nb]));
            }
        }
        e = E;
        v.rcell[c] = -E;
    }
    block_max3(v.res_max + step, e);
}

// Segment residuals: E13 = F^a + F^b (Eq. 13.2), E14 = F^a - F^b - 2 |t| U
// (Eq. 14.2, divided by beta), outward integrated fluxes of the two sides;
// they enter the correction solve as right-hand sides of the two interface
// rows of the segment.
__global__ void __launch_bounds__(128) residual3_segments_kernel(DevView v, int step) {
    const Grid3& G = v.g3;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    double E13 = 0.0, E14 = 0.0;
    if (t < v.nseg) {
        const int d = v.seg_axis[t], line = v.seg_line[t];
        const int lo1 = v.seg_lo[t], len1 = v.seg_len[t], lo2 = v.seg_lo2[t], len2 = v.seg_len2[t];
        const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
        const double2 l2a = v.seg_lam_dd[2 * t], l2b = v.seg_lam_dd[2 * t + 1];
        const double la = l2a.x + l2a.y, lb = l2b.x + l2b.y;
        const double* cL = d == 0 ? v.cxL : (d == 1 ? v.cyL : v.czL);
        const double* cU = d == 0 ? v.cxU : (d == 1 ? v.cyU : v.czU);
        double Fa = 0.0, Fb = 0.0;
        for (int w = lo2; w < lo2 + len2; ++w)
            for (int u = lo1; u < lo1 + len1; ++u) {
                int pos[3];
                pos[d] = line; pos[t1] = u; pos[t2] = w;
                const long long cb = cell3(G, pos[0], pos[1], pos[2]);
                const long long f = d == 0 ? xface3(G, pos[0], pos[1], pos[2])
                                           : (d == 1 ? yface3(G, pos[0], pos[1], pos[2]) : zface3(G, pos[0], pos[1], pos[2]));
                pos[d] = line - 1;
                const long long ca = cell3(G, pos[0], pos[1], pos[2]);
                Fa += cL[f] * ((v.p_hi[ca] + v.p_lo[ca]) - la);
                Fb += cU[f] * ((v.p_hi[cb] + v.p_lo[cb]) - lb);
            }
        const double area = len1 * len2 * area3(G, d);
        const double two_u = 2.0 * area * (v.segU[t] + v.segU_lo[t]);
        E13 = Fa + Fb;
        E14 = (Fa - Fb) - two_u;
        v.sadj[v.seg_lam_a[t]] = -0.5 * (E13 + E14);
        v.sadj[v.seg_lam_b[t]] = -0.5 * (E13 - E14);
    }
    block_max3(v.res_max + step, fmax(fabs(E13), fabs(E14)));
}

// Cell pressures and face fluxes (+axis sign) from the state (p_hi + p_lo,
// the segments' Robin data of the interface unknowns); on the skeleton the
// mean of the two one-sided values rho (p_c - lambda) of the blocks on either
// side.  iface (optional): the one-sided values [Fa_x, Fb_x, Fa_y, Fb_y,
// Fa_z, Fb_z], side a the lower block, both equal to F off the skeleton.
__global__ void face_flux3_kernel(DevView v, const double* __restrict__ bc_val, double* __restrict__ p,
                                  double* __restrict__ Fx, double* __restrict__ Fy, double* __restrict__ Fz,
                                  double* __restrict__ iface) {
    const Grid3& G = v.g3;
    const long long nf = v.nxface + v.nyface + v.nzface;
    for (long long f = blockIdx.x * (long long)blockDim.x + threadIdx.x; f < nf + v.ncell;
         f += (long long)gridDim.x * blockDim.x) {
        if (f >= nf) {
            const long long c = f - nf;
            p[c] = v.p_hi[c] + v.p_lo[c];
            continue;
        }
        int d, i, j, k;
        long long fl;
        const double *cL, *cU;
        const int* fseg;
        double* out;
        if (f < v.nxface) {
            d = 0; fl = f; cL = v.cxL; cU = v.cxU; fseg = v.xface_seg; out = Fx;
            i = (int)(fl % (G.nx + 1)); const long long r = fl / (G.nx + 1); j = (int)(r % G.ny); k = (int)(r / G.ny);
        } else if (f < v.nxface + v.nyface) {
            d = 1; fl = f - v.nxface; cL = v.cyL; cU = v.cyU; fseg = v.yface_seg; out = Fy;
            i = (int)(fl % G.nx); const long long r = fl / G.nx; j = (int)(r % (G.ny + 1)); k = (int)(r / (G.ny + 1));
        } else {
            d = 2; fl = f - v.nxface - v.nyface; cL = v.czL; cU = v.czU; fseg = v.zface_seg; out = Fz;
            i = (int)(fl % G.nx); const long long r = fl / G.nx; j = (int)(r % G.ny); k = (int)(r / G.ny);
        }
        const int n_d = d == 0 ? G.nx : (d == 1 ? G.ny : G.nz);
        const int pos = d == 0 ? i : (d == 1 ? j : k);
        const double area = area3(G, d);
        double F, fa1 = 0.0, fb1 = 0.0;
        bool skel = false;
        if (pos == 0) {
            const double pb = v.p_hi[cell3(G, i, j, k)] + v.p_lo[cell3(G, i, j, k)];
            const double g = bc_value3(G, bc_val, 2 * d, i, j, k);
            F = G.bc[2 * d] ? -(cU[fl] * (pb - g)) : -(area * g);
        } else {
            const int ai = i - (d == 0), aj = j - (d == 1), ak = k - (d == 2);
            const long long ca = cell3(G, ai, aj, ak);
            const double pa = v.p_hi[ca] + v.p_lo[ca];
            if (pos == n_d) {
                const double g = bc_value3(G, bc_val, 2 * d + 1, ai, aj, ak);
                F = G.bc[2 * d + 1] ? cL[fl] * (pa - g) : area * g;
            } else {
                const long long cb = cell3(G, i, j, k);
                const double pb = v.p_hi[cb] + v.p_lo[cb];
                const int t = fseg[fl];
                if (t >= 0) {
                    const double2 la = v.seg_lam_dd[2 * t], lb = v.seg_lam_dd[2 * t + 1];
                    const double fa = cL[fl] * (pa - (la.x + la.y));
                    const double fb = -(cU[fl] * (pb - (lb.x + lb.y)));
                    F = 0.5 * (fa + fb);
                    fa1 = fa;
                    fb1 = fb;
                    skel = true;
                } else {
                    F = cL[fl] * (pa - pb);
                }
            }
        }
        out[fl] = F;
        if (iface) {
            // block of this axis: Fa at 2 (faces of the earlier axes), Fb after it
            const long long nd = d == 0 ? v.nxface : (d == 1 ? v.nyface : v.nzface);
            const long long base = 2 * (d == 0 ? 0 : (d == 1 ? v.nxface : v.nxface + v.nyface));
            iface[base + fl] = skel ? fa1 : F;
            iface[base + nd + fl] = skel ? fb1 : F;
        }
    }
}

inline unsigned grid_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    if (b > 152LL * 16) b = 152LL * 16;
    return (unsigned)std::max(b, 1LL);
}

}  // namespace

cudaError_t launch_coef3(const DevView& v, cudaStream_t s) {
    if (v.nseg > 0) seg_beta3_kernel<<<(v.nseg + 127) / 128, 128, 0, s>>>(v);
    face_coef3_kernel<<<grid_for(v.nxface + v.nyface + v.nzface, 256), 256, 0, s>>>(v);
    return cudaGetLastError();
}

cudaError_t launch_residual3(const DevView& v, const double* q, const double* bc_val, int step, cudaStream_t s) {
    residual3_cells_kernel<<<(unsigned)((v.ncell + 255) / 256), 256, 0, s>>>(v, q, bc_val, step);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || v.nseg == 0) return e;
    residual3_segments_kernel<<<(v.nseg + 127) / 128, 128, 0, s>>>(v, step);
    return cudaGetLastError();
}

cudaError_t launch_face_fluxes3(const DevView& v, const double* bc_val, double* p, double* Fx, double* Fy,
                                double* Fz, double* iface, cudaStream_t s) {
    const long long n = v.nxface + v.nyface + v.nzface + v.ncell;
    face_flux3_kernel<<<grid_for(n, 256), 256, 0, s>>>(v, bc_val, p, Fx, Fy, Fz, iface);
    return cudaGetLastError();
}

}  // namespace mrcm
