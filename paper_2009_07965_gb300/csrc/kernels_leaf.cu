// Leaf kernels: the local Robin problems of every finest-level block, 2D
// leaves and 3D patch-shaped blocks alike.
//
// arXiv 2009.07965, Eqs. (11.2)-(12.2) on one leaf with lumped RT0 (two-point
// fluxes).  On a skeleton face e of segment t the Robin term gives the
// outward flux F_e = rho_e (p_c - lambda_t), lambda_t = P_t - beta_t U_t
// (n_t . n^i), so the interface data of the MMBF problems (Eqs.
// 11Hhatbasisa / 11Hhatbasisb) enter only through one Robin datum per
// segment.  With the leaf pressure matrix A (SPD: two-point couplings plus
// the Robin / Dirichlet diagonal) and B[c, s] = rho_e for the face e of cell
// c in segment s:
//     p = A^-1 (bbar + B lambda),   F_s = (B^T A^-1 B - W) lambda + B^T A^-1 bbar,
// W_s = sum_{e in s} rho_e.  The Robin-to-flux map R = B^T A^-1 B - W holds
// the traces of all MMBFs of the leaf (coefficient-tracking remark, Section
// 3.2); bbar carries the source and external boundary data (Eqs. addu, addp).
//
// Elimination.  A leaf is a stack of H planes of nb <= 16 cells (2D: the grid
// rows of the leaf; 3D: its x-y planes), and the two-point coupling between
// neighbouring planes is diagonal: A is block tridiagonal with diagonal
// off-diagonal blocks -T_k.  It is eliminated plane by plane from both ends
// towards a middle plane M = H / 2 (half the sequential chain of an
// elimination from one end, and fewer columns of B meet each plane):
//     S_k = A_k - T P T (P of the plane eliminated before),   P_k = S_k^-1,
//     Z_k = B_k + T P Z,   y_k = b_k + T P y                   (likewise),
// with both neighbours' contributions at M.  Then
//     R = sum_k Z_k^T P_k Z_k - W,   rbar = sum_k Z_k^T P_k y_k,
//     x_M = P_M y_M,   x_k = P_k (y_k + T x of the plane next to it towards M).
// The explicit P_k make every pass of the solve phase a chain of H / 2 + 1
// small matrix-vector products.
//
// Arithmetic.  An FP64 instruction holds its scheduler's FP64 pipe for 64
// cycles, so the FP64 instructions of a warp set the pace: only the
// inversions of S_k (Gauss-Jordan on the lower triangle, no pivot search: S_k
// is SPD) and the diagonal scalings run there; the products V = P Z and
// Z^T V go to the tensor cores as split products (split_gemm.cuh) on
// fragments cut from shared memory.
//
// Measured against the elimination cell by cell (banded LDL^T, FP64 FMA loops)
// of before: build 4096^2 13.4 -> 9.4 ms, 333x517 with two-face segments 2.86 ->
// 0.47, box 256x256x64 34.9 -> 16.8; particular problems and pressures of
// 1500x700 per pass 0.20 and 0.22 -> 0.11 and 0.12, of 256x256x64 3.3 and 3.0 ->
// 2.1 and 1.1 (4096^2 1.21 and 1.08 -> 1.22 and 1.11: FP64 pipe either way).
// Of the build's 9.3 ms, 6.0 are FP64 instructions (1690 per leaf, 64 cycles
// each).
//
// Stored for the solve phase: P_k (nb x nb per plane, planes in order) and Z_k
// (nb x c_k, column-major, only the c_k columns that have met the plane): the
// planes below M, then M, then the planes from H - 1 down to M + 1.
#include "block_invert.cuh"
#include "leaf_geometry.cuh"
#include "mrcm_internal.h"
#include "split_gemm.cuh"

#include <algorithm>

namespace mrcm {
namespace {

constexpr int kTeams = 4;         // independent warps of a build CTA (leaf_build_kernel)

// Shared memory of one leaf of a build CTA; mp, cz: the launch's largest
// segment count and the largest column count off the middle plane.
constexpr int kTriP = kPlane * (kPlane + 1) / 2;
__host__ __device__ __forceinline__ int tri_at(int r, int c) {
    const int hi = r > c ? r : c, lo = r > c ? c : r;
    return hi * (hi + 1) / 2 + lo;
}
template <int DIM, class T>
struct LeafBuildSmem {
    T (*P)[kTriP];                  // [2]: the halves' current P (lower triangle, zero outside nb)
    T (*Z)[kPlane + 1];             // [2 cz]: the halves' current Z, by column; V of the middle plane
    T (*V)[kPlane + 1];             // [mp]: P Z; Z of the middle plane
    double* R;                      // packed lower triangle (local segments)
    T (*col)[2][kColSize];          // [2]: pivot columns of each half (sweep_block)
    double (*dg)[kPlane];           // [2]: diagonal of the plane, couplings to cell i - 1 and
    double (*cx)[kPlane];           // i - w0, to the plane before and to the one after
    double (*cy)[kPlane];           // (3D)
    double (*tp)[kPlane];
    double (*tn)[kPlane];
    short *ord, *pos;               // [2 mp]: column -> segment and back, per half
    __host__ __device__ static int zrows(int mp, int cz) { return 2 * cz > mp ? 2 * cz : mp; }
    __host__ __device__ static size_t bytes(int mp, int cz) {
        size_t t = sizeof(T) * (2 * kTriP + (zrows(mp, cz) + mp) * (kPlane + 1) + 4 * kColSize);
        t = (t + 7) / 8 * 8 + sizeof(double) * ((size_t)mp * (mp + 1) / 2 + (DIM == 3 ? 10 : 8) * kPlane) + sizeof(short) * 4 * mp;
        return (t + 15) / 16 * 16;
    }
    __device__ LeafBuildSmem(unsigned char* p, int mp, int cz) {
        T* t = reinterpret_cast<T*>(p);
        P = reinterpret_cast<T (*)[kTriP]>(t); t += 2 * kTriP;
        Z = reinterpret_cast<T (*)[kPlane + 1]>(t); t += zrows(mp, cz) * (kPlane + 1);
        V = reinterpret_cast<T (*)[kPlane + 1]>(t); t += mp * (kPlane + 1);
        col = reinterpret_cast<T (*)[2][kColSize]>(t); t += 4 * kColSize;
        size_t o = (size_t)(reinterpret_cast<unsigned char*>(t) - p);
        double* d = reinterpret_cast<double*>(p + (o + 7) / 8 * 8);
        R = d; d += (size_t)mp * (mp + 1) / 2;
        dg = reinterpret_cast<double (*)[kPlane]>(d); d += 2 * kPlane;
        cx = reinterpret_cast<double (*)[kPlane]>(d); d += 2 * kPlane;
        cy = reinterpret_cast<double (*)[kPlane]>(d); d += DIM == 3 ? 2 * kPlane : 0;
        tp = reinterpret_cast<double (*)[kPlane]>(d); d += 2 * kPlane;
        tn = reinterpret_cast<double (*)[kPlane]>(d); d += 2 * kPlane;
        ord = reinterpret_cast<short*>(d);
        pos = ord + 2 * mp;
    }
};

template <int NW>
__device__ __forceinline__ void leaf_sync() {
    if (NW == 1) __syncwarp();
    else __syncthreads();
}

// A team of NW warps builds LPC leaves (LPC = 2: two leaves in one warp, four
// blocks inverted at a time; LPC = 1: one leaf, two blocks at a time, the
// tensor-core products spread over the warps); a CTA holds TM teams.  The
// teams are independent, but start each inversion and each round of products
// together: the code of a plane is larger than the instruction caches next to
// the schedulers, and warps at different places of it waited for instructions
// a third of their time (4096^2: one warp per CTA 13.0 ms; two 9.7, four 9.4,
// six 9.8, twelve 10.5).
template <int DIM, class T, int NW, int LPC, int TM>
__global__ void __launch_bounds__(32 * NW * TM, NW == 1 ? 12 / TM : (DIM == 3 ? 3 : 4))
leaf_build_kernel(DevView v, int mp, int cz, int bytes) {
    constexpr int GL = 16 / LPC, S = Slices<T>::S, NT = 32 * NW;
    static_assert(LPC == 1 || NW == 1, "two leaves per team only in one warp");
    static_assert(TM == 1 || NW == 1, "several teams only of one warp each");
    extern __shared__ __align__(16) unsigned char smem_all[];
    __shared__ LeafGeo geo_all[LPC * TM];
    const int team = NW == 1 ? threadIdx.x >> 5 : 0;
    unsigned char* smem_raw = smem_all + (size_t)team * LPC * bytes;
    LeafGeo* geos = geo_all + team * LPC;
    const int tid = threadIdx.x - 32 * team, lane = tid & 31, warp = tid >> 5;
    const int leaf0 = (blockIdx.x * TM + team) * LPC;
    // the warp that inverts: warps of one index share a scheduler, so CTAs
    // take turns (as many as SMs are dealt at a time)
    const int wsweep = NW == 1 ? 0 : (blockIdx.x / kRuleSMs) % NW;
    // this lane's block in the inversions: half hf of leaf lf
    const int q = lane / GL, lf = q >> 1, hf = q & 1, gl = lane & (GL - 1);
    const bool present = leaf0 + lf < v.nleaf;
    if (tid < LPC) geos[tid] = leaf_geo<DIM>(v, min(leaf0 + tid, v.nleaf - 1));
    if (TM > 1) __syncthreads();
    leaf_sync<NW>();
    const LeafGeo& G = geos[lf];
    const LeafBuildSmem<DIM, T> Sm(smem_raw + (size_t)lf * bytes, mp, cz);
    bool bad = false;

    // column orders, zeroed R
#pragma unroll 1
    for (int f = 0; f < LPC; ++f) {
        const LeafGeo& g = geos[f];
        const LeafBuildSmem<DIM, T> s(smem_raw + (size_t)f * bytes, mp, cz);
        for (int i = tid; i < 2 * g.m; i += NT) s.pos[(i / g.m) * mp + i % g.m] = (short)-1;
        leaf_sync<NW>();
        for (int h = 0; h < 2; ++h)
            for (int p = tid; p < g.ncols(h); p += NT) {
                const int t = g.segment(h, p);
                s.ord[h * mp + p] = (short)t;
                s.pos[h * mp + t] = (short)p;
            }
        for (int i = tid; i < g.m * (g.m + 1) / 2; i += NT) s.R[i] = 0.0;
        for (int i = tid; i < 2 * cz * (kPlane + 1); i += NT) (&s.Z[0][0])[i] = (T)0;
        for (int i = tid; i < 2 * kTriP; i += NT) s.P[0][i] = (T)0;
    }
    leaf_sync<NW>();

    const BlockSlots<GL> B;
    int steps = 0;                                             // uniform over the CTA
#pragma unroll 1
    for (int f = 0; f < LPC * TM; ++f) steps = max(steps, max(geo_all[f].M, geo_all[f].H - 1 - geo_all[f].M));
    // entry (r, c), r >= c, of the plane's matrix block
    auto plane_entry = [&](const LeafGeo& g, const LeafBuildSmem<DIM, T>& s, int h, int r, int c) -> double {
        if (r == c) return s.dg[h][r];
        double a = 0.0;
        if (r - c == 1 && (DIM == 2 || r % g.w0 != 0)) a = neg_bits(s.cx[h][r]);
        if (DIM == 3 && r - c == g.w0) a = neg_bits(s.cy[h][r]);
        return a;
    };
    const int r16 = tid >> 4, c16 = tid & 15;                  // a half warp per row of 16

    for (int j = 0; j <= steps; ++j) {
        const bool mid = j == steps;
        if (TM > 1) __syncthreads();
        // ---- the planes' coefficients and blocks; inversion (one warp) ------
        if (NW == 1 || warp == wsweep) {
            const int k = mid ? G.M : (hf ? G.H - 1 - j : j);
            const bool act = present && (mid ? hf == 0 : j < G.halfplanes(hf));
            if (act) {
                for (int i = gl; i < G.nb; i += GL) {
                    const CellFaces<DIM> c = cell_faces<DIM>(v, leaf0 + lf, G, k, i);
                    Sm.dg[hf][i] = c.diag();
                    Sm.cx[hf][i] = c.c[0];
                    if (DIM == 3) Sm.cy[hf][i] = c.c[2];
                    Sm.tp[hf][i] = mid || !hf ? c.down() : c.up();  // coupling to the plane before (mid: below)
                    Sm.tn[hf][i] = mid || !hf ? c.up() : c.down();  // after (mid: above)
                    if (!mid)                                       // B's entries of the plane
                        plane_faces<DIM>(v, G, c, k, i,
                                         [&](int t, double rho) { Sm.Z[hf * cz + Sm.pos[hf * mp + t]][i] += (T)rho; });
                }
            }
            __syncwarp();
            T e[BlockSlots<GL>::kN];
#pragma unroll
            for (int s = 0; s < BlockSlots<GL>::kN; ++s) {
                e[s] = (T)0;
                if (!B.valid(s)) continue;
                const int r = B.row(s), c = B.colm(s);
                if (!act || r >= G.nb) continue;
                double x = plane_entry(G, Sm, hf, r, c);
                if (!mid) {
                    if (j > 0) x -= (double)Sm.P[hf][tri_at(r, c)] * (Sm.tp[hf][r] * Sm.tp[hf][c]);
                } else {
                    if (G.halfplanes(0) > 0) x -= (double)Sm.P[0][tri_at(r, c)] * (Sm.tp[0][r] * Sm.tp[0][c]);
                    if (G.halfplanes(1) > 0) x -= (double)Sm.P[1][tri_at(r, c)] * (Sm.tn[0][r] * Sm.tn[0][c]);
                }
                e[s] = (T)x;
            }
            __syncwarp();
            // lanes of absent or smaller blocks follow the longest one
            const int nb = act ? G.nb : 0;
            const int nbmax = __reduce_max_sync(0xffffffffu, nb);
            bad |= !sweep_block<GL, T>(e, B, Sm.col[hf], nb, nbmax, [](T p, int) { return positive_finite_bits(p); });
            if (act)
#pragma unroll
                for (int s = 0; s < BlockSlots<GL>::kN; ++s) {
                    if (!B.valid(s)) continue;
                    const int r = B.row(s), c = B.colm(s);
                    if (r < G.nb) Sm.P[hf][tri_at(r, c)] = neg_bits(e[s]);
                }
        }
        if (TM > 1) __syncthreads();
        leaf_sync<NW>();
        // ---- products, per leaf and half (loops kept rolled: one copy of the
        // code of a product, or the instruction fetch sets the pace)
#pragma unroll 1
        for (int fh = 0; fh < 2 * LPC; ++fh) {
            const int f = fh >> 1, h = fh & 1;
            const LeafGeo& g = geos[f];
            if (leaf0 + f >= v.nleaf || (mid ? h : j >= g.halfplanes(h))) continue;
            const LeafBuildSmem<DIM, T> s(smem_raw + (size_t)f * bytes, mp, cz);
            const int k = mid ? g.M : (h ? g.H - 1 - j : j), cc = mid ? g.m : g.cols(h, k);
            // Z of the plane by column, V = P Z, column -> segment
            T (*zs)[kPlane + 1] = mid ? s.V : s.Z + h * cz;
            T (*vs)[kPlane + 1] = mid ? s.Z : s.V;
            const short* ord = s.ord + h * mp;
            if (mid) {
                // Z of the middle plane: both halves' contributions and B
                for (int t = r16; t < g.m; t += NT / 16) {
                    const int pt = s.pos[t], pb = s.pos[mp + t];
                    T z = (T)0;
                    if (g.M > 0 && pt >= 0 && pt < g.cols(0, g.M - 1)) z += s.Z[pt][c16];
                    if (g.H - 1 - g.M > 0 && pb >= 0 && pb < g.cols(1, g.M + 1)) z += s.Z[cz + pb][c16];
                    s.V[t][c16] = z;
                }
                leaf_sync<NW>();
                for (int i = tid; i < g.nb; i += NT)
                    plane_faces<DIM>(v, g, cell_faces<DIM>(v, leaf0 + f, g, g.M, i), g.M, i,
                                     [&](int t, double rho) { s.V[t][i] += (T)rho; });
                leaf_sync<NW>();
            }
            {
                T* Lk = leaf_L<T>(v) + g.L_off + (long long)k * g.nb * g.nb;
                T* Zk = leaf_Z<T>(v) + g.Z_off + g.zoff(mid ? 0 : h, k);
                if (c16 < g.nb) {
                    for (int r = r16; r < g.nb; r += NT / 16) Lk[r * g.nb + c16] = s.P[h][tri_at(r, c16)];
                    for (int n = r16; n < cc; n += NT / 16) Zk[n * g.nb + c16] = zs[n][c16];
                }
            }
            // stage 0: V = P Z; stage 1: R += Z^T V, entries (row, n), row >= n, of
            // the column order; 16 x 8 tiles dealt to the warps
            // (P goes as P_kk^1/2 over k, Z as P_kk^-1/2, V as P_kk^1/2 again)
            int item = 0, sk[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) sk[i] = half_exponent(s.P[h][tri_at(frag_k(i), frag_k(i))]);
#pragma unroll 1
            for (int stage = 0; stage < 2; ++stage) {
                const int mt = stage ? (cc + 15) / 16 : 1;
#pragma unroll 1
                for (int ri = 0; ri < mt; ++ri) {
                    const int nt = stage ? min((cc + 7) / 8, 2 * ri + 2) : (cc + 7) / 8;
                    const int rows = stage ? min(cc - 16 * ri, 16) : g.nb;
                    FragA<S> a;
                    bool loaded = false;
#pragma unroll 1
                    for (int ni = 0; ni < nt; ++ni) {
                        if (NW > 1 && (item + ni) % NW != warp) continue;
                        if (!loaded) {
                            const T *zp = &zs[16 * ri][0], *pp = s.P[h];
                            load_frag_a<S, T>(a, sk, stage ? 1 : -1, [&](int r, int k) {
                                return r < rows ? (stage ? zp[r * (kPlane + 1) + k] : pp[tri_at(r, k)]) : (T)0;
                            });
                            loaded = true;
                        }
                        const T* bp = &(stage ? vs : zs)[8 * ni][0];
                        FragB<S> b;
                        load_frag_b<S, T>(
                            b, sk, stage ? -1 : 1, [&](int n, int k) { return 8 * ni + n < cc ? bp[n * (kPlane + 1) + k] : (T)0; });
                        typename SplitAcc<S>::T out[4];
                        frag_product(a, b, out, rows);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const int i = (lane >> 2) + 8 * (r >> 1), row = 16 * ri + i;
                            const int n = 8 * ni + 2 * (lane & 3) + (r & 1);
                            if (!stage) {
                                if (n < cc) vs[n][i] = (T)out[r];
                            } else if (row < cc && n <= row)
                                s.R[mid ? tri_at(row, n) : tri_at(ord[row], ord[n])] += (double)out[r];
                        }
                    }
                    item += nt;
                }
                leaf_sync<NW>();
            }
            if (mid) continue;
            // what the next plane receives: T V
            for (int p = r16; p < cc; p += NT / 16)
                zs[p][c16] = c16 < g.nb ? (T)(s.tn[h][c16] * (double)s.V[p][c16]) : (T)0;
            leaf_sync<NW>();
        }
    }
    if (bad) atomicOr(v.status, kStatusSingular);
    // R = Z^T P Z - W
#pragma unroll 1
    for (int f = 0; f < LPC; ++f) {
        if (leaf0 + f >= v.nleaf) break;
        const LeafGeo& g = geos[f];
        const LeafBuildSmem<DIM, T> s(smem_raw + (size_t)f * bytes, mp, cz);
        for (int t = tid; t < g.m; t += NT) s.R[t * (t + 1) / 2 + t] -= segment_rho_sum<DIM>(v, leaf0 + f, g, t);
        leaf_sync<NW>();
        double* Rg = v.R + g.R_off;
        for (int r = r16; r < g.m; r += NT / 16)
            for (int c = c16; c < g.m; c += 16) Rg[r * g.m + c] = s.R[tri_at(r, c)];
    }
}

// ---------------------------------------------------------------------------
// Solve phase, 2 PL lanes per leaf (one warp: PL = 16; four blocks per warp:
// PL = 4): lanes 0 .. PL - 1 the planes below the middle one (lane = cell), the
// others those above, in step; the middle plane by both (each half takes half
// of the products).  FP32 factors are widened by integer operations: a
// conversion holds the FP64 pipe like the FP64 multiply-add it feeds.
//
// PL = 4 serves 3D blocks whose planes have at most four cells, where most lanes
// of a warp per block idle (particular problems / pressures, ms a pass: 16384
// blocks of 1^3 0.075 / 0.042 -> 0.020 / 0.018, 4096 of 2^3 0.049 / 0.035 -> 0.024 /
// 0.025, 32768 of 2^3 0.293 / 0.180 -> 0.079 / 0.076; the kernels before the planes
// 0.053 / 0.030, 0.054 / 0.038, 0.352 / 0.208).
constexpr int kSolveWarps = 4;
template <int PL>
struct SolveLanes {
    int sg, gl, h, l;             // leaf of the warp, lane of the leaf, half, cell of the plane
    int leaf;
    bool on;                      // (past the last leaf the lanes follow it and store nothing)
    __device__ __forceinline__ SolveLanes(int warp_leaves0, int n) {
        const int lane = threadIdx.x & 31;
        sg = lane / (2 * PL);
        gl = lane % (2 * PL);
        h = gl / PL;
        l = gl % PL;
        leaf = warp_leaves0 + sg;
        on = leaf < n;
        leaf = min(leaf, n - 1);
    }
};

// Right-hand side of the particular problem at one cell (Eqs. addu/addp):
// the source plus Dirichlet and Neumann data of its domain-boundary faces.
template <int DIM>
__device__ __forceinline__ double particular_rhs(const DevView& v, int leaf, const CellFaces<DIM>& f,
                                                 const double* q, const double* bc_val) {
    double b = q[f.cell];
    if (!bc_val) return b;
    if constexpr (DIM == 2) {
        const GridDesc& G = v.grids[v.leaves[leaf].grid];
        const double* bv = bc_val + G.b0;
        if (f.x == 0) b += G.bc[0] ? f.c[0] * bv[f.y] : -G.hy * bv[f.y];
        if (f.x == G.nx - 1) b += G.bc[1] ? f.c[1] * bv[G.ny + f.y] : -G.hy * bv[G.ny + f.y];
        if (f.y == 0) b += G.bc[2] ? f.c[2] * bv[2 * G.ny + f.x] : -G.hx * bv[2 * G.ny + f.x];
        if (f.y == G.ny - 1) {
            const double g = bv[2 * G.ny + G.nx + f.x];
            b += G.bc[3] ? f.c[3] * g : -G.hx * g;
        }
    } else {
        const Grid3& G = v.g3;
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            const int pos = s < 2 ? f.x : (s < 4 ? f.y : f.z), n = s < 2 ? G.nx : (s < 4 ? G.ny : G.nz);
            if (s & 1 ? pos != n - 1 : pos != 0) continue;
            const double g = bc_value3(G, bc_val, s, f.x, f.y, f.z);
            b += G.bc[s] ? f.c[s] * g : -(area3(G, s >> 1) * g);
        }
    }
    return b;
}

// Column l of the stored P of plane k (P is symmetric: entry j is P(l, j)).
template <int PL, class TS>
__device__ __forceinline__ void load_p(TS (&p)[PL], const TS* Lg, int nb, int k, int l, bool on) {
    const TS* c = Lg + (long long)k * nb * nb + l;
#pragma unroll
    for (int j = 0; j < PL; ++j) p[j] = (on && l < nb && j < nb) ? c[j * nb] : (TS)0;
}
// sum_j p[j] y[j], and column l of plane k in p's place: each entry is loaded
// as soon as the one before it is used, a plane ahead of its own use.  One
// chain: its latency (75 cycles) is little above what an FP64 instruction
// holds the pipe for, and partial sums would only add to it.
template <int PL, class TS>
__device__ __forceinline__ double row_product_next(TS (&p)[PL], const double* y, const TS* Lg, int nb, int k, int l,
                                                   bool on) {
    const TS* c = Lg + (long long)k * nb * nb + l;
    const int n = on && l < nb ? nb : 0;
    double a = 0.0;
#pragma unroll
    for (int j = 0; j < PL; ++j) {
        a = fma(widen(p[j]), y[j], a);
        p[j] = j < n ? c[j * nb] : (TS)0;
    }
    return a;
}
// the half of the product over j in [PL / 2 part, PL / 2 (part + 1))
template <int PL, class TS>
__device__ __forceinline__ double half_product(const TS (&p)[PL], const double* y, int part) {
    double a = 0.0;
#pragma unroll
    for (int j = 0; j < PL / 2; ++j) a = fma(widen(part ? p[j + PL / 2] : p[j]), y[j + part * (PL / 2)], a);
    return a;
}

// Sums x[c], c < 8, over the 16 lanes of each half warp; lane l returns
// column l / 2 (both lanes of a pair the same).
__device__ __forceinline__ double reduce_columns8(double (&x)[8], int l) {
#pragma unroll
    for (int w = 8, n = 4; w >= 2; w >>= 1, n >>= 1) {
        const bool up = l & w;
#pragma unroll
        for (int c = 0; c < n; ++c) {
            const double mine = up ? x[c + n] : x[c], theirs = up ? x[c] : x[c + n];
            x[c] = mine + __shfl_xor_sync(0xffffffffu, theirs, w);
        }
    }
    return x[0] + __shfl_xor_sync(0xffffffffu, x[0], 1);
}

// y_k (into leafzb), w_k = P_k y_k and rbar = sum_k Z_k^T w_k.  SMALL: at most
// 8 columns meet a plane off the middle one and m <= 16 (partial sums in
// registers; PL = 16 only); otherwise they go through shared memory (acc: (2 cz +
// mp) rows of PL + 1 doubles per leaf).  TS: storage type of the factors (float in the
// mixed form's FP32 leaves); the arithmetic is FP64.
template <int DIM, class TS, bool SMALL, int PL>
__global__ void __launch_bounds__(32 * kSolveWarps)
leaf_particular_kernel(DevView v, const double* __restrict__ q, const double* __restrict__ bc_val, bool with_sadj,
                       int mp, int cz) {
    static_assert(!SMALL || PL == 16, "partial sums in registers over 16 lanes");
    __shared__ double ysh_all[kSolveWarps][32];
    extern __shared__ __align__(16) double acc_raw[];
    constexpr int kLeaves = 16 / PL;                  // leaves per warp
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int first = (blockIdx.x * kSolveWarps + warp) * kLeaves;
    if (first >= v.nleaf) return;                     // uniform over the warp
    const SolveLanes<PL> q4(first, v.nleaf);
    const int h = q4.h, l = q4.l, leaf = q4.leaf;
    double* ysh = ysh_all[warp] + (2 * q4.sg + h) * PL;   // y of the lane's plane
    const LeafGeo g = leaf_geo<DIM>(v, leaf);
    const int nb = g.nb, hp = g.halfplanes(h);
    int steps = max(g.halfplanes(0), g.halfplanes(1));
    if (kLeaves > 1) steps = __reduce_max_sync(0xffffffffu, steps);
    const TS* Lg = leaf_L<TS>(v) + g.L_off;
    const TS* Zg = leaf_Z<TS>(v) + g.Z_off;
    double* zb = v.leafzb + g.zb_off;
    double (*acc)[PL + 1] =
        reinterpret_cast<double (*)[PL + 1]>(acc_raw) + (size_t)(warp * kLeaves + q4.sg) * (2 * cz + mp);
    double part[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) part[p] = 0.0;
    if constexpr (!SMALL)
        for (int p = 0; p < cz; ++p) acc[h * cz + p][l] = 0.0;
    TS p[PL];
    double w = 0.0, yn = 0.0, tn = 0.0;
    // right-hand side and coupling to the plane before, a plane ahead
    auto ahead = [&](int j) {
        if (j >= hp || l >= nb) return;
        const CellFaces<DIM> f = cell_faces<DIM>(v, leaf, g, h ? g.H - 1 - j : j, l);
        yn = particular_rhs<DIM>(v, leaf, f, q, bc_val);
        tn = h ? f.up() : f.down();
    };
    ahead(0);
    load_p(p, Lg, nb, h ? g.H - 1 : 0, l, hp > 0);
    const int ccw = __reduce_max_sync(0xffffffffu, g.ncols(h));    // columns of the warp's widest plane
    for (int j = 0; j < steps; ++j) {
        const bool act = j < hp && l < nb;
        const int k = h ? g.H - 1 - j : j;
        const double y = act ? (j > 0 ? fma(tn, w, yn) : yn) : 0.0;
        if (act && q4.on) zb[k * nb + l] = y;
        const int cc = j < hp ? g.cols(h, k) : 0;
        const TS* Zk = Zg + g.zoff(h, k);
        TS z[8];
        if (SMALL)
#pragma unroll
            for (int c = 0; c < 8; ++c) z[c] = act && c < cc ? Zk[c * nb + l] : (TS)0;
        ysh[l] = y;
        __syncwarp();
        ahead(j + 1);
        const double wn = row_product_next(p, ysh, Lg, nb, h ? k - 1 : k + 1, l, j + 1 < hp);
        if (act) w = wn;
        if (SMALL) {
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c < ccw) part[c] = fma(widen(z[c]), wn, part[c]);
        } else {
            for (int c = 0; c < cc; ++c)
                acc[h * cz + c][l] = fma(act ? widen(Zk[c * nb + l]) : 0.0, wn, acc[h * cz + c][l]);
        }
        __syncwarp();
    }
    // the middle plane
    {
        load_p(p, Lg, nb, g.M, l, true);
        const double other = __shfl_xor_sync(0xffffffffu, w, PL);
        const double wt = h ? other : w, wb = h ? w : other;       // (0 for a half without planes)
        double y = 0.0;
        if (l < nb) {
            const CellFaces<DIM> f = cell_faces<DIM>(v, leaf, g, g.M, l);
            y = particular_rhs<DIM>(v, leaf, f, q, bc_val);
            if (g.halfplanes(0) > 0) y = fma(f.down(), wt, y);
            if (g.halfplanes(1) > 0) y = fma(f.up(), wb, y);
            if (h == 0 && q4.on) zb[g.M * nb + l] = y;
        }
        ysh[l] = y;
        __syncwarp();
        w = half_product(p, ysh, h);
        w += __shfl_xor_sync(0xffffffffu, w, PL);
    }
    const TS* Zm = Zg + g.zoff(0, g.M);
    double* rb = v.rbar + g.r_off;
    auto store = [&](int t, double x) {
        // a right-hand side sigma on this segment's interface row,
        // F - D (lambda_other - lambda_own) = sigma, acts as rbar - sigma
        if (q4.on) rb[t] = with_sadj ? x - v.sadj[g.r_off + t] : x;
    };
    if constexpr (SMALL) {
        // columns 8 h + c of the middle plane
        double zm[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int t = 8 * h + c;
            zm[c] = l < nb && t < g.m ? widen(Zm[t * nb + l]) * w : 0.0;
        }
        double* rs = ysh_all[warp];                                // rbar by segment (m <= 16)
        const double r = reduce_columns8(zm, l);
        __syncwarp();
        if (!(l & 1) && 8 * h + (l >> 1) < g.m) rs[8 * h + (l >> 1)] = r;
        __syncwarp();
        const double o = reduce_columns8(part, l);
        for (int s = 0; s < 2; ++s) {
            if (h == s && !(l & 1) && (l >> 1) < g.ncols(s)) rs[g.segment(s, l >> 1)] += o;
            __syncwarp();
        }
        if (lane < g.m) store(lane, rs[lane]);
        return;
    }
    for (int t = h; t < g.m; t += 2) acc[2 * cz + t][l] = l < nb ? widen(Zm[t * nb + l]) * w : 0.0;
    __syncwarp();
    // each row summed by one lane (over the cells), then the halves' rows
    // added to their segments
    for (int p = q4.gl; p < 2 * cz + g.m; p += 2 * PL) {
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int c = 0; c < PL; c += 2) {
            s0 += acc[p][c];
            s1 += acc[p][c + 1];
        }
        acc[p][0] = s0 + s1;
    }
    __syncwarp();
    for (int s = 0; s < 2; ++s) {
        for (int p = q4.gl; p < g.ncols(s); p += 2 * PL) acc[2 * cz + g.segment(s, p)][0] += acc[s * cz + p][0];
        __syncwarp();
    }
    for (int t = q4.gl; t < g.m; t += 2 * PL) store(t, acc[2 * cz + t][0]);
}

// x = A^-1 (A-elimination's right-hand sides), from the middle plane outwards;
// rhs(h, k, l, Zk, cc): y_k + Z_k lambda at cell l (h < 0: the middle plane,
// where each half of the lanes returns its share), out(k, l, x); ysh: PL doubles
// of the lane's leaf and half.
template <int DIM, int PL, class TS, class Rhs, class Out>
__device__ __forceinline__ void solve_outward(const DevView& v, const SolveLanes<PL>& q4, const LeafGeo& g,
                                              const TS* Lg, double* ysh, Rhs&& rhs, Out&& out) {
    const int h = q4.h, l = q4.l, nb = g.nb, hp = g.halfplanes(h), leaf = q4.leaf;
    int steps = max(g.halfplanes(0), g.halfplanes(1));
    if (PL < 16) steps = __reduce_max_sync(0xffffffffu, steps);
    TS p[PL];
    double x, tn = 0.0;
    auto ahead = [&](int d) {                                      // coupling to the plane before, a plane ahead
        if (d > hp || l >= nb) return;
        const CellFaces<DIM> f = cell_faces<DIM>(v, leaf, g, h ? g.M + d : g.M - d, l);
        tn = h ? f.down() : f.up();
    };
    ahead(1);
    {
        TS pm[PL];
        load_p(pm, Lg, nb, g.M, l, true);
        load_p(p, Lg, nb, h ? g.M + 1 : g.M - 1, l, hp > 0);
        double y = rhs(-1, g.M, l);
        y += __shfl_xor_sync(0xffffffffu, y, PL);
        ysh[l] = y;
        __syncwarp();
        x = half_product(pm, ysh, h);
        x += __shfl_xor_sync(0xffffffffu, x, PL);
        __syncwarp();
        if (h == 0 && l < nb && q4.on) out(g.M, l, x);
    }
    double r = steps > 0 && hp > 0 ? rhs(h, h ? g.M + 1 : g.M - 1, l) : 0.0;
    for (int d = 1; d <= steps; ++d) {
        const bool act = d <= hp;
        const int k = h ? g.M + d : g.M - d;
        ysh[l] = act && l < nb ? fma(tn, x, r) : 0.0;
        __syncwarp();
        ahead(d + 1);
        const double xn = row_product_next(p, ysh, Lg, nb, h ? k + 1 : k - 1, l, d + 1 <= hp);
        if (d + 1 <= hp) r = rhs(h, h ? k + 1 : k - 1, l);         // the next plane's
        if (act) x = xn;
        if (act && l < nb && q4.on) out(k, l, x);
        __syncwarp();
    }
}

// Final pressures p = A^-1 (bbar + B lambda), written into the state (p_hi,
// p_lo) or added to it in double-double (refinement corrections).
template <int DIM, class TS, int PL>
__global__ void __launch_bounds__(32 * kSolveWarps) leaf_pressure_kernel(DevView v, bool accumulate, int mp, int cz) {
    __shared__ double ysh[kSolveWarps][32];
    extern __shared__ __align__(16) double lam_raw[];              // per leaf: lambda in the halves' orders
    constexpr int kLeaves = 16 / PL;                               // leaves per warp
    const int warp = threadIdx.x >> 5, first = (blockIdx.x * kSolveWarps + warp) * kLeaves;
    if (first >= v.nleaf) return;                                  // uniform over the warp
    const SolveLanes<PL> q4(first, v.nleaf);
    const int leaf = q4.leaf;
    const LeafGeo g = leaf_geo<DIM>(v, leaf);
    double* lam = lam_raw + (size_t)(warp * kLeaves + q4.sg) * (2 * cz + mp);
    for (int t = q4.gl; t < g.m; t += 2 * PL) lam[2 * cz + t] = v.lam[g.r_off + t];
    __syncwarp();
    for (int s = 0; s < 2; ++s)
        for (int p = q4.gl; p < g.ncols(s); p += 2 * PL) lam[s * cz + p] = lam[2 * cz + g.segment(s, p)];
    __syncwarp();
    const TS* Zg = leaf_Z<TS>(v) + g.Z_off;
    const double* zb = v.leafzb + g.zb_off;
    const int nb = g.nb;
    auto rhs = [&](int h, int k, int l) -> double {
        const bool mid = h < 0;
        const int half = q4.h, cc = mid ? g.m : g.cols(h, k), step = mid ? 2 : 1;
        const TS* Zk = Zg + g.zoff(mid ? 0 : h, k) + l;
        const double* lm = lam + (mid ? 2 * cz : h * cz);
        if (l >= nb) return 0.0;
        double a = mid && half ? 0.0 : zb[k * nb + l];
        int c = mid ? half : 0;
        for (; c + 7 * step < cc; c += 8 * step) {                 // eight loads in flight
            TS z[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) z[u] = Zk[(c + u * step) * nb];
#pragma unroll
            for (int u = 0; u < 8; ++u) a = fma(widen(z[u]), lm[c + u * step], a);
        }
        TS z[8];
#pragma unroll
        for (int u = 0; u < 7; ++u) z[u] = c + u * step < cc ? Zk[(c + u * step) * nb] : (TS)0;
#pragma unroll
        for (int u = 0; u < 7; ++u)
            if (c + u * step < cc) a = fma(widen(z[u]), lm[c + u * step], a);
        return a;
    };
    double* ys = ysh[warp] + (2 * q4.sg + q4.h) * PL;
    solve_outward<DIM, PL, TS>(v, q4, g, leaf_L<TS>(v) + g.L_off, ys, rhs, [&](int k, int l, double x) {
        long long c;
        if constexpr (DIM == 2) {
            const LeafDesc& L = v.leaves[leaf];
            const GridDesc& G = v.grids[L.grid];
            c = G.c0 + (long long)(L.j0 + k) * G.nx + L.i0 + l;
        } else {
            const LeafDesc3& L = v.leaves3[leaf];
            c = cell3(v.g3, L.i0 + l % g.w0, L.j0 + l / g.w0, L.k0 + k);
        }
        if (accumulate) {
            const DD s = dd_add_d(DD{v.p_hi[c], v.p_lo[c]}, x);
            v.p_hi[c] = s.h;
            v.p_lo[c] = s.l;
        } else {
            v.p_hi[c] = x;
            v.p_lo[c] = 0.0;
        }
    });
}

// Training targets of the learned surrogate: psi[item][k][s] (float; cell
// k = i + 16 j, segment s fastest) = A^-1 B e_s of the leaves ids[item], from
// the stored factors.
template <class TS>
__global__ void __launch_bounds__(32 * kSolveWarps) leaf_fields_kernel(DevView v, const int* __restrict__ ids,
                                                                      int count, float* __restrict__ psi) {
    __shared__ double ysh[kSolveWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int item = blockIdx.x * kSolveWarps + warp;
    if (item >= count) return;                                     // uniform over the warp
    const int id = ids[item];
    if ((unsigned)id >= (unsigned)v.nleaf || v.leaves[id].m > 16) {
        if (lane == 0) atomicOr(v.status, kStatusBadIndex);
        return;
    }
    const LeafGeo g = leaf_geo<2>(v, id);
    const SolveLanes<16> q4(id, v.nleaf);
    const TS* Zg = leaf_Z<TS>(v) + g.Z_off;
    const int nb = g.nb;
    for (int s = 0; s < g.m; ++s) {
        int pos[2] = {-1, -1};
        for (int h = 0; h < 2; ++h)
            for (int p = 0; p < g.ncols(h); ++p)
                if (g.segment(h, p) == s) pos[h] = p;
        auto rhs = [&](int h, int k, int l) -> double {
            if (l >= nb) return 0.0;
            if (h < 0) return lane < 16 ? widen(Zg[g.zoff(0, k) + s * nb + l]) : 0.0;
            return pos[h] >= 0 && pos[h] < g.cols(h, k) ? widen(Zg[g.zoff(h, k) + pos[h] * nb + l]) : 0.0;
        };
        double* ys = ysh[warp] + q4.h * 16;
        solve_outward<2, 16, TS>(v, q4, g, leaf_L<TS>(v) + g.L_off, ys, rhs, [&](int k, int l, double x) {
            psi[((long long)item * 256 + k * nb + l) * 16 + s] = (float)x;
        });
    }
}

constexpr int kRedBlocks = 256;

__global__ void mean_partial_kernel(const double* __restrict__ ph, const double* __restrict__ pl, long long n,
                                    double* red) {
    __shared__ double sh[256];
    double acc = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        acc += ph[i] + pl[i];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) red[blockIdx.x] = sh[0];
}

// Subtracts the mean of the rounded cell pressures from p and P, in
// double-double (the shift is exact up to its own rounding).
template <bool kPlain>
__global__ void mean_subtract_kernel(DevView v, long long n) {
    __shared__ double mean;
    if (threadIdx.x < 32) {
        // fixed-order warp reduction of the block partial sums: every block
        // obtains the identical mean
        double acc = 0.0;
        for (int b = threadIdx.x; b < kRedBlocks; b += 32) acc += v.red[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) mean = acc / (double)n;
    }
    __syncthreads();
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (kPlain) {
        // no low parts: shift the high parts
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += stride) v.p_hi[i] -= mean;
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < v.nseg; i += stride) {
            v.segP[i] -= mean;
            v.seg_lam_dd[2 * i].x -= mean;
            v.seg_lam_dd[2 * i + 1].x -= mean;
        }
        return;
    }
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += stride) {
        const DD x = dd_add(DD{v.p_hi[i], v.p_lo[i]}, DD{-mean, 0.0});
        v.p_hi[i] = x.h;
        v.p_lo[i] = x.l;
    }
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < v.nseg; i += stride) {
        const DD x = dd_add(DD{v.segP[i], v.segP_lo[i]}, DD{-mean, 0.0});
        v.segP[i] = x.h;
        v.segP_lo[i] = x.l;
        // the Robin data P -/+ beta U move with P
        for (int side = 0; side < 2; ++side) {
            const double2 l = v.seg_lam_dd[2 * i + side];
            const DD y = dd_add(DD{l.x, l.y}, DD{-mean, 0.0});
            v.seg_lam_dd[2 * i + side] = make_double2(y.h, y.l);
        }
    }
}

template <int DIM, class T, int NW, int LPC, int TM = 1>
cudaError_t build_launch(const DevView& v, int mp, int cz, cudaStream_t s) {
    const int bytes = (int)LeafBuildSmem<DIM, T>::bytes(mp, cz), per = LPC * TM;
    auto* kern = leaf_build_kernel<DIM, T, NW, LPC, TM>;
    // set on every launch (a host call; the attribute belongs to the current device)
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes * per);
    if (e != cudaSuccess) return e;
    kern<<<(v.nleaf + per - 1) / per, 32 * NW * TM, bytes * per, s>>>(v, mp, cz, bytes);
    return cudaGetLastError();
}
template <int DIM, class T>
cudaError_t build_dispatch(const DevView& v, int mp, int cz, cudaStream_t s) {
    // 2D leaves of up to 16 segments: one warp per two leaves (the FP64
    // instructions of the inversions serve four blocks: a quarter fewer per
    // leaf), one leaf per warp for fewer, and four warps to a leaf where not even
    // that fills the schedulers.  Waves are 1824 leaves one per warp, 3648 two
    // per warp; 16 x 16 leaves, ms four warps / one / two leaves per warp: 160
    // 0.201 / 0.199 / 0.351, 304 0.204 / 0.199 / 0.354, 800 0.417 / 0.245 / 0.355,
    // 1824 0.71 / 0.307 / 0.439, 2432 0.96 / 0.477 / 0.443, 3648 1.46 / 0.603 /
    // 0.542, 4096 1.63 / 0.750 / 0.844, 4864 1.93 / 0.820 / 0.851, 6000 2.38 / 1.033 /
    // 0.951, 12000 4.74 / 1.96 / 1.85.  The line lies past the one-per-warp
    // form's third wave; between its first and its second the other form would
    // be up to 10% shorter.  More segments: four warps per leaf share the
    // products.
    if (DIM == 2 && mp <= 16) {
        if (v.nleaf <= kRuleSMs * 2) return build_launch<2, T, 4, 1>(v, mp, cz, s);
        if (v.nleaf <= kRuleSMs * 32) return build_launch<2, T, 1, 1, kTeams>(v, mp, cz, s);
        return build_launch<2, T, 1, 2, kTeams>(v, mp, cz, s);
    }
    return build_launch<DIM, T, 4, 1>(v, mp, cz, s);
}
template <int DIM, class TS, bool SMALL, int PL>
cudaError_t particular_go(const DevView& v, const double* q, const double* bc_val, bool with_sadj, int mp, int cz,
                          cudaStream_t s) {
    constexpr int per = kSolveWarps * (16 / PL);
    const int bytes = SMALL ? 0 : (int)sizeof(double) * per * (2 * cz + mp) * (PL + 1);
    auto* kern = leaf_particular_kernel<DIM, TS, SMALL, PL>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    kern<<<(v.nleaf + per - 1) / per, 32 * kSolveWarps, bytes, s>>>(v, q, bc_val, with_sadj, mp, cz);
    return cudaGetLastError();
}
// Planes of at most four cells (3D): four blocks per warp, as long as their
// partial sums fit in shared memory.
bool narrow_planes(const DevView& v, int mp, int cz) {
    return v.nb3 <= 4 && (size_t)kSolveWarps * 4 * (2 * cz + mp) * 5 * sizeof(double) <= 200 * 1024;
}
template <int DIM, class TS>
cudaError_t particular_launch(const DevView& v, const double* q, const double* bc_val, bool with_sadj, int mp, int cz,
                              cudaStream_t s) {
    if (DIM == 3 && narrow_planes(v, mp, cz))
        return particular_go<DIM, TS, false, DIM == 3 ? 4 : 16>(v, q, bc_val, with_sadj, mp, cz, s);
    if (cz <= 8 && mp <= 16) return particular_go<DIM, TS, true, 16>(v, q, bc_val, with_sadj, mp, cz, s);
    return particular_go<DIM, TS, false, 16>(v, q, bc_val, with_sadj, mp, cz, s);
}
template <int DIM, class TS, int PL>
cudaError_t pressure_go(const DevView& v, bool accumulate, int mp, int cz, cudaStream_t s) {
    constexpr int per = kSolveWarps * (16 / PL);
    const int bytes = (int)sizeof(double) * per * (2 * cz + mp);
    auto* kern = leaf_pressure_kernel<DIM, TS, PL>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    kern<<<(v.nleaf + per - 1) / per, 32 * kSolveWarps, bytes, s>>>(v, accumulate, mp, cz);
    return cudaGetLastError();
}
template <int DIM, class TS>
cudaError_t pressure_launch(const DevView& v, bool accumulate, int mp, int cz, cudaStream_t s) {
    if (DIM == 3 && narrow_planes(v, mp, cz)) return pressure_go<DIM, TS, DIM == 3 ? 4 : 16>(v, accumulate, mp, cz, s);
    return pressure_go<DIM, TS, 16>(v, accumulate, mp, cz, s);
}

}  // namespace

cudaError_t launch_leaf_build(const DevView& v, int max_m, int max_c, cudaStream_t s) {
    const int mp = std::max(max_m, 1), cz = std::max(max_c, 1);
    if (v.dim == 3) return build_dispatch<3, double>(v, mp, cz, s);
    if (v.banded) return launch_banded_build(v, max_m, s);
    return v.leaf32 ? build_dispatch<2, float>(v, mp, cz, s) : build_dispatch<2, double>(v, mp, cz, s);
}

cudaError_t launch_leaf_particular(const DevView& v, const double* q, const double* bc_val, bool with_sadj, int max_m,
                                   int max_c, cudaStream_t s) {
    const int mp = std::max(max_m, 1), cz = std::max(max_c, 1);
    if (v.dim == 3) return particular_launch<3, double>(v, q, bc_val, with_sadj, mp, cz, s);
    if (v.banded) return launch_banded_particular(v, q, bc_val, with_sadj, s);
    return v.leaf32 ? particular_launch<2, float>(v, q, bc_val, with_sadj, mp, cz, s)
                    : particular_launch<2, double>(v, q, bc_val, with_sadj, mp, cz, s);
}

cudaError_t launch_leaf_pressure(const DevView& v, bool accumulate, int max_m, int max_c, cudaStream_t s) {
    const int mp = std::max(max_m, 1), cz = std::max(max_c, 1);
    if (v.dim == 3) return pressure_launch<3, double>(v, accumulate, mp, cz, s);
    if (v.banded) return launch_banded_pressure(v, accumulate, s);
    return v.leaf32 ? pressure_launch<2, float>(v, accumulate, mp, cz, s)
                    : pressure_launch<2, double>(v, accumulate, mp, cz, s);
}

cudaError_t launch_leaf_fields(const DevView& v, const int* ids, int count, float* psi, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    if (v.banded) return launch_banded_fields(v, ids, count, psi, s);
    const int grid = (count + kSolveWarps - 1) / kSolveWarps;
    if (v.leaf32) leaf_fields_kernel<float><<<grid, 32 * kSolveWarps, 0, s>>>(v, ids, count, psi);
    else leaf_fields_kernel<double><<<grid, 32 * kSolveWarps, 0, s>>>(v, ids, count, psi);
    return cudaGetLastError();
}

cudaError_t launch_mean_shift(const DevView& v, bool plain, cudaStream_t s) {
    const long long n = v.ncell;      // all-Neumann problems: single-grid contexts only
    mean_partial_kernel<<<kRedBlocks, 256, 0, s>>>(v.p_hi, v.p_lo, n, v.red);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (plain)
        mean_subtract_kernel<true><<<kRedBlocks, 256, 0, s>>>(v, n);
    else
        mean_subtract_kernel<false><<<kRedBlocks, 256, 0, s>>>(v, n);
    return cudaGetLastError();
}

}  // namespace mrcm
