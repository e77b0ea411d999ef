// The matrix products of the blocked merges on the tensor cores (the split
// products of split_gemm.cuh): X = -W C and the merged map R = R_oo + C^T X
// of every node of a tree height (Eqs. new_bfs.1-2; kernels_merge.cu has the
// derivation and the launches around these).
#include "block_invert.cuh"
#include "merge_common.cuh"
#include "split_gemm.cuh"
#include "tc_split.cuh"

#include <algorithm>

namespace mrcm {
namespace {

// X = -W blockdiag(R^a_go, R^b_go): column j < o1 uses the first g columns
// of W and child a's map, the others the last g and child b's, so the tiles
// of X's columns are cut on either side of o1.  W is symmetric: its row r is
// read as column r, contiguous in k, and the map of a child is symmetric:
// column j of C is read along the map's row of that segment.
//
// Powers of two of the two products: column k of W (and row k of X) goes as
// D_k^-1/2, row k of C as D_k^1/2, D the Robin coefficient of the segment.
struct GammaScale {
    const double* sq;                      // D^1/2 of the node's gamma segments
    int sign;
    __device__ __forceinline__ int operator()(int k) const { return sign * whole_exponent(sq[k]); }
};
template <int S>
__global__ void __launch_bounds__(kGemmThreads, 2) merge_x_kernel(DevView v, int first) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SplitSmem<S>& sm = *reinterpret_cast<SplitSmem<S>*>(smem_raw);
    const MergeDesc D = v.merges[first + blockIdx.x];
    const NodeRefs N = node_refs(v, D);
    const int g = N.g, g2 = N.g2, m = N.m;
    const int rt = (g2 + kTileM - 1) / kTileM;
    const int na = (N.o1 + kTileN - 1) / kTileN, nb = (m - N.o1 + kTileN - 1) / kTileN;
    if ((int)blockIdx.y >= rt * (na + nb)) return;                     // uniform per CTA
    const int r0 = (blockIdx.y % rt) * kTileM, ct = blockIdx.y / rt;
    const bool half = ct >= na;
    const int j0 = half ? N.o1 + (ct - na) * kTileN : ct * kTileN, jend = half ? m : N.o1;
    const double* W = v.W + D.W_off + (half ? g : 0);
    const double* Rc = half ? N.R2 : N.R1;
    const int* gpos = half ? N.gpos2 : N.gpos1;
    const int* opos = half ? N.opos2 - N.o1 : N.opos1;
    const int mc = half ? N.m2 : N.m1;
    typename SplitAcc<S>::T sum[2][4];
    split_product<S, double, false, true>(
        sm, g, gpos, [&](int r) { return r0 + r < g2 ? W + (long long)(r0 + r) * g2 : nullptr; },
        [&](int j) { return j0 + j < jend ? Rc + (long long)opos[j0 + j] * mc : nullptr; },
        GammaScale{v.gam_sq + D.gamma_off, 1}, sum);
    double* X = v.X + D.X_off;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = r0 + out_row(mt, q), j = j0 + out_col(q);
            if (r < g2 && j < jend) X[(long long)j * g2 + r] = neg_bits(widen(sum[mt][q]));
        }
}

// R = blockdiag(R^a_oo, R^b_oo) + blockdiag(R^a_og, R^b_og) X, lower triangle
// formed and mirrored (R is symmetric).  Tiles of 64 rows cut on either side
// of o1 (a row uses its child's map and that child's half of X) by 32
// columns up to the diagonal.
template <int S>
__global__ void __launch_bounds__(kGemmThreads, 2) merge_rupdate_kernel(DevView v, int first, int coltiles) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SplitSmem<S>& sm = *reinterpret_cast<SplitSmem<S>*>(smem_raw);
    const MergeDesc D = v.merges[first + blockIdx.x];
    const NodeRefs N = node_refs(v, D);
    const int g = N.g, g2 = N.g2, m = N.m, o1 = N.o1;
    const int na = (o1 + kTileM - 1) / kTileM, nb = (m - o1 + kTileM - 1) / kTileM;
    const int rt = blockIdx.y / coltiles, j0 = (blockIdx.y % coltiles) * kTileN;
    if (rt >= na + nb) return;                                          // uniform per CTA
    const bool half = rt >= na;
    const int i0 = half ? o1 + (rt - na) * kTileM : rt * kTileM, iend = min(i0 + kTileM, half ? m : o1);
    if (j0 >= iend) return;                                             // uniform per CTA
    const double* X = v.X + D.X_off + (half ? g : 0);
    const double* Rc = half ? N.R2 : N.R1;
    const int* gpos = half ? N.gpos2 : N.gpos1;
    const int* opos = half ? N.opos2 - o1 : N.opos1;
    const int mc = half ? N.m2 : N.m1;
    typename SplitAcc<S>::T sum[2][4];
    split_product<S, double, true, false>(
        sm, g, gpos, [&](int i) { return i0 + i < iend ? Rc + (long long)opos[i0 + i] * mc : nullptr; },
        [&](int j) { return j0 + j < m ? X + (long long)(j0 + j) * g2 : nullptr; },
        GammaScale{v.gam_sq + D.gamma_off, -1}, sum);
    double* Rp = v.R + D.R_off;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + out_row(mt, q), j = j0 + out_col(q);
            if (i >= iend || j > i) continue;
            double val = widen(sum[mt][q]);
            if (half == (j >= o1)) val += Rc[(long long)opos[i] * mc + opos[j]];   // both on one child
            Rp[(long long)i * m + j] = val;
            Rp[(long long)j * m + i] = val;
        }
}

// The same products where g <= kChunkK and the level has CTAs enough: one CTA
// per 64 rows of X and child, and per 64 rows of R, over all their column
// tiles (the digits of the rows are cut once and a tile's loads hide behind
// the products before it: box 128x128x64 R of 2g <= 128 6.0 -> 3.9 ms, the mixed
// 256x256x64 box 20 -> 8).
template <int S>
__global__ void __launch_bounds__(kGemmThreads, 2) merge_x_strip_kernel(DevView v, int first) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SplitSmem<S>& sm = *reinterpret_cast<SplitSmem<S>*>(smem_raw);
    const MergeDesc D = v.merges[first + blockIdx.x];
    const NodeRefs N = node_refs(v, D);
    const int g = N.g, g2 = N.g2, m = N.m, r0 = (blockIdx.y >> 1) * kTileM;
    const bool half = blockIdx.y & 1;
    const int jbeg = half ? N.o1 : 0, jend = half ? m : N.o1;
    if (r0 >= g2 || jbeg >= jend) return;                              // uniform per CTA
    const double* W = v.W + D.W_off + (half ? g : 0);
    const double* Rc = half ? N.R2 : N.R1;
    const int* opos = half ? N.opos2 - N.o1 : N.opos1;
    const int mc = half ? N.m2 : N.m1;
    double* X = v.X + D.X_off;
    strip_product<S, false, true>(
        sm, g, half ? N.gpos2 : N.gpos1, 0, (jend - jbeg + kTileN - 1) / kTileN,
        [&](int r) { return r0 + r < g2 ? W + (long long)(r0 + r) * g2 : nullptr; },
        [&](int t, int c) {
            const int j = jbeg + t * kTileN + c;
            return j < jend ? Rc + (long long)opos[j] * mc : nullptr;
        },
        GammaScale{v.gam_sq + D.gamma_off, 1}, [](int, int, int) { return 0.0; },
        [&](int t, int i, int c, double x, double) {
            const int r = r0 + i, j = jbeg + t * kTileN + c;
            if (r < g2 && j < jend) X[(long long)j * g2 + r] = neg_bits(x);
        });
}
template <int S>
__global__ void __launch_bounds__(kGemmThreads, 2) merge_rupdate_strip_kernel(DevView v, int first) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SplitSmem<S>& sm = *reinterpret_cast<SplitSmem<S>*>(smem_raw);
    const MergeDesc D = v.merges[first + blockIdx.x];
    const NodeRefs N = node_refs(v, D);
    const int g = N.g, g2 = N.g2, m = N.m, o1 = N.o1;
    const int na = (o1 + kTileM - 1) / kTileM, nb = (m - o1 + kTileM - 1) / kTileM;
    if ((int)blockIdx.y >= na + nb) return;                             // uniform per CTA
    const int rt = na + nb - 1 - blockIdx.y;                            // long rows first
    const bool half = rt >= na;
    const int i0 = half ? o1 + (rt - na) * kTileM : rt * kTileM, iend = min(i0 + kTileM, half ? m : o1);
    const double* X = v.X + D.X_off + (half ? g : 0);
    const double* Rc = half ? N.R2 : N.R1;
    const int* opos = half ? N.opos2 - o1 : N.opos1;
    const int mc = half ? N.m2 : N.m1;
    double* Rp = v.R + D.R_off;
    strip_product<S, true, false>(
        sm, g, half ? N.gpos2 : N.gpos1, 0, (iend + kTileN - 1) / kTileN,
        [&](int i) { return i0 + i < iend ? Rc + (long long)opos[i0 + i] * mc : nullptr; },
        [&](int t, int c) { return t * kTileN + c < m ? X + (long long)(t * kTileN + c) * g2 : nullptr; },
        GammaScale{v.gam_sq + D.gamma_off, -1},
        [&](int t, int r, int c) {
            const int i = i0 + r, j = t * kTileN + c;                   // R_oo: both on one child
            return i < iend && j <= i && half == (j >= o1) ? Rc[(long long)opos[i] * mc + opos[j]] : 0.0;
        },
        [&](int t, int r, int c, double x, double old) {
            const int i = i0 + r, j = t * kTileN + c;
            if (i >= iend || j > i) return;
            Rp[(long long)i * m + j] = x + old;
            Rp[(long long)j * m + i] = x + old;
        });
}

// Whether a level's products run as strips: one chunk of k, and the strips
// fill the resident CTAs (two per SM) three times over; with fewer a strip's
// tiles in series outlast the tiles of their own CTAs side by side.  (Strips of
// 128 rows on tcgen05, one CTA per SM, three to five tiles behind a prologue that
// nothing overlaps: X of 2g = 128 0.94 -> 0.67 ms, but X of 2g = 64 0.50 -> 0.88
// and R 1.21 -> 1.44, box 128x128x64 as a whole 36.9 -> 37.2; not kept.)
bool strips(int max_g2, long long ctas) { return max_g2 <= 2 * kChunkK && ctas >= 3 * 2 * kRuleSMs; }

template <int S>
cudaError_t x_launch(const DevView& v, int first, int count, int max_g2, int max_m, cudaStream_t s) {
    const int bytes = (int)sizeof(SplitSmem<S>);
    cudaError_t e = cudaFuncSetAttribute(merge_x_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    const int rt = (max_g2 + kTileM - 1) / kTileM, ct = (max_m + kTileN - 1) / kTileN + 1;
    if (strips(max_g2, (long long)count * rt * 2)) {
        e = cudaFuncSetAttribute(merge_x_strip_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
        merge_x_strip_kernel<S><<<dim3(count, 2 * rt), kGemmThreads, bytes, s>>>(v, first);
        return cudaGetLastError();
    }
    merge_x_kernel<S><<<dim3(count, rt * ct), kGemmThreads, bytes, s>>>(v, first);
    return cudaGetLastError();
}
template <int S>
cudaError_t r_launch(const DevView& v, int first, int count, int max_g2, int max_m, cudaStream_t s) {
    const int bytes = (int)sizeof(SplitSmem<S>);
    cudaError_t e = cudaFuncSetAttribute(merge_rupdate_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    const int rt = (max_m + kTileM - 1) / kTileM + 1, ct = (max_m + kTileN - 1) / kTileN;
    if (strips(max_g2, (long long)count * rt)) {
        e = cudaFuncSetAttribute(merge_rupdate_strip_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
        merge_rupdate_strip_kernel<S><<<dim3(count, rt), kGemmThreads, bytes, s>>>(v, first);
        return cudaGetLastError();
    }
    merge_rupdate_kernel<S><<<dim3(count, rt * ct), kGemmThreads, bytes, s>>>(v, first, ct);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Inversion of the interface systems in blocks of kSweepB rows: the symmetric
// sweep operator of block_invert.cuh, a block K of 64 rows at a time, over
// the quasi-definite T (kernels_merge.cu).  With P = A_KK^-1 and C_x = A_xK,
//     A_KK <- -P,  A_xK <- U_x = C_x P,  A_xy <- A_xy - C_x U_y^T,
// and -T^-1 is left in the end.  Only the lower triangle is kept (row-major,
// in the W storage, or the FP32 work array of a mixed level).
//
// One cooperative launch per tree height, two CTAs of eight warps per SM: T of
// every node, the inverse of the first diagonal blocks; per step the panel
// items (U = C P; C and U into scratch, 64 entries a row), then the update
// items, 64 x 32 tiles of one chunk of k each, behind one item per node that
// updates the next diagonal block and inverts it meanwhile, so that the
// sequential chain of pivots runs beside the other tiles' products; then W.
// A grid barrier between the phases (two per 64 rows); with more items than
// CTAs the update items are handed out by ticket.
//
// Bound by its chain (90 to 100 us per 64 rows: 64 pivots, two barriers) where
// systems are few, else by the update.  Measured against the FP64 sweep of
// gj_sweep_kernel: 256 nodes of 2g = 512 63.7 -> 8.1 ms, 512 of 256 19.1 -> 3.1
// (both go to the phase launches below since), 2 of 1024 3.0 -> 1.5, 1 of 2048
// (the root of 4096^2, a factorisation before) 4.2 -> 3.3.
constexpr int kSweepB = kInvert;
static_assert(kSweepB == kChunkK && kSweepB == kTileM && kSweepB == 2 * kTileN, "one chunk, one tile row per block");

template <class T> __device__ __forceinline__ T* sweep_matrix(const DevView& v);
template <> __device__ __forceinline__ double* sweep_matrix<double>(const DevView& v) { return v.W; }
template <> __device__ __forceinline__ float* sweep_matrix<float>(const DevView& v) { return v.W32; }

// Scratch of a node: C and U of the current block (nmax rows of kSweepB) and
// two P (by step parity).
template <class T>
struct SweepScratch {
    T *C, *U, *P;
    __device__ __forceinline__ SweepScratch(T* scratch, int slot, int nmax) {
        C = scratch + (long long)slot * sweep_node_scratch(nmax);
        U = C + (long long)nmax * kSweepB;
        P = U + (long long)nmax * kSweepB;
    }
    __device__ __forceinline__ T* p(int step) const { return P + (step & 1) * kSweepB * kSweepB; }
};
// Powers of two of the products over a swept block's columns: C_xk goes as
// P_kk^-1/2 of its inverse, P_kc and U_xk as P_kk^1/2.
template <class T>
struct BlockScale {
    const T* P;
    __device__ __forceinline__ int operator()(int k) const { return half_exponent(P[k * (kSweepB + 1)]); }
};

// 1 / sum D of a pinned node's gamma segments (the regularised all-Neumann
// root), 0 otherwise; red: a double per warp of the NT threads.
template <int NT>
__device__ double pinned_inv_sum(const DevView& v, const MergeDesc& D, double* red) {
    if (!D.pinned) return 0.0;                                          // uniform per CTA
    double part = 0.0;
    for (int i = threadIdx.x; i < D.g; i += NT) part += gamma_D(v, D, i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
    __syncthreads();
    double sum = 0.0;
    for (int w = 0; w < NT / 32; ++w) sum += red[w];
    return sum > 0.0 ? 1.0 / sum : 0.0;
}

// Rows [r0, r0 + 16) of T's lower triangle.
template <class T>
__device__ void form_rows(const DevView& v, const MergeDesc& D, int r0, double* red) {
    const NodeRefs N = node_refs(v, D);
    const int g = N.g, n = N.g2;
    const double* sq = v.gam_sq + D.gamma_off;
    const double* sd = v.gam_sd + D.gamma_off;
    const double inv_sum = pinned_inv_sum<kGemmThreads>(v, D, red);
    T* A = sweep_matrix<T>(v) + D.W_off;
    for (int r = r0; r < min(r0 + 16, n); ++r) {
        const int i = r < g ? r : r - g;
        for (int c = threadIdx.x; c <= r; c += kGemmThreads) {
            const int j = c < g ? c : c - g;
            A[(long long)r * n + c] = (T)t_entry(N, c, r, sd[j], sd[i], sq[j], sq[i], inv_sum);
        }
    }
}

// The inverse left in S (zero outside nb) as a full kSweepB x kSweepB matrix.
template <class T>
__device__ void store_inverse(const InvertSmem<T>& S, int nb, T* P) {
    for (int idx = threadIdx.x; idx < kSweepB * kSweepB; idx += kGemmThreads) {
        const int r = idx / kSweepB, c = idx % kSweepB, a = max(r, c), b = min(r, c);
        P[idx] = a < nb ? neg_bits(S.A[a][b]) : (T)0;
    }
}
template <int NT, class T>
__device__ void invert_checked(const DevView& v, InvertSmem<T>& S, int nb, int d_rows) {
    if (!invert_block<NT>(S, nb, [&](T p, int k) { return pivot_ok_bits(p, k < d_rows); }) && threadIdx.x == 0)
        atomicOr(v.status, kStatusSingular);
}

// P of block 0.
template <class T>
__device__ void first_inverse(const DevView& v, const MergeDesc& D, const SweepScratch<T>& sc, InvertSmem<T>& S) {
    const int n = 2 * D.g, nb = min(kSweepB, n);
    const T* A = sweep_matrix<T>(v) + D.W_off;
    __syncthreads();
    for (int idx = threadIdx.x; idx < kSweepB * kSweepB; idx += kGemmThreads) {
        const int r = idx / kSweepB, c = idx % kSweepB;
        S.A[r][c] = r < nb && c <= r ? A[(long long)r * n + c] : (T)0;
    }
    invert_checked<kGemmThreads>(v, S, nb, D.g);
    store_inverse(S, nb, sc.p(0));
}

// U_x = C_x P for 64 rows x outside K and half of K's columns; C and U to
// scratch.
template <class T>
__device__ void panel_item(const DevView& v, const MergeDesc& D, const SweepScratch<T>& sc, int step, int xt, int h0,
                           unsigned char* smem_raw) {
    constexpr int S = Slices<T>::S;
    SplitSmem<S>& sm = *reinterpret_cast<SplitSmem<S>*>(smem_raw);
    const int n = 2 * D.g, k0 = step * kSweepB, nb = min(kSweepB, n - k0), x0 = xt * kSweepB, tid = threadIdx.x;
    if (nb <= 0 || x0 >= n || xt == step || h0 >= nb) return;           // uniform per CTA
    const T* A = sweep_matrix<T>(v) + D.W_off;
    T* C = sc.C + (long long)x0 * kSweepB;
    const int nx = min(kSweepB, n - x0);
    __syncthreads();
    if (xt < step) {
        // rows above K: C_x = A_Kx^T, transposed through shared memory (both
        // halves' items write the same values)
        T (*tile)[kSweepB + 1] = reinterpret_cast<T (*)[kSweepB + 1]>(smem_raw);
        for (int idx = tid; idx < nb * kSweepB; idx += kGemmThreads)
            tile[idx / kSweepB][idx % kSweepB] = A[(long long)(k0 + idx / kSweepB) * n + x0 + idx % kSweepB];
        __syncthreads();
        for (int idx = tid; idx < kSweepB * kSweepB; idx += kGemmThreads) {
            const int x = idx / kSweepB, k = idx % kSweepB;
            if (k < nb) C[idx] = tile[k][x];
        }
        __syncthreads();
    } else if (h0 == 0) {
        for (int idx = tid; idx < nx * kSweepB; idx += kGemmThreads) {
            const int x = idx / kSweepB, k = idx % kSweepB;
            if (k < nb) C[idx] = A[(long long)(x0 + x) * n + k0 + k];
        }
    }
    const T* rows = xt < step ? C : A + (long long)x0 * n + k0;
    const long long ld = xt < step ? kSweepB : n;
    const T* P = sc.p(step);
    typename SplitAcc<S>::T sum[2][4];
    split_product<S, T, false, false>(
        sm, nb, nullptr, [&](int x) { return x < nx ? rows + x * ld : nullptr; },
        [&](int c) { return h0 + c < nb ? P + (h0 + c) * kSweepB : nullptr; }, BlockScale<T>{P}, sum);
    T* U = sc.U + (long long)x0 * kSweepB;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int x = out_row(mt, q), c = h0 + out_col(q);
            if (x < nx && c < nb) U[x * kSweepB + c] = (T)sum[mt][q];
        }
}

// Two adjacent entries in one load (rows of the scratch are aligned to it).
__device__ __forceinline__ void load_pair(double& a, double& b, const double* p) {
    const double2 x = *reinterpret_cast<const double2*>(p);
    a = x.x;
    b = x.y;
}
__device__ __forceinline__ void load_pair(float& a, float& b, const float* p) {
    const float2 x = *reinterpret_cast<const float2*>(p);
    a = x.x;
    b = x.y;
}
// This lane's entries of a scratch row (nb of its 64 entries are set; nb is
// even).
template <class T>
__device__ __forceinline__ void load_scratch_row(T (&v)[kLaneK], const T* p, bool on, int nb) {
#pragma unroll
    for (int i = 0; i < kLaneK; i += 2) {
        v[i] = v[i + 1] = (T)0;
        if (on && lane_k(i) < nb) load_pair(v[i], v[i + 1], p + lane_k(i));
    }
}

// The update of half tiles [h0, h1) (32 columns each) of the 64 rows of tile
// row ti: the digits of C are cut once for the strip, and a half tile's U
// and old entries are loaded while the products of the one before run.
template <class T>
__device__ void update_strip(const DevView& v, const MergeDesc& D, const SweepScratch<T>& sc, int step, int ti, int h0,
                             int h1, unsigned char* smem_raw) {
    constexpr int S = Slices<T>::S;
    SplitSmem<S>& sm = *reinterpret_cast<SplitSmem<S>*>(smem_raw);
    const int n = 2 * D.g, k0 = step * kSweepB, nb = min(kSweepB, n - k0), r0 = ti * kSweepB;
    if (nb <= 0 || r0 >= n) return;                                     // uniform per CTA
    T* A = sweep_matrix<T>(v) + D.W_off;
    const int tid = threadIdx.x, row = stage_slot();
    h1 = min(h1, (n + kTileN - 1) / kTileN);
    // a half tile formed by a product: not in the swept block's rows or
    // columns, not the next diagonal block (its own item, not read again)
    auto product = [&](int h) {
        const int tj = h >> 1;
        return h < h1 && ti != step && tj != step && !(ti == step + 1 && tj == ti);
    };
    auto next_product = [&](int h) {
        while (h < h1 && !product(h)) ++h;
        return h;
    };
    const T* P = sc.p(step);
    for (int h = h0; h < h1; ++h) {
        const int tj = h >> 1, c0 = h * kTileN;
        if (ti != step && tj != step) continue;
        // the swept block's rows and columns, from P and U
        for (int idx = tid; idx < kTileM * kTileN; idx += kGemmThreads) {
            const int r = r0 + idx / kTileN, c = c0 + idx % kTileN;
            if (r >= n || c > r) continue;
            T x;
            if (ti == tj) x = neg_bits(P[(r - k0) * kSweepB + c - k0]);
            else if (tj == step) x = sc.U[(long long)r * kSweepB + c - k0];
            else x = sc.U[(long long)c * kSweepB + r - k0];
            A[(long long)r * n + c] = x;
        }
    }
    int h = next_product(h0);
    if (h >= h1) return;
    const int power = tid < nb ? BlockScale<T>{P}(tid) : 0;             // in flight with the rows
    T vb[kLaneK];
    load_scratch_row(vb, sc.U + (long long)(h * kTileN + row) * kSweepB, h * kTileN + row < n, nb);
    {
        T va[2][kLaneK];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int r = r0 + row + p * kPassRows;
            load_scratch_row(va[p], sc.C + (long long)r * kSweepB, r < n, nb);
        }
        if (tid < kChunkK) sm.sk[tid] = power;                          // (the CTA's previous item has ended)
        __syncthreads();
        int s[kLaneK];
        load_scale(s, sm.sk);
#pragma unroll
        for (int p = 0; p < 2; ++p) stage_row<S, 1>(sm.A, sm.ea, row + p * kPassRows, nb, va[p], s);
    }
    for (;;) {
        const int c0 = h * kTileN;
        {
            int s[kLaneK];
            load_scale(s, sm.sk);
            stage_row<S, -1>(sm.B, sm.eb, row, nb, vb, s);
        }
        __syncthreads();
        const int hn = next_product(h + 1);
        if (hn < h1) load_scratch_row(vb, sc.U + (long long)(hn * kTileN + row) * kSweepB, hn * kTileN + row < n, nb);
        T old[2][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + out_row(mt, q), c = c0 + out_col(q);
                old[mt][q] = r < n && c <= r ? A[(long long)r * n + c] : (T)0;
            }
        float acc[S][2][4];
        chunk_mma<S>(sm, nb, acc);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float l[S];
#pragma unroll
                for (int i = 0; i < S; ++i) l[i] = acc[i][mt][q];
                const T x = (T)combine_levels(l, sm.ea[out_row(mt, q)], sm.eb[out_col(q)]);
                const int r = r0 + out_row(mt, q), c = c0 + out_col(q);
                if (r < n && c <= r) A[(long long)r * n + c] = old[mt][q] - x;
            }
        if (hn >= h1) return;
        h = hn;
        __syncthreads();
    }
}

// The next diagonal block: its update and its inverse, P of step + 1.
template <class T>
__device__ void next_inverse(const DevView& v, const MergeDesc& D, const SweepScratch<T>& sc, int step,
                             unsigned char* smem_raw) {
    constexpr int S = Slices<T>::S;
    SplitSmem<S>& sm = *reinterpret_cast<SplitSmem<S>*>(smem_raw);
    InvertSmem<T>& I = *reinterpret_cast<InvertSmem<T>*>(smem_raw);
    static_assert(sizeof(InvertSmem<T>) <= sizeof(SplitSmem<S>), "the inversion reuses the digits' storage");
    const int n = 2 * D.g, k1 = (step + 1) * kSweepB;
    if (k1 >= n) return;                                                // uniform per CTA
    const int nb1 = min(kSweepB, n - k1);
    const T* A = sweep_matrix<T>(v) + D.W_off;
    typename SplitAcc<S>::T sum[2][2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        __syncthreads();
        split_product<S, T, false, false>(
            sm, kSweepB, nullptr, [&](int x) { return x < nb1 ? sc.C + (long long)(k1 + x) * kSweepB : nullptr; },
            [&](int c) { return h * kTileN + c < nb1 ? sc.U + (long long)(k1 + h * kTileN + c) * kSweepB : nullptr; },
            BlockScale<T>{sc.p(step)}, sum[h]);
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = out_row(mt, q), c = h * kTileN + out_col(q);
                I.A[r][c] = r < nb1 && c <= r ? A[(long long)(k1 + r) * n + k1 + c] - (T)sum[h][mt][q] : (T)0;
            }
    invert_checked<kGemmThreads>(v, I, nb1, D.g - k1);
    store_inverse(I, nb1, sc.p(step + 1));
}

// W = D^-1/2 Q T^-1 Q^T D^-1/2 (both triangles) from the entries dd, sd (s_i,
// d_j), ds (d_i, s_j), ss of -T^-1: the entries (a_i, a_j), (b_i, b_j), (a_i,
// b_j), (b_i, a_j) of W.
template <class T>
__device__ __forceinline__ void back_entries(T dd, T sd, T ds, T ss, T sc, double (&w)[4]) {
    const T sum = dd + ss, cross = ds + sd, dif = ss - dd, skew = sd - ds;
    w[0] = (double)((cross - sum) * sc);
    w[1] = (double)(neg_bits(sum + cross) * sc);
    w[2] = (double)(neg_bits(dif + skew) * sc);
    w[3] = (double)((skew - dif) * sc);
}

// ... by 32 x 32 tiles of (i, j), i, j < g, i's tile at or below j's; a tile
// pair is read and written by its own item only (in FP64 the two matrices
// share their storage).
constexpr int kBackTile = 32;
template <class T>
struct BackSmem {
    T z[4][kBackTile][kBackTile + 1];          // dd, sd, ds, ss
    double w[2][kBackTile][kBackTile + 1];
};
template <class T>
__device__ void back_item(const DevView& v, const MergeDesc& D, int ti, int tj, BackSmem<T>& S) {
    const int g = D.g, n = 2 * g, tid = threadIdx.x;
    const int i0 = ti * kBackTile, j0 = tj * kBackTile;
    if (i0 >= g) return;                                                // uniform per CTA
    const T* A = sweep_matrix<T>(v) + D.W_off;
    double* W = v.W + D.W_off;
    const double* sd = v.gam_sd + D.gamma_off;
    auto at = [&](int r, int c) -> T { return r >= c ? A[(long long)r * n + c] : A[(long long)c * n + r]; };
    __syncthreads();
    for (int idx = tid; idx < kBackTile * kBackTile; idx += kGemmThreads) {
        const int a = idx / kBackTile, b = idx % kBackTile;             // b along the rows of A
        const int i = i0 + a, j = j0 + b;
        if (i < g && j < g) {
            S.z[0][a][b] = at(i, j);
            S.z[1][a][b] = A[(long long)(g + i) * n + j];
            S.z[3][a][b] = at(g + i, g + j);
        }
        const int jj = j0 + a, ii = i0 + b;
        if (ii < g && jj < g) S.z[2][b][a] = A[(long long)(g + jj) * n + ii];
    }
    __syncthreads();
    // blocks (a_i, a_j) and (b_i, b_j), then (a_i, b_j) and (b_i, a_j); each
    // written with its mirror
    for (int pass = 0; pass < 2; ++pass) {
        for (int idx = tid; idx < kBackTile * kBackTile; idx += kGemmThreads) {
            const int a = idx / kBackTile, b = idx % kBackTile, i = i0 + a, j = j0 + b;
            if (i >= g || j >= g) continue;
            double w[4];
            back_entries(S.z[0][a][b], S.z[1][a][b], S.z[2][a][b], S.z[3][a][b], (T)(0.5 * sd[i] * sd[j]), w);
            S.w[0][a][b] = w[2 * pass];
            S.w[1][a][b] = w[2 * pass + 1];
        }
        __syncthreads();
        for (int idx = tid; idx < kBackTile * kBackTile; idx += kGemmThreads) {
            const int a = idx / kBackTile, b = idx % kBackTile;
            {
                const int i = i0 + a, j = j0 + b;
                if (i < g && j < g) {
                    W[(long long)i * n + j + (pass ? g : 0)] = S.w[0][a][b];
                    W[(long long)(g + i) * n + j + (pass ? 0 : g)] = S.w[1][a][b];
                }
            }
            if (ti != tj) {
                const int i = i0 + b, j = j0 + a;
                if (i < g && j < g) {
                    W[(long long)(j + (pass ? g : 0)) * n + i] = S.w[0][b][a];
                    W[(long long)(j + (pass ? 0 : g)) * n + g + i] = S.w[1][b][a];
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// The same sweep for levels with work enough to fill the GPU at every step:
// one launch per phase and step instead of one cooperative launch, each with
// the CTA shape that suits it, and the update on the fifth-generation tensor
// cores (tc_split.cuh).
template <class T>
__global__ void __launch_bounds__(kGemmThreads) sweep_form_kernel(DevView v, int first, int runs) {
    __shared__ double red[kGemmWarps];
    const MergeDesc& D = v.merges[first + blockIdx.x / runs];
    const int r0 = (int)(blockIdx.x % runs) * 16;
    if (r0 < 2 * D.g) form_rows<T>(v, D, r0, red);
}
// P of block `step`.
constexpr int kNodeThreads = 128;
template <class T>
__global__ void __launch_bounds__(kNodeThreads, 4) sweep_inverse_kernel(DevView v, int first, int nmax, T* scratch,
                                                                        int step) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    InvertSmem<T>& I = *reinterpret_cast<InvertSmem<T>*>(smem_raw);
    const MergeDesc& D = v.merges[first + blockIdx.x];
    const int n = 2 * D.g, k0 = step * kSweepB, nb = min(kSweepB, n - k0);
    if (nb <= 0) return;
    const T* A = sweep_matrix<T>(v) + D.W_off + (long long)k0 * n + k0;
    for (int idx = threadIdx.x; idx < kInvert * kInvert; idx += kNodeThreads) {
        const int r = idx / kInvert, c = idx % kInvert;
        I.A[r][c] = r < nb && c <= r ? A[(long long)r * n + c] : (T)0;
    }
    invert_checked<kNodeThreads>(v, I, nb, D.g - k0);
    T* P = SweepScratch<T>(scratch, blockIdx.x, nmax).p(step);
    for (int idx = threadIdx.x; idx < kSweepB * kSweepB; idx += kNodeThreads) {
        const int r = idx / kSweepB, c = idx % kSweepB, a = max(r, c), b = min(r, c);
        P[idx] = a < nb ? neg_bits(I.A[a][b]) : (T)0;
    }
}
template <class T>
__global__ void __launch_bounds__(kGemmThreads, 2) sweep_panel_kernel(DevView v, int first, int count, int nmax,
                                                                      T* scratch, int step) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int q = blockIdx.x % count, r = blockIdx.x / count;
    panel_item<T>(v, v.merges[first + q], SweepScratch<T>(scratch, q, nmax), step, r >> 1, (r & 1) * kTileN, smem_raw);
}
// Eight entries of a scratch row (zeros where !on and past the nb set ones).
template <class T>
__device__ __forceinline__ void load_eight(T (&x)[8], const T* p, bool on, int nb) {
    const int j = (threadIdx.x & 7) * 8;
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
        x[i] = x[i + 1] = (T)0;
        if (on && j + i < nb) load_pair(x[i], x[i + 1], p + j + i);
    }
}
__device__ __forceinline__ void store_pair(double* p, double a, double b) {
    *reinterpret_cast<double2*>(p) = make_double2(a, b);
}
__device__ __forceinline__ void store_pair(float* p, float a, float b) {
    *reinterpret_cast<float2*>(p) = make_float2(a, b);
}
// Half tiles (32 columns) per update item, and the items of a row pair's
// (128 rows, pair p) half tiles up to the diagonal.
constexpr int kTcStrip = 8;
__host__ __device__ __forceinline__ int tc_pieces(int p, int nmax) {
    const int halves = min(4 * p + 4, (nmax + kTcN - 1) / kTcN);
    return (halves + kTcStrip - 1) / kTcStrip;
}
// The update of a strip of one row pair: the digits of C cut once, U's a half
// tile ahead of the tensor cores, the results combined a half tile behind
// them; then the swept block's rows and columns, from P and U.  FP64: one CTA
// per SM (203 KB of digits, all of tensor memory), 16 warps, because the cutting
// and combining (about 75 integer instructions an output), not the MMAs, set
// the pace: a 128 x 32 half tile takes 2.3k cycles of tensor pipe; with eight
// warps 15.5k cycles in all (256 x 512: 6.3 ms), with sixteen 5.8 ms, as 64 x 32
// tiles of mma.sync at two CTAs per SM 8.1 ms.
template <class T>
__global__ void __launch_bounds__(kTcThreads, sizeof(T) == 8 ? 1 : 2)
sweep_update_kernel(DevView v, int first, int count, int nmax, T* scratch, int step) {
    constexpr int S = Slices<T>::S;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TcSmem<S>& sm = *reinterpret_cast<TcSmem<S>*>(smem_raw);
    const int q = blockIdx.x % count, tid = threadIdx.x;
    int piece = blockIdx.x / count, p = (nmax + kTcM - 1) / kTcM - 1;
    for (; piece >= tc_pieces(p, nmax); --p) piece -= tc_pieces(p, nmax);       // long rows first
    const MergeDesc& D = v.merges[first + q];
    const int n = 2 * D.g, k0 = step * kSweepB, nb = min(kSweepB, n - k0), r0 = p * kTcM;
    if (nb <= 0 || r0 >= n) return;                                     // uniform per CTA
    const int h0 = piece * kTcStrip, h1 = min(h0 + kTcStrip, min(4 * p + 4, (n + kTcN - 1) / kTcN));
    const SweepScratch<T> sc(scratch, q, nmax);
    T* A = sweep_matrix<T>(v) + D.W_off;
    const bool lo = 2 * p != step, hi = 2 * p + 1 != step && r0 + kSweepB < n;  // the row blocks with products
    auto next_product = [&](int h) {
        for (; h < h1; ++h) {
            const int tj = h >> 1;
            if (tj != step && ((lo && tj <= 2 * p) || (hi && tj <= 2 * p + 1))) break;
        }
        return h;
    };
    const T* P = sc.p(step);
    const int power = tid < nb ? BlockScale<T>{P}(tid) : 0;             // in flight with what follows
    for (int h = h0; h < h1; ++h) {
        const int tj = h >> 1, c0 = h * kTcN;
        for (int ti = 2 * p; ti < 2 * p + 2; ++ti) {
            if (ti != step && tj != step) continue;
            // rows of the swept block are columns of U: a warp takes 8 rows x 4
            // columns, whole sectors on both sides
            const bool flip = ti == step && tj != step;
            for (int idx = tid; idx < kSweepB * kTcN; idx += kTcThreads) {
                const int b = idx >> 5, l = idx & 31;
                const int r = ti * kSweepB + (flip ? 8 * (b >> 3) + (l >> 2) : b);
                const int c = c0 + (flip ? 4 * (b & 7) + (l & 3) : l);
                if (r >= n || c > r) continue;
                T x;
                if (ti == tj) x = neg_bits(P[(r - k0) * kSweepB + c - k0]);
                else if (tj == step) x = sc.U[(long long)r * kSweepB + c - k0];
                else x = sc.U[(long long)c * kSweepB + r - k0];
                A[(long long)r * n + c] = x;
            }
        }
    }
    int h = next_product(h0);
    if (h >= h1) return;
    if (tid < kSweepB) sm.sk[tid] = power;
    tc_begin(sm);
    const int row = tid >> 3;                                           // (B: the first 32 of the CTA's 64 rows)
    const bool stages_b = row < kTcN;                                   // uniform per warp
    T vb[8];
    auto load_b = [&](int hh) {
        const int r = hh * kTcN + row;
        load_eight(vb, sc.U + (long long)r * kSweepB, stages_b && hh < h1 && r < n, nb);
    };
    load_b(h);
#pragma unroll
    for (int i = 0; i < kTcM; i += kTcThreads / 8) {
        const int r = r0 + i + row;
        T va[8];
        load_eight(va, sc.C + (long long)r * kSweepB, r < n && r / kSweepB != step, nb);
        tc_stage_a<S>(sm, i + row, va);
    }
    if (stages_b) tc_stage_b<S>(sm, 0, row, vb);
    tc_staged();
    if (tid == 0) tc_issue(sm, 0, nb);
    int hn = next_product(h + 1);
    load_b(hn);
    const int r = r0 + tc_row();
    const bool mine = r < n && r / kSweepB != step;
    bool ok = true;                                                     // (uniform per warp)
    int issued = 0;
    for (int tile = 0;; ++tile) {
        const int c0 = h * kTcN + tc_col();
        T* Ar = A + (long long)r * n + c0;
        T old[kTcOut];
#pragma unroll
        for (int c = 0; c < kTcOut; c += 2) {
            old[c] = old[c + 1] = (T)0;
            if (mine && c0 + c <= r) load_pair(old[c], old[c + 1], Ar + c);
        }
        if (hn < h1) {
            if (stages_b && ok) tc_stage_b<S>(sm, tile + 1, row, vb);
            if (tc_staged(!ok)) break;                                  // a warp gave up on a tile
            if (tid == 0) tc_issue(sm, tile + 1, nb);
            issued = tile + 1;
        }
        const int h2 = next_product(hn + 1);
        load_b(h2);
        ok = ok && tc_wait(sm, tile, v.spin_limit);
        if (ok) {
#pragma unroll
            for (int u = 0; u < kTcOut / 4; ++u) {
                typename SplitAcc<S>::T x[4];
                tc_outputs(sm, tile, u, x);
#pragma unroll
                for (int c = 0; c < 4; c += 2) {
                    const int cc = 4 * u + c;
                    const T y0 = old[cc] - (T)x[c], y1 = old[cc + 1] - (T)x[c + 1];
                    if (mine && c0 + cc + 1 <= r) store_pair(Ar + cc, y0, y1);
                    else if (mine && c0 + cc == r) Ar[cc] = y0;
                }
            }
        }
        if (hn >= h1) break;
        h = hn;
        hn = h2;
    }
    tc_end(sm, ok, issued, v.status);
}
template <class T>
__global__ void __launch_bounds__(kGemmThreads) sweep_back_kernel(DevView v, int first, int tiles) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int ti, tj;
    tri_rc((int)(blockIdx.x % tiles), ti, tj);
    back_item<T>(v, v.merges[first + blockIdx.x / tiles], ti, tj, *reinterpret_cast<BackSmem<T>*>(smem_raw));
}

template <class T>
cudaError_t phase_sweep(const DevView& v, int first, int count, int nmax, T* scratch, cudaStream_t s) {
    constexpr int S = Slices<T>::S;
    constexpr int panel_bytes = (int)sizeof(SplitSmem<S>), inv_bytes = (int)sizeof(InvertSmem<T>);
    constexpr int up_bytes = (int)sizeof(TcSmem<S>), back_bytes = (int)sizeof(BackSmem<T>);
    cudaError_t e;
    auto allow = [&](auto* kern, int bytes) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    if ((e = allow(sweep_inverse_kernel<T>, inv_bytes)) != cudaSuccess) return e;
    if ((e = allow(sweep_panel_kernel<T>, panel_bytes)) != cudaSuccess) return e;
    if ((e = allow(sweep_update_kernel<T>, up_bytes)) != cudaSuccess) return e;
    if ((e = allow(sweep_back_kernel<T>, back_bytes)) != cudaSuccess) return e;
    const int nt = (nmax + kSweepB - 1) / kSweepB, runs = (nmax + 15) / 16;
    const int gt = (nmax / 2 + kBackTile - 1) / kBackTile, tiles = gt * (gt + 1) / 2;
    int pieces = 0;
    for (int p = 0; p < (nmax + kTcM - 1) / kTcM; ++p) pieces += tc_pieces(p, nmax);
    sweep_form_kernel<T><<<count * runs, kGemmThreads, 0, s>>>(v, first, runs);
    for (int step = 0; step < nt; ++step) {
        sweep_inverse_kernel<T><<<count, kNodeThreads, inv_bytes, s>>>(v, first, nmax, scratch, step);
        sweep_panel_kernel<T><<<count * 2 * nt, kGemmThreads, panel_bytes, s>>>(v, first, count, nmax, scratch, step);
        sweep_update_kernel<T><<<count * pieces, kTcThreads, up_bytes, s>>>(v, first, count, nmax, scratch, step);
    }
    sweep_back_kernel<T><<<count * tiles, kGemmThreads, back_bytes, s>>>(v, first, tiles);
    return cudaGetLastError();
}

template <class T>
constexpr size_t sweep_smem() {
    return std::max({sizeof(SplitSmem<Slices<T>::S>), sizeof(InvertSmem<T>), sizeof(BackSmem<T>)});
}

template <class T>
__global__ void __launch_bounds__(kGemmThreads, 2) block_sweep_kernel(DevView v, int first, int count, int nmax,
                                                                      T* scratch, unsigned int* counter) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[kGemmWarps];
    __shared__ int s_item;
    unsigned int* work = counter + 1;                       // ticket counter of the update items
    unsigned int wbase = 0, round = 0;
    const int nt = (nmax + kSweepB - 1) / kSweepB, gt = (nmax / 2 + kBackTile - 1) / kBackTile;
    const int grid = gridDim.x;
    auto node = [&](int q) -> const MergeDesc& { return v.merges[first + q]; };
    auto scr = [&](int q) { return SweepScratch<T>(scratch, q, nmax); };
    {
        const int runs = (nmax + 15) / 16;
        for (long long item = blockIdx.x; item < (long long)count * runs; item += grid) {
            const int q = (int)(item / runs), r0 = (int)(item % runs) * 16;
            if (r0 < 2 * node(q).g) form_rows<T>(v, node(q), r0, red);
        }
    }
    if (!grid_barrier(counter, round, v.status, v.spin_limit)) return;
    for (int q = blockIdx.x; q < count; q += grid)
        first_inverse<T>(v, node(q), scr(q), *reinterpret_cast<InvertSmem<T>*>(smem_raw));
    if (!grid_barrier(counter, round, v.status, v.spin_limit)) return;
    for (int step = 0; step < nt; ++step) {
        if (nt > 1) {
            for (int item = blockIdx.x; item < count * 2 * nt; item += grid) {
                const int q = item % count, r = item / count;
                panel_item<T>(v, node(q), scr(q), step, r >> 1, (r & 1) * kTileN, smem_raw);
            }
            if (!grid_barrier(counter, round, v.status, v.spin_limit)) return;
        }
        // the next diagonal blocks, then strips of half tiles, a few per CTA
        const int halves = count * nt * (nt + 1);
        const int len = max(1, min(2 * nt, halves / (3 * grid)));
        int pieces = 0;
        for (int t = 0; t < nt; ++t) pieces += (2 * t + 1 + len) / len;
        const int nitems = count * (1 + pieces);
        const bool dyn = nitems > grid;
        int item = dyn ? grab_item(work, wbase, &s_item) : (int)blockIdx.x;
        while (item < nitems) {
            // the next ticket is taken while this item runs
            if (dyn && threadIdx.x == 0) s_item = (int)(atomicAdd(work, 1u) - wbase);
            const int q = item % count;
            int r = item / count - 1;
            if (r < 0) {
                next_inverse<T>(v, node(q), scr(q), step, smem_raw);
            } else {
                // long rows first
                int ti = nt - 1;
                for (; r >= (2 * ti + 1 + len) / len; --ti) r -= (2 * ti + 1 + len) / len;
                update_strip<T>(v, node(q), scr(q), step, ti, r * len, min((r + 1) * len, 2 * ti + 2), smem_raw);
            }
            __syncthreads();
            item = dyn ? s_item : nitems;
            __syncthreads();
        }
        if (dyn) wbase += (unsigned int)nitems + grid;
        if (!grid_barrier(counter, round, v.status, v.spin_limit)) return;
    }
    for (int item = blockIdx.x; item < count * (gt * (gt + 1) / 2); item += grid) {
        int ti, tj;
        tri_rc(item / count, ti, tj);
        back_item<T>(v, node(item % count), ti, tj, *reinterpret_cast<BackSmem<T>*>(smem_raw));
    }
}

// One CTA per node for levels of many small systems (2g <= 64): T, its
// inverse and W without leaving shared memory.  Four CTAs of four warps per SM:
// a CTA waits for its chain of pivots most of the time, the others fill in
// (4096 nodes of 2g = 64, FP64: 0.78 ms, 1.08 with two CTAs of eight warps).
template <class T>
__global__ void __launch_bounds__(kNodeThreads, 4) node_invert_kernel(DevView v, int first) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[kNodeThreads / 32];
    InvertSmem<T>& S = *reinterpret_cast<InvertSmem<T>*>(smem_raw);
    const MergeDesc D = v.merges[first + blockIdx.x];
    const NodeRefs N = node_refs(v, D);
    const int g = N.g, n = N.g2;
    const double* sq = v.gam_sq + D.gamma_off;
    const double* sd = v.gam_sd + D.gamma_off;
    const double inv_sum = pinned_inv_sum<kNodeThreads>(v, D, red);
    for (int idx = threadIdx.x; idx < kInvert * kInvert; idx += kNodeThreads) {
        const int r = idx / kInvert, c = idx % kInvert;
        const int i = r < g ? r : r - g, j = c < g ? c : c - g;
        S.A[r][c] = r < n && c <= r ? (T)t_entry(N, c, r, sd[j], sd[i], sq[j], sq[i], inv_sum) : (T)0;
    }
    invert_checked<kNodeThreads>(v, S, n, g);
    double* W = v.W + D.W_off;
    auto at = [&](int r, int c) -> T { return r >= c ? S.A[r][c] : S.A[c][r]; };
    for (int idx = threadIdx.x; idx < g * g; idx += kNodeThreads) {
        const int i = idx / g, j = idx % g;
        double w[4];
        back_entries(at(i, j), S.A[g + i][j], S.A[g + j][i], at(g + i, g + j), (T)(0.5 * sd[i] * sd[j]), w);
        W[i * n + j] = w[0];
        W[(g + i) * n + g + j] = w[1];
        W[i * n + g + j] = w[2];
        W[(g + i) * n + j] = w[3];
    }
}

template <class T>
cudaError_t block_sweep(const DevView& v, int first, int count, int nmax, T* scratch, void* barrier, int sms,
                        int per_sm, cudaStream_t s) {
    constexpr int bytes = (int)sweep_smem<T>();
    auto* kern = block_sweep_kernel<T>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    const int nt = (nmax + kSweepB - 1) / kSweepB;
    const long long items = std::max<long long>((long long)count * (1 + nt * (nt + 1)), (long long)count * ((nmax + 15) / 16));
    int fit = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, kGemmThreads, bytes)) != cudaSuccess) return e;
    const int grid = (int)std::min<long long>(items, (long long)sms * std::max(1, std::min(per_sm, fit)));
    // the grid barrier's arrival counter and the ticket counter
    if ((e = cudaMemsetAsync(barrier, 0, 2 * sizeof(unsigned int), s)) != cudaSuccess) return e;
    unsigned int* bar = reinterpret_cast<unsigned int*>(barrier);
    DevView vv = v;
    void* args[] = {&vv, &first, &count, &nmax, &scratch, &bar};
    return cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kGemmThreads), args, bytes, s);
}
template <class T>
cudaError_t node_invert(const DevView& v, int first, int count, cudaStream_t s) {
    constexpr int bytes = (int)sizeof(InvertSmem<T>);
    cudaError_t e = cudaFuncSetAttribute(node_invert_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    node_invert_kernel<T><<<count, kNodeThreads, bytes, s>>>(v, first);
    return cudaGetLastError();
}

// D^1/2 and D^-1/2 of every gamma segment of the tree.
__global__ void gamma_scale_kernel(DevView v, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double sq = sqrt(v.seg_D[v.gamma_segs[i]]);
    v.gam_sq[i] = sq;
    v.gam_sd[i] = 1.0 / sq;
}

}  // namespace

cudaError_t launch_gamma_scale(const DevView& v, int n, cudaStream_t s) {
    if (n > 0) gamma_scale_kernel<<<(n + 127) / 128, 128, 0, s>>>(v, n);
    return cudaGetLastError();
}
cudaError_t launch_block_sweep(const DevView& v, int first, int count, int max_g2, bool fp32, double* scratch,
                               void* barrier, int sms, int per_sm, cudaStream_t s) {
    return fp32 ? block_sweep<float>(v, first, count, max_g2, reinterpret_cast<float*>(scratch), barrier, sms, per_sm, s)
                : block_sweep<double>(v, first, count, max_g2, scratch, barrier, sms, per_sm, s);
}
cudaError_t launch_phase_sweep(const DevView& v, int first, int count, int max_g2, bool fp32, double* scratch,
                               cudaStream_t s) {
    return fp32 ? phase_sweep<float>(v, first, count, max_g2, reinterpret_cast<float*>(scratch), s)
                : phase_sweep<double>(v, first, count, max_g2, scratch, s);
}
cudaError_t launch_node_invert(const DevView& v, int first, int count, bool fp32, cudaStream_t s) {
    return fp32 ? node_invert<float>(v, first, count, s) : node_invert<double>(v, first, count, s);
}

cudaError_t launch_merge_x(const DevView& v, int first, int count, int max_g2, int max_m, bool fp32, cudaStream_t s) {
    return fp32 ? x_launch<4>(v, first, count, max_g2, max_m, s) : x_launch<8>(v, first, count, max_g2, max_m, s);
}
cudaError_t launch_merge_r(const DevView& v, int first, int count, int max_g2, int max_m, bool fp32, cudaStream_t s) {
    return fp32 ? r_launch<4>(v, first, count, max_g2, max_m, s) : r_launch<8>(v, first, count, max_g2, max_m, s);
}

}  // namespace mrcm
