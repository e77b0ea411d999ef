// The matrix products of the blocked merges on the tensor cores (the split
// products of split_gemm.cuh): X = -W C and the merged map R = R_oo + C^T X
// of every node of a tree height (Eqs. new_bfs.1-2; kernels_merge.cu has the
// derivation and the launches around these).
#include "merge_common.cuh"
#include "split_gemm.cuh"

namespace mrcm {
namespace {

// X = -W blockdiag(R^a_go, R^b_go): column j < o1 uses the first g columns
// of W and child a's map, the others the last g and child b's, so the tiles
// of X's columns are cut on either side of o1.  W is symmetric: its row r is
// read as column r, contiguous in k, and the map of a child is symmetric:
// column j of C is read along the map's row of that segment.
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
    typename SplitAcc<S>::T sum[2][2][4];
    split_product<S, double, false, true>(
        sm, g, gpos, [&](int r) { return r0 + r < g2 ? W + (long long)(r0 + r) * g2 : nullptr; },
        [&](int j) { return j0 + j < jend ? Rc + (long long)opos[j0 + j] * mc : nullptr; }, sum);
    double* X = v.X + D.X_off;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + (warp >> 1) * 32 + 16 * mt + (lane >> 2) + 8 * (q >> 1);
                const int j = j0 + (warp & 1) * 16 + 8 * nt + 2 * (lane & 3) + (q & 1);
                if (r < g2 && j < jend) X[(long long)j * g2 + r] = -(double)sum[mt][nt][q];
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
    typename SplitAcc<S>::T sum[2][2][4];
    split_product<S, double, true, false>(
        sm, g, gpos, [&](int i) { return i0 + i < iend ? Rc + (long long)opos[i0 + i] * mc : nullptr; },
        [&](int j) { return j0 + j < m ? X + (long long)(j0 + j) * g2 : nullptr; }, sum);
    double* Rp = v.R + D.R_off;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + (warp >> 1) * 32 + 16 * mt + (lane >> 2) + 8 * (q >> 1);
                const int j = j0 + (warp & 1) * 16 + 8 * nt + 2 * (lane & 3) + (q & 1);
                if (i >= iend || j > i) continue;
                double val = (double)sum[mt][nt][q];
                if (half == (j >= o1)) val += Rc[(long long)opos[i] * mc + opos[j]];   // both on one child
                Rp[(long long)i * m + j] = val;
                Rp[(long long)j * m + i] = val;
            }
}

template <int S>
cudaError_t x_launch(const DevView& v, int first, int count, int max_g2, int max_m, cudaStream_t s) {
    const int bytes = (int)sizeof(SplitSmem<S>);
    cudaError_t e = cudaFuncSetAttribute(merge_x_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    const int rt = (max_g2 + kTileM - 1) / kTileM, ct = (max_m + kTileN - 1) / kTileN + 1;
    merge_x_kernel<S><<<dim3(count, rt * ct), kGemmThreads, bytes, s>>>(v, first);
    return cudaGetLastError();
}
template <int S>
cudaError_t r_launch(const DevView& v, int first, int count, int max_m, cudaStream_t s) {
    const int bytes = (int)sizeof(SplitSmem<S>);
    cudaError_t e = cudaFuncSetAttribute(merge_rupdate_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    const int rt = (max_m + kTileM - 1) / kTileM + 1, ct = (max_m + kTileN - 1) / kTileN;
    merge_rupdate_kernel<S><<<dim3(count, rt * ct), kGemmThreads, bytes, s>>>(v, first, ct);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_merge_x(const DevView& v, int first, int count, int max_g2, int max_m, bool fp32, cudaStream_t s) {
    return fp32 ? x_launch<4>(v, first, count, max_g2, max_m, s) : x_launch<7>(v, first, count, max_g2, max_m, s);
}
cudaError_t launch_merge_r(const DevView& v, int first, int count, int max_m, bool fp32, cudaStream_t s) {
    return fp32 ? r_launch<4>(v, first, count, max_m, s) : r_launch<7>(v, first, count, max_m, s);
}

}  // namespace mrcm
