// What the merge kernels share: a node's operands and the entries of its
// quasi-definite form T (see kernels_merge.cu for the form itself).
#pragma once
#include "mrcm_internal.h"

namespace mrcm {
namespace {

struct NodeRefs {
    int g, g2, m, o1, m1, m2;
    const int *gpos1, *gpos2, *opos1, *opos2;
    const double *R1, *R2;
};

__device__ __forceinline__ NodeRefs node_refs(const DevView& v, const MergeDesc& D) {
    NodeRefs r;
    r.g = D.g; r.g2 = 2 * D.g; r.m = D.m; r.o1 = D.o1; r.m1 = D.m1; r.m2 = D.m2;
    r.gpos1 = v.node_map + D.map_off;
    r.gpos2 = r.gpos1 + D.g;
    r.opos1 = r.gpos2 + D.g;
    r.opos2 = r.opos1 + D.o1;
    r.R1 = v.R + D.R1_off;
    r.R2 = v.R + D.R2_off;
    return r;
}

__device__ __forceinline__ double gamma_D(const DevView& v, const MergeDesc& D, int i) {
    return v.seg_D[v.gamma_segs[D.gamma_off + i]];
}

// Entry of T at (row r, column c), r, c in [0, 2g): d block first.  sd* =
// D^-1/2 and sq* = D^1/2 of the two gamma segments, inv_sum = 1 / sum D for
// the regularised all-Neumann root (0 otherwise).
__device__ __forceinline__ double t_entry(const NodeRefs& N, int r, int c, double sdi, double sdj, double sqi,
                                          double sqj, double inv_sum) {
    const int g = N.g;
    const bool dr = r < g, dc = c < g;
    const int i = dr ? r : r - g, j = dc ? c : c - g;
    // R is stored symmetric: read it along the column of j, so that
    // consecutive r (consecutive i) read consecutive entries
    const double ra = N.R1[N.gpos1[j] * N.m1 + N.gpos1[i]] * sdi * sdj;
    const double rb = N.R2[N.gpos2[j] * N.m2 + N.gpos2[i]] * sdi * sdj;
    if (dr && dc) return 0.5 * (ra + rb) + (i == j ? 2.0 : 0.0);
    if (!dr && !dc) return 0.5 * (ra + rb) - sqi * sqj * inv_sum;
    return 0.5 * (rb - ra);
}

constexpr double kTinyPivot = 1e-14;   // pivots of the scaled form are O(1)

// Whether a pivot has the expected sign (positive on the d block, negative
// on the s block), a magnitude above kTinyPivot and is finite, tested on the
// bit pattern (an FP64 compare takes a full FP64 instruction).
__device__ __forceinline__ bool pivot_ok_bits(double p, bool d_row) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(p);
    const unsigned long long mag = b & 0x7fffffffffffffffull;
    const unsigned long long tiny = (unsigned long long)__double_as_longlong(kTinyPivot);
    return ((b >> 63) == (d_row ? 0ull : 1ull)) && mag > tiny && mag < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool pivot_ok_bits(float p, bool d_row) {
    const unsigned int b = __float_as_uint(p);
    const unsigned int mag = b & 0x7fffffffu;
    const unsigned int tiny = __float_as_uint((float)kTinyPivot);
    return ((b >> 31) == (d_row ? 0u : 1u)) && mag > tiny && mag < 0x7f800000u;
}

// (row, column) of entry r of a row-packed lower triangle
__device__ __forceinline__ void tri_rc(int r, int& a, int& b) {
    a = (int)((sqrtf(8.0f * r + 1.0f) - 1.0f) * 0.5f);
    while ((a + 1) * (a + 2) / 2 <= r) ++a;
    while (a * (a + 1) / 2 > r) --a;
    b = r - a * (a + 1) / 2;
}

// A load that acquires what was released before the value was written.
__device__ __forceinline__ unsigned int ld_acquire_gpu(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Grid-wide barrier of a cooperative launch: a monotonic arrival counter
// (reset before the launch); round n ends when it reaches (n + 1) * grid.
// What a CTA wrote before the barrier is visible to the others after it, plain
// loads included: its threads' writes are ordered before thread 0's fence and
// arrival by the CTA barrier, thread 0 of the reader acquires the counter, and
// its CTA barrier orders the reader's loads behind that.  (Kernels that read a
// location both before and after a barrier through __ldcg do so to keep it out
// of L1, not for correctness.)  Every wait is bounded (`limit` polls, about a
// second by default); a CTA that gives up sets kStatusTimeout and the caller
// returns.
__device__ bool grid_barrier(unsigned int* counter, unsigned int& round, int* status, long long limit) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned int target = (round + 1) * gridDim.x;
        __threadfence();
        atomicAdd(counter, 1u);
        long long spins = 0;
        while (ld_acquire_gpu(counter) < target) {
            if (++spins > limit) {
                ok = 0;
                atomicOr(status, kStatusTimeout);
                break;
            }
        }
        s_ok = ok;
    }
    ++round;
    __syncthreads();
    return s_ok != 0;
}

// Next item of a dynamically distributed loop: thread 0 takes a ticket from
// the launch's work counter (work; zeroed with the barrier counter before
// the launch) and the CTA reads it.  The tickets of one loop run from base;
// every CTA leaves the loop at its first ticket past the loop's items, so a
// loop of n items consumes n + gridDim.x tickets (the next loop's base).
__device__ __forceinline__ int grab_item(unsigned int* work, unsigned int base, int* s_item) {
    if (threadIdx.x == 0) *s_item = (int)(atomicAdd(work, 1u) - base);
    __syncthreads();
    const int item = *s_item;
    __syncthreads();
    return item;
}

}  // namespace
}  // namespace mrcm
