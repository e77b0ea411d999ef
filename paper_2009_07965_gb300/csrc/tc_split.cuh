// Split products (split_gemm.cuh) on the fifth-generation tensor cores.
//
// Tiles of 128 rows of A by 32 rows of B, k <= 64, by a CTA of 512 threads.  The
// digits of both operands lie in shared memory as FP16 integers; those of B
// one under the other, so that digit i of A times digits 0 .. S - 1 - i of B is
// one MMA of N = 32 (S - i) columns, and the accumulator columns 32 l + c of
// tensor memory are the sums of level l = i + j: S MMAs per 16 entries of k do
// all S (S + 1) / 2 digit products.  The sums are exact as in split_gemm.cuh
// (the same terms, below 2^24 in units of 1), and so are the results bit for
// bit.  Two sets of B and of accumulators: while the tensor cores run a tile,
// the CTA combines the one before and cuts the digits of the next.
#pragma once
#include "split_gemm.cuh"

namespace mrcm {
namespace {

constexpr int kTcM = 128, kTcN = 32, kTcThreads = 512;
constexpr int kTcOut = kTcM * kTcN / kTcThreads;     // outputs per thread

// Shared-memory operands, K-major, no swizzle: 8 rows x 16 bytes contiguous,
// 128 bytes between row groups, kStep bytes between 8-entry columns of k (64
// more than the rows need, which spreads the stores over the banks).
template <int S>
struct TcSmem {
    static constexpr int kStepA = kTcM * 16 + 64, kStepB = S * kTcN * 16 + 64;
    __align__(16) unsigned char A[S][8 * kStepA];
    __align__(16) unsigned char B[2][8 * kStepB];
    int ea[kTcM], eb[4][kTcN];           // (eb: by tile, a tile ahead of the one being combined)
    __align__(16) int sk[64];            // powers of two of the k (A's entries; B's the inverse ones)
    __align__(8) unsigned long long bar[2];
    unsigned int tmem;
};

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long tc_desc(unsigned addr, int kstep) {
    return (unsigned long long)((addr >> 4) & 0x3fffu) | (unsigned long long)((kstep >> 4) & 0x3fff) << 16 |
           (unsigned long long)(128 >> 4) << 32 | 1ull << 46;
}
__device__ __forceinline__ void tc_mma(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc, bool acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"((unsigned)acc) : "memory");
}
// FP16 x FP16 -> FP32, both operands K-major, M = 128
__device__ __forceinline__ unsigned tc_idesc(int n) { return 1u << 4 | (unsigned)(n >> 3) << 17 | (kTcM >> 4) << 24; }

// The .sync.aligned forms of tcgen05 want every lane of the warp together; what
// comes before them here (predicated loads and stores, loops with early ends)
// may leave a warp split, so each is preceded by a __syncwarp().
//
// Tensor memory for the two accumulator sets, and the barriers; by the whole CTA.
template <int S>
__device__ __forceinline__ void tc_begin(TcSmem<S>& sm) {
    if (threadIdx.x < 32) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem)),
                     "r"(2 * S * kTcN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&sm.bar[b])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// The digits of row `row` of an operand (eight lanes per row, lane j entries
// 8 j .. 8 j + 7 in v, times 2^(SIGN sk)) to dst + digit * dig.
template <int S, int SIGN, class T>
__device__ __forceinline__ void tc_stage(unsigned char* dst, int dig, int kstep, int* e, int row, const T (&v)[8],
                                         const int* sk) {
    const int j = threadIdx.x & 7;
    int ex[8], E = kZeroExp;
#pragma unroll
    for (int i = 0; i < 8; i += 4) {
        const int4 s = *reinterpret_cast<const int4*>(sk + 8 * j + i);
        ex[i] = scaled_exponent(v[i], SIGN * s.x);
        ex[i + 1] = scaled_exponent(v[i + 1], SIGN * s.y);
        ex[i + 2] = scaled_exponent(v[i + 2], SIGN * s.z);
        ex[i + 3] = scaled_exponent(v[i + 3], SIGN * s.w);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) E = max(E, ex[i]);
#pragma unroll
    for (int w = 1; w < 8; w <<= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, w));
    if (j == 0) e[row] = common_exponent<T>(E);
    unsigned d[4][S];
#pragma unroll
    for (int p = 0; p < 4; ++p) digit_pair<S>(v[2 * p], v[2 * p + 1], E - ex[2 * p], E - ex[2 * p + 1], d[p]);
    unsigned char* at = dst + j * kstep + row * 16;
#pragma unroll
    for (int s = 0; s < S; ++s)
        *reinterpret_cast<uint4*>(at + s * dig) = make_uint4(d[0][s], d[1][s], d[2][s], d[3][s]);
}
template <int S, class T>
__device__ __forceinline__ void tc_stage_a(TcSmem<S>& sm, int row, const T (&v)[8]) {
    tc_stage<S, 1>(&sm.A[0][0], 8 * TcSmem<S>::kStepA, TcSmem<S>::kStepA, sm.ea, row, v, sm.sk);
}
template <int S, class T>
__device__ __forceinline__ void tc_stage_b(TcSmem<S>& sm, int tile, int row, const T (&v)[8]) {
    tc_stage<S, -1>(&sm.B[tile & 1][0], kTcN * 16, TcSmem<S>::kStepB, sm.eb[tile & 3], row, v, sm.sk);
}
// Makes the CTA's staged digits visible to the tensor cores; then thread 0
// may issue.  True (all threads) when stop holds on any thread.
__device__ __forceinline__ bool tc_staged(bool stop = false) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    return __syncthreads_or(stop);
}
// All digit products of a tile (kn entries of k), by one thread.
template <int S>
__device__ __forceinline__ void tc_issue(TcSmem<S>& sm, int tile, int kn) {
    const int buf = tile & 1;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned d = sm.tmem + buf * S * kTcN;
    for (int k = 0; k < kn; k += 16) {
        const unsigned long long b = tc_desc(smem_u32(&sm.B[buf][0]) + (k >> 3) * TcSmem<S>::kStepB, TcSmem<S>::kStepB);
#pragma unroll 1
        for (int i = 0; i < S; ++i) {
            const unsigned long long a =
                tc_desc(smem_u32(&sm.A[i][0]) + (k >> 3) * TcSmem<S>::kStepA, TcSmem<S>::kStepA);
            tc_mma(d + kTcN * i, a, b, tc_idesc(kTcN * (S - i)), k > 0 || i > 0);
        }
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(&sm.bar[buf])) : "memory");
}
// Waits for a tile, at most `limit` blocking polls (and at most kTcPolls: a
// poll may suspend the warp for many microseconds) after one that does not
// block.  False, on every lane of the warp, when the tile did not come.
constexpr int kTcPolls = 1 << 16;
template <int S>
__device__ __forceinline__ bool tc_wait(TcSmem<S>& sm, int tile, long long limit) {
    const unsigned bar = smem_u32(&sm.bar[tile & 1]), parity = (tile >> 1) & 1;
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    const int polls = (int)min(limit, (long long)kTcPolls);
    for (int spin = 0; spin < polls && !done; ++spin)
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    const bool all = __all_sync(0xffffffffu, done);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return all;
}
// Row and first column of this thread's outputs of a tile.
__device__ __forceinline__ int tc_row() { return threadIdx.x & 127; }
__device__ __forceinline__ int tc_col() { return (threadIdx.x >> 7) * kTcOut; }
// Entries tc_col() + 4 q .. + 3 of this thread's row, from the level sums.
template <int S>
__device__ __forceinline__ void tc_outputs(TcSmem<S>& sm, int tile, int q, typename SplitAcc<S>::T (&out)[4]) {
    const int c = tc_col() + 4 * q;
    const unsigned t = sm.tmem + (tile & 1) * S * kTcN + c + ((threadIdx.x & 96) << 16);
    float n[S][4];
    __syncwarp();
#pragma unroll
    for (int l = 0; l < S; ++l)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(n[l][0]), "=f"(n[l][1]), "=f"(n[l][2]), "=f"(n[l][3]) : "r"(t + kTcN * l));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    const int ea = sm.ea[tc_row()];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        float x[S];
#pragma unroll
        for (int l = 0; l < S; ++l) x[l] = n[l][u];
        out[u] = combine_levels(x, ea, sm.eb[tile & 3][c + u]);
    }
}
// Frees the tensor memory; by the whole CTA.  ok: this warp saw every tile it
// waited for.  Where one did not, the tiles still in flight (up to `last`, the
// last one issued) are waited for first, again with a limit: the tensor cores
// read this CTA's shared memory and write its tensor memory until then.
template <int S>
__device__ __forceinline__ void tc_end(TcSmem<S>& sm, bool ok, int last, int* status) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) atomicOr(status, kStatusTimeout);
        for (int tile = max(last - 1, 0); tile <= last; ++tile) tc_wait(sm, tile, kTcPolls);
        __syncthreads();
    }
    if (threadIdx.x < 32) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem), "r"(2 * S * kTcN));
    }
}

}  // namespace
}  // namespace mrcm
