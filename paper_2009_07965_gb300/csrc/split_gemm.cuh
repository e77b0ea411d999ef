// Matrix products of FP64 accuracy on the FP16 tensor cores.
//
// GB300's FP64 pipe retires two multiply-adds per SM and clock, its tensor
// cores about five hundred FP16 ones (mma.sync m16n8k16).  A product of FP64
// matrices is therefore formed from integer digits (the error-free splitting
// of Ootomo, Ozaki and Yokota, "DGEMM on integer matrix multiplication unit",
// IJHPCA 2024, here with FP16 operands and FP32 accumulators holding
// integers): within one chunk of k (kChunkK entries) a row of A is written
// as 2^(Ea - 1076) V, V an integer of at most 54 bits and a sign, and V as
// S = 7 digits of 8 bits, d in [-128, 127] (|d_0| <= 64); a row of B (a column of the
// product's right factor, read along k) likewise.  Digit products are exact
// in FP16 x FP16 -> FP32, and all products of one level l = i + j are summed
// in one accumulator: at most 7 x 64 terms of magnitude 2^14, below 2^24, so
// every sum is an exact integer.  Levels past S - 1 are dropped (below
// 2^-54 of the largest product); 28 products of digits remain.  At the end
// of a chunk the seven integers of an output are combined in 64-bit integer
// arithmetic, rounded once to FP64 and added to the running sum.
//
// Against an FP64 fused multiply-add loop: operands are rounded to 2^-54 of
// the largest entry of their row in the chunk (an FP64 operand is exact, but
// every addition of the loop rounds), and only one rounding per 64 terms
// follows.
//
// S = 4 (30 bits, 10 digit products) serves the FP32 merges of the mixed
// form: more than an FP32 operand's 24 bits of the largest entry, sums
// exact up to the one FP32 rounding per chunk.
//
// Work split.  A CTA of four warps forms a 64 x 32 tile of the product; a
// warp a 32 x 16 part of it with all levels in registers (7 x 16
// accumulators), so that a k-step of 16 loads 21 fragments from shared
// memory for 112 MMAs.  The digits are cut by the CTA that uses them (about
// 30 integer instructions per entry, hidden behind the other resident CTA's
// MMAs: two CTAs of 97 KB per SM); digits kept in global memory would cost
// 14 bytes per entry and more L2 bandwidth than the FP64 entries do.
//
// Measured (4096^2 quarter-five-spot, all heights, one GB300): X 14.46 ->
// 2.29 ms, R 12.65 -> 2.75 ms against FP64 FMA loops at 97 and 92% of the
// FP64 peak; 7 to 9 TFLOP/s of FP64 products.  Tensor pipe 35% busy, stalls
// mostly on fixed latencies with two warps per scheduler.  Node maps against
// quadruple precision (sigma^2 = 1..4, alpha = 0.5..2): relative errors
// 4e-17..3e-16, those of the FMA loops to within 20%.
#pragma once
#include <cuda_fp16.h>
#include "mrcm_internal.h"

namespace mrcm {
namespace {

constexpr int kChunkK = 64;              // k entries staged (and scaled) at a time
constexpr int kTileM = 64, kTileN = 32;  // product tile of a CTA
constexpr int kGemmThreads = 128;
constexpr int kSmemStride = kChunkK + 8; // halves per staged row: 144 bytes, an odd number of 16-byte
                                         // units (ldmatrix rows and the digit stores hit distinct banks)

template <int S>
struct SplitSmem {
    __half A[S][kTileM][kSmemStride];
    __half B[S][kTileN][kSmemStride];
    int ea[kTileM], eb[kTileN];          // largest biased exponent of each row in the chunk
};

// The digits of |x| relative to the row exponent E, one byte each (the
// leading digit as it is, in [0, 128]; the others + 128), the last digit in
// the lowest byte.  S = 7 leaves 0x64 in the highest byte, the upper half of
// the FP16 number 1024 + byte.
__device__ __forceinline__ unsigned high_word(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ unsigned high_word(float x) { return __float_as_uint(x); }
__device__ __forceinline__ int exponent_bits(double x) { return __double2hiint(x) & 0x7ff00000; }
__device__ __forceinline__ int exponent_bits(float x) { return __float_as_int(x) & 0x7f800000; }
template <int S>
__device__ __forceinline__ unsigned long long digit_bytes(double x, int E) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int d = min(E - (int)((hi >> 20) & 0x7ffu), S == 7 ? 63 : 39);
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 34) | ((unsigned long long)lo << 2);
    if (S == 7) return (m >> d) + 0x6400808080808080ull;
    return (m >> (d + 24)) + 0x00808080ull;
}
template <int S>
__device__ __forceinline__ unsigned digit_bytes(float x, int E) {       // S = 4
    const unsigned b = __float_as_uint(x);
    return ((((b & 0x7fffffu) | 0x800000u) << 7) >> min(E - (int)((b >> 23) & 0xffu), 31)) + 0x00808080u;
}

// The digits of two entries of a row as FP16 pairs (the layout of an MMA
// operand register).
template <int S, class T>
__device__ __forceinline__ void digit_pair(T x, T y, int E, unsigned (&out)[S]) {
    const unsigned ha = high_word(x), hb = high_word(y);
    const unsigned long long ua = digit_bytes<S>(x, E), ub = digit_bytes<S>(y, E);
    // the signs as FP16 factors sigma = +-1, and -1152 sigma, -1024 sigma: a
    // digit is (1024 + byte) sigma - (1024 or 1152) sigma, exact
    const unsigned sg = __byte_perm(ha, hb, 0x7030);
    const unsigned one = (sg & 0x80008000u) | 0x3c003c00u;
    const unsigned off = (sg & 0x80008000u) ^ 0xe480e480u, off0 = (sg & 0x80008000u) ^ 0xe400e400u;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const int byte = S - 1 - s;              // digit s (0: the leading one)
        unsigned w;
        if (S == 7 && byte >= 4)
            w = __byte_perm((unsigned)(ua >> 32), (unsigned)(ub >> 32), (byte - 4) | 3 << 4 | byte << 8 | 7 << 12);
        else
            w = (__byte_perm((unsigned)ua, (unsigned)ub, byte | (4 + byte) << 8) & 0x00ff00ffu) | 0x64006400u;
        const __half2 h = __hfma2(*reinterpret_cast<const __half2*>(&w), *reinterpret_cast<const __half2*>(&one),
                                  *reinterpret_cast<const __half2*>(s == 0 ? &off0 : &off));
        out[s] = *reinterpret_cast<const unsigned*>(&h);
    }
}
// The biased FP64 exponent of a row from the largest exponent field of its
// entries (FP32's 255, an infinity or NaN, as 2047).
template <class T>
__device__ __forceinline__ int common_exponent(int E) {
    return sizeof(T) == 8 || E == 0 ? E : (E == 255 ? 2047 : E + 896);
}

// Writes the digit pairs (k, k + 1) of one row's 16 entries held by this
// lane (entries 8 i + 2 q and 8 i + 2 q + 1 of the chunk).
template <int S, int ROWS, class T>
__device__ __forceinline__ void stage_row(__half (*dst)[ROWS][kSmemStride], int* e, int row, int kn,
                                          const T (&v)[2 * kChunkK / 8]) {
    const int q = threadIdx.x & 3;
    int E = 0;
#pragma unroll
    for (int i = 0; i < 2 * kChunkK / 8; ++i) E = max(E, exponent_bits(v[i]));
    E = max(E, __shfl_xor_sync(0xffffffffu, E, 1));
    E = max(E, __shfl_xor_sync(0xffffffffu, E, 2));
    E = sizeof(T) == 8 ? E >> 20 : E >> 23;
    if (q == 0) e[row] = common_exponent<T>(E);
    const int kend = (kn + 15) & ~15;
#pragma unroll
    for (int i = 0; i < kChunkK / 8; ++i) {
        if (8 * i >= kend) break;
        unsigned d[S];
        digit_pair<S>(v[2 * i], v[2 * i + 1], E, d);
#pragma unroll
        for (int s = 0; s < S; ++s) *reinterpret_cast<unsigned*>(&dst[s][row][8 * i + 2 * q]) = d[s];
    }
}

__device__ __forceinline__ void ldmatrix_x4(unsigned (&r)[4], const __half* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The digit products of the staged chunk: acc[l][mt][nt] += level l of the
// warp's 16 x 8 tiles (mt, nt).
template <int S>
__device__ __forceinline__ void chunk_mma(const SplitSmem<S>& sm, int kn, float (&acc)[S][2][2][4]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int m0 = (warp >> 1) * 32, n0 = (warp & 1) * 16;
    const int arow = m0 + (lane & 15), acol = (lane >> 4) * 8;
    const int brow = n0 + (lane & 7) + (lane >> 4) * 8, bcol = ((lane >> 3) & 1) * 8;
#pragma unroll
    for (int l = 0; l < S; ++l)
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[l][mt][nt][r] = 0.f;
#pragma unroll 1
    for (int k0 = 0; k0 < kn; k0 += 16) {
        unsigned b[S][4];
#pragma unroll
        for (int j = 0; j < S; ++j) ldmatrix_x4(b[j], &sm.B[j][brow][k0 + bcol]);
#pragma unroll
        for (int i = 0; i < S; ++i) {
            unsigned a[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) ldmatrix_x4(a[mt], &sm.A[i][arow + 16 * mt][k0 + acol]);
#pragma unroll
            for (int j = 0; j < S - i; ++j)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt) mma_f16(acc[i + j][mt][nt], a[mt], b[j][2 * nt], b[j][2 * nt + 1]);
        }
    }
}

// One output of a chunk in FP64 from its level sums and the exponents of its
// row and column.
__device__ __forceinline__ double combine_levels(const float (&n)[7], int ea, int eb) {
    const int m = (__float2int_rn(n[4]) << 8) + __float2int_rn(n[5]);
    const int h = (__float2int_rn(n[2]) << 8) + __float2int_rn(n[3]);
    const int t = (__float2int_rn(n[0]) << 8) + __float2int_rn(n[1]);
    const long long low = (long long)m * 4 + ((__float2int_rn(n[6]) + 32) >> 6);
    const long long v = ((long long)(t << 2) << 32) + (long long)h * 262144 + low;      // |v| < 2^63
    const unsigned long long s = (unsigned long long)(v >> 63), u = ((unsigned long long)v ^ s) - s;
    const int lz = __clzll((long long)u);
    // leading bit to bit 62, rounded at bit 10; the carry of the rounding
    // moves into the exponent field
    const unsigned long long mant = ((u << (lz - 1)) + 0x200ull) >> 10;
    const int be = ea + eb - lz - 1014;
    unsigned long long bits = ((unsigned long long)(be - 1) << 52) + mant;
    if (u == 0 || be <= 0) bits = 0;                                          // zero or underflow
    if (be >= 2047) bits = 0x7ff0000000000000ull;                             // overflow
    if (ea == 2047 || eb == 2047) bits = 0x7ff8000000000000ull;               // an infinity or NaN among the entries
    return __longlong_as_double((long long)(bits | (s & 0x8000000000000000ull)));
}
// The same for S = 4 in FP32 (the levels are exact integers; one rounding
// per step of the Horner sum).
__device__ __forceinline__ float pow2f(int e) {         // 2^e, flushed to 0 / infinity outside the FP32 range
    return __int_as_float(e < -126 ? 0 : (e > 127 ? 0x7f800000 : (e + 127) << 23));
}
__device__ __forceinline__ float combine_levels(const float (&n)[4], int ea, int eb) {
    const float v = fmaf(fmaf(fmaf(n[0], 256.f, n[1]), 256.f, n[2]), 256.f, n[3]);
    const float f = v * pow2f(ea - 1041) * pow2f(eb - 1041);
    return (ea == 2047 || eb == 2047) ? __int_as_float(0x7fc00000) : f;
}
template <int S> struct SplitAcc { using T = double; };
template <> struct SplitAcc<4> { using T = float; };

// The 16 entries 8 i + 2 q (+ 1) of a row from p on (nullptr: zeros), through
// the index registers ix when the row is gathered.
template <bool GATHER, class T>
__device__ __forceinline__ void load_row(T (&v)[2 * kChunkK / 8], const T* p, const int (&ix)[2 * kChunkK / 8],
                                         int kn) {
    const int q = threadIdx.x & 3;
#pragma unroll
    for (int i = 0; i < 2 * kChunkK / 8; ++i) {
        const int k = 8 * (i >> 1) + 2 * q + (i & 1);
        v[i] = (p && k < kn) ? p[GATHER ? ix[i] : k] : (T)0;
    }
}

// The warp's part of sum_k A(row, k) B(col, k), k < K (K >= 1): sum[mt][nt][r] for
// row m0 + 16 mt + lane / 4 + 8 (r / 2), column n0 + 8 nt + 2 (lane % 4) +
// (r % 2).  arow(row) / brow(col): pointer to the operand's row (nullptr:
// zeros), entry k at [k], or at [idx[k]] where AG / BG say that the operand
// is gathered.
template <int S, class T, bool AG, bool BG, class ASrc, class BSrc>
__device__ __forceinline__ void split_product(SplitSmem<S>& sm, int K, const int* idx, ASrc&& arow, BSrc&& brow,
                                              typename SplitAcc<S>::T (&sum)[2][2][4]) {
    constexpr int kPer = 2 * kChunkK / 8;             // entries of a row per lane
    constexpr int kRows = kGemmThreads / 4;           // rows staged per pass
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane & 3, row = threadIdx.x >> 2;
    const int m0 = (warp >> 1) * 32, n0 = (warp & 1) * 16;
    const T *pa[kTileM / kRows], *pb[kTileN / kRows];
#pragma unroll
    for (int p = 0; p < kTileM / kRows; ++p) pa[p] = arow(row + p * kRows);
#pragma unroll
    for (int p = 0; p < kTileN / kRows; ++p) pb[p] = brow(row + p * kRows);
#pragma unroll 1
    for (int k0 = 0; k0 < K; k0 += kChunkK) {
        const int kn = min(kChunkK, K - k0);
        {
            int ix[kPer];
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int k = 8 * (i >> 1) + 2 * q + (i & 1);
                ix[i] = ((AG || BG) && k < kn) ? idx[k0 + k] : 0;
            }
            // every row's entries in flight together
            T va[kTileM / kRows][kPer], vb[kTileN / kRows][kPer];
#pragma unroll
            for (int p = 0; p < kTileM / kRows; ++p)
                load_row<AG>(va[p], pa[p] ? pa[p] + (AG ? 0 : k0) : nullptr, ix, kn);
#pragma unroll
            for (int p = 0; p < kTileN / kRows; ++p)
                load_row<BG>(vb[p], pb[p] ? pb[p] + (BG ? 0 : k0) : nullptr, ix, kn);
            if (k0) __syncthreads();                  // the previous chunk's digits are read
#pragma unroll
            for (int p = 0; p < kTileM / kRows; ++p) stage_row<S>(sm.A, sm.ea, row + p * kRows, kn, va[p]);
#pragma unroll
            for (int p = 0; p < kTileN / kRows; ++p) stage_row<S>(sm.B, sm.eb, row + p * kRows, kn, vb[p]);
        }
        __syncthreads();
        float acc[S][2][2][4];
        chunk_mma<S>(sm, kn, acc);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    float n[S];
#pragma unroll
                    for (int l = 0; l < S; ++l) n[l] = acc[l][mt][nt][r];
                    const auto c = combine_levels(n, sm.ea[m0 + 16 * mt + (lane >> 2) + 8 * (r >> 1)],
                                                  sm.eb[n0 + 8 * nt + 2 * (lane & 3) + (r & 1)]);
                    sum[mt][nt][r] = k0 ? sum[mt][nt][r] + c : c;
                }
    }
}

// ---------------------------------------------------------------------------
// Products of small matrices by one warp, operands cut straight into MMA
// fragments (no shared-memory staging of digits).  Lane (g, t) = (lane / 4,
// lane % 4) of an A fragment (16 x 16) holds rows g and g + 8, entries 2 t,
// 2 t + 1, 2 t + 8, 2 t + 9; of a B fragment (16 x 8) the same entries of
// column g.
template <int S>
struct FragA {
    unsigned d[S][4];
    int e0, e1;                 // exponents of rows g, g + 8
};
template <int S>
struct FragB {
    unsigned d[S][2];
    int e;                      // exponent of column g
};
template <class T>
__device__ __forceinline__ int quad_exponent(T a, T b, T c, T d) {
    int E = max(max(exponent_bits(a), exponent_bits(b)), max(exponent_bits(c), exponent_bits(d)));
    E = max(E, __shfl_xor_sync(0xffffffffu, E, 1));
    E = max(E, __shfl_xor_sync(0xffffffffu, E, 2));
    return sizeof(T) == 8 ? E >> 20 : E >> 23;
}
// at(row, k): the operand's entry
template <int S, class T, class At>
__device__ __forceinline__ void load_frag_a(FragA<S>& f, At&& at) {
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
    T v[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[h][i] = at(g + 8 * h, 2 * t + (i & 1) + 8 * (i >> 1));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int E = quad_exponent(v[h][0], v[h][1], v[h][2], v[h][3]);
        (h ? f.e1 : f.e0) = common_exponent<T>(E);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            unsigned d[S];
            digit_pair<S>(v[h][2 * p], v[h][2 * p + 1], E, d);
#pragma unroll
            for (int s = 0; s < S; ++s) f.d[s][h + 2 * p] = d[s];
        }
    }
}
// at(col, k)
template <int S, class T, class At>
__device__ __forceinline__ void load_frag_b(FragB<S>& f, At&& at) {
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
    T v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = at(g, 2 * t + (i & 1) + 8 * (i >> 1));
    const int E = quad_exponent(v[0], v[1], v[2], v[3]);
    f.e = common_exponent<T>(E);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        unsigned d[S];
        digit_pair<S>(v[2 * p], v[2 * p + 1], E, d);
#pragma unroll
        for (int s = 0; s < S; ++s) f.d[s][p] = d[s];
    }
}
// out[r]: row g + 8 (r / 2), column 2 t + r % 2 of the 16 x 8 product
template <int S>
__device__ __forceinline__ void frag_product(const FragA<S>& a, const FragB<S>& b, typename SplitAcc<S>::T (&out)[4]) {
    float acc[S][4];
#pragma unroll
    for (int l = 0; l < S; ++l)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[l][r] = 0.f;
#pragma unroll
    for (int i = 0; i < S; ++i)
#pragma unroll
        for (int j = 0; j < S - i; ++j) mma_f16(acc[i + j], a.d[i], b.d[j][0], b.d[j][1]);
    const int t = threadIdx.x & 3;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float n[S];
#pragma unroll
        for (int l = 0; l < S; ++l) n[l] = acc[l][r];
        out[r] = combine_levels(n, r < 2 ? a.e0 : a.e1, __shfl_sync(0xffffffffu, b.e, (2 * t + (r & 1)) * 4));
    }
}

}  // namespace
}  // namespace mrcm
