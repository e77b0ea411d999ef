// Matrix products of FP64 accuracy on the FP16 tensor cores.
//
// GB300's FP64 pipe retires two multiply-adds per SM and clock, its tensor
// cores about five hundred FP16 ones (mma.sync m16n8k16).  A product of FP64
// matrices is therefore formed from integer digits (the error-free splitting
// of Ootomo, Ozaki and Yokota, "DGEMM on integer matrix multiplication unit",
// IJHPCA 2024, here with FP16 operands and FP32 accumulators holding
// integers): within one chunk of k (kChunkK entries) a row of A is written
// as 2^(Ea - 1085) V, V an integer of at most 63 bits and a sign, and V as
// S = 8 digits of 8 bits, d in [-128, 128]; a row of B (a column of the
// product's right factor, read along k) likewise.  Digit products are exact
// in FP16 x FP16 -> FP32, and all products of one level l = i + j are summed
// in one accumulator: at most 8 x 64 terms of magnitude 2^14, below 2^24, so
// every sum is an exact integer.  Levels past S - 1 are dropped (below
// 2^-62 of the largest product); 36 products of digits remain.  At the end
// of a chunk the eight integers of an output are combined in 64-bit integer
// arithmetic, rounded once to FP64 and added to the running sum.
//
// Accuracy.  An operand is exact unless it is more than 2^10 below the largest
// entry of its row in the chunk; then it is cut off at 2^-62 of that entry.
// With the dropped levels the error of a chunk's sum is below a few 2^-62
// max_k |a_k| max_k |b_k|, plus the one rounding (an FP64 loop: 2^-53 of every
// partial sum).  Where the terms themselves are as large as that product of
// maxima, this is the smaller error; where a and b are large at different k
// (a = (1, 2^-20), b = (2^-20, 1): 3e-13 of the sum) it would be the larger.
// The operands of the merges and leaves are graded like that by the contrast
// of the permeability, but by factors that are known: the column k of one
// operand goes as 1 / d_k, the row k of the other as d_k, with d = D^1/2 of
// the interface segments, or the square root of a diagonal of an inverse.  So
// each product takes the power of two nearest below d_k (sc), which the cutting
// adds to the exponents: no rounding, and both rows are level in k.  (K
// contrast 1e11, one-face segments, node maps against quadruple precision,
// entries over the roots of their diagonals: without the powers 7.5e-15 to
// 1.2e-14, with them and in FMA loops 1e-16 to 1.6e-15.  They cost up to 0.6%
// of an FP64 step and 1% of a mixed one, whose cutting is the larger part.)
//
// S = 4 (31 bits, 10 digit products) serves the FP32 merges of the mixed
// form: more than an FP32 operand's 24 bits of the largest entry, sums
// exact up to the one FP32 rounding per chunk.
//
// Work split.  A CTA of eight warps forms a 64 x 32 tile of the product; a
// warp a 32 x 8 part of it with all levels in registers (8 x 8
// accumulators), so that a k-step of 16 loads 20 fragments from shared
// memory for 72 MMAs.  The digits are cut by the CTA that uses them (about
// 25 integer instructions per entry, hidden behind the other resident CTA's
// MMAs: two CTAs of 97 KB and 16 warps per SM); digits kept in global memory
// would cost 16 bytes per entry and more L2 bandwidth than the FP64 entries
// do.  Shared memory holds a digit row's 64 entries in 8 units of 16 bytes,
// unit u at u ^ (row % 8): the eight rows an ldmatrix reads and the four rows
// a staging warp writes then lie in distinct banks.
//
// Measured (one GB300, all heights): 4096^2 X 14.46 -> 2.37 ms, R 12.65 -> 2.49
// against FP64 FMA loops at 97 and 92% of the FP64 peak; box 128x128x64 X
// 27.5 -> 4.7, R 23.6 -> 5.6.  Seven digits in four warps per CTA were as fast
// (2.25 and 2.67 ms) and less exact: node maps against quadruple precision 2.1e-15
// at alpha = 100 (now 1.9e-16, the FMA loops 2.4e-16), boxes against a dense
// FP64 solution 6.3e-13 (now 2.6e-13, the FMA loops 2.7e-13).
#pragma once
#include <cuda_fp16.h>
#include "mrcm_internal.h"

namespace mrcm {
namespace {

constexpr int kChunkK = 64;              // k entries staged (and scaled) at a time
constexpr int kTileM = 64, kTileN = 32;  // product tile of a CTA
constexpr int kGemmThreads = 256, kGemmWarps = kGemmThreads / 32;

template <class T> struct Slices { static constexpr int S = 8; };
template <> struct Slices<float> { static constexpr int S = 4; };

template <int S>
struct SplitSmem {
    __half A[S][kTileM][kChunkK];
    __half B[S][kTileN][kChunkK];
    int ea[kTileM], eb[kTileN];          // largest biased exponent of each row in the chunk
    __align__(8) int sk[kChunkK];        // powers of two of the chunk's k (where a strip keeps them)
};
// Position of entry k of a staged row.
__device__ __forceinline__ int swizzled(int row, int k) { return ((k >> 3) ^ (row & 7)) * 8 + (k & 7); }

// Staging: a pass of the CTA covers 32 rows, eight lanes per row, entries
// 16 i + 2 q and 16 i + 2 q + 1 (i < kLaneK / 2) on lane q, so that the lanes of
// a row read 128 consecutive bytes.
constexpr int kLaneK = kChunkK / 8;      // entries of a row per lane
constexpr int kPassRows = kGemmThreads / 8;
__device__ __forceinline__ int stage_q() { return threadIdx.x & 7; }
__device__ __forceinline__ int stage_slot() {          // row of this lane within a pass
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    return 8 * (warp >> 1) + (warp & 1) + 2 * (lane >> 3);
}
__device__ __forceinline__ int lane_k(int i) { return 16 * (i >> 1) + 2 * stage_q() + (i & 1); }

// The warp's 32 x 8 part of a tile: output r of the 16 x 8 tile mt lies in
// row out_row(mt, r), column out_col(r).
__device__ __forceinline__ int warp_m0() { return ((threadIdx.x >> 5) >> 2) * 32; }
__device__ __forceinline__ int warp_n0() { return ((threadIdx.x >> 5) & 3) * 8; }
__device__ __forceinline__ int out_row(int mt, int r) {
    return warp_m0() + 16 * mt + ((threadIdx.x & 31) >> 2) + 8 * (r >> 1);
}
__device__ __forceinline__ int out_col(int r) { return warp_n0() + 2 * (threadIdx.x & 3) + (r & 1); }

// Exponents of rows without numbers, and of rows with an infinity or a NaN.
constexpr int kZeroExp = -(1 << 14), kNonFiniteExp = 1 << 14;
__device__ __forceinline__ unsigned high_word(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ unsigned high_word(float x) { return __float_as_uint(x); }
__device__ __forceinline__ int exponent_field(double x) { return (int)((high_word(x) >> 20) & 0x7ffu); }
__device__ __forceinline__ int exponent_field(float x) { return (int)((high_word(x) >> 23) & 0xffu); }
// Biased exponent of x 2^s, |s| <= 512 (FP32: 64; the square root of a number's
// range).  Zeros, and subnormals with them, must lie 63 (31) places below
// every number of a row: an FP64 zero's exponent is s itself, below the 640
// that common_exponent() asks of a row; FP32 has no such room and takes a
// select.
__device__ __forceinline__ int scaled_exponent(double x, int s) { return exponent_field(x) + s; }
__device__ __forceinline__ int scaled_exponent(float x, int s) {
    const int f = exponent_field(x);
    return f + (f == 0 ? kZeroExp : s);
}
// floor(log2(x^(1/2))), 0 for what has none: the power of two that levels the
// products with an inverse of diagonal x.
template <class T>
__device__ __forceinline__ int half_exponent(T x) {
    const int f = exponent_field(x);
    return (f == 0 || f == (sizeof(T) == 8 ? 2047 : 255)) ? 0 : (f - (sizeof(T) == 8 ? 1023 : 127)) >> 1;
}
// floor(log2(x)) of a positive normal x
__device__ __forceinline__ int whole_exponent(double x) { return exponent_field(x) - 1023; }

// The digits of |x|, d binary places below the row's exponent, one byte each
// (the leading digit as it is, in [0, 128]; the others + 128), the last digit
// in the lowest byte.
template <int S>
__device__ __forceinline__ unsigned long long digit_bytes(double x, int d) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned top = (hi & 0xfffffu) | 0x100000u;
    if (S == 4) return (__funnelshift_l(lo, top, 10) >> min(d, 31)) + 0x00808080u;    // the upper 31 bits alone
    const unsigned long long m = ((unsigned long long)top << 42) | ((unsigned long long)lo << 10);
    return (m >> min(d, 63)) + 0x0080808080808080ull;
}
template <int S>
__device__ __forceinline__ unsigned digit_bytes(float x, int d) {       // S = 4
    const unsigned b = __float_as_uint(x);
    return ((((b & 0x7fffffu) | 0x800000u) << 7) >> min(d, 31)) + 0x00808080u;
}

// The digits of two entries of a row as FP16 pairs (the layout of an MMA
// operand register), dx and dy places below their row's exponent.
template <int S, class T>
__device__ __forceinline__ void digit_pair(T x, T y, int dx, int dy, unsigned (&out)[S]) {
    const unsigned ha = high_word(x), hb = high_word(y);
    const unsigned long long ua = digit_bytes<S>(x, dx), ub = digit_bytes<S>(y, dy);
    // the signs as FP16 factors sigma = +-1, and -1152 sigma, -1024 sigma: a
    // digit is (1024 + byte) sigma - (1024 or 1152) sigma, exact
    const unsigned sg = __byte_perm(ha, hb, 0x7030);
    const unsigned one = (sg & 0x80008000u) | 0x3c003c00u;
    const unsigned off = (sg & 0x80008000u) ^ 0xe480e480u, off0 = (sg & 0x80008000u) ^ 0xe400e400u;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const int byte = S - 1 - s, b = byte & 3;    // digit s (0: the leading one)
        const unsigned wa = (unsigned)(byte >= 4 ? ua >> 32 : ua), wb = (unsigned)(byte >= 4 ? ub >> 32 : ub);
        const unsigned w = (__byte_perm(wa, wb, b | (4 + b) << 8) & 0x00ff00ffu) | 0x64006400u;   // 1024 + byte
        const __half2 h = __hfma2(*reinterpret_cast<const __half2*>(&w), *reinterpret_cast<const __half2*>(&one),
                                  *reinterpret_cast<const __half2*>(s == 0 ? &off0 : &off));
        out[s] = *reinterpret_cast<const unsigned*>(&h);
    }
}
// The biased FP64 exponent of a row from the largest exponent of its entries:
// below 2^-383 (FP64) a row counts as zero, and from 2^512 (FP32: 2^64) on,
// where an infinity or NaN lies whatever its power of two, as not finite.
// Scaled entries go as the square root of the data's range and stay inside.
template <class T>
__device__ __forceinline__ int common_exponent(int E) {
    if (sizeof(T) == 8) return E < 640 ? kZeroExp : (E >= 1535 ? kNonFiniteExp : E);
    return E >= 191 ? kNonFiniteExp : E + 896;
}

// Writes the digit pairs of this lane's entries of one row (eight lanes),
// entry i times 2^(SIGN s[i]).
template <int S, int SIGN, int ROWS, class T>
__device__ __forceinline__ void stage_row(__half (*dst)[ROWS][kChunkK], int* e, int row, int kn, const T (&v)[kLaneK],
                                          const int (&s)[kLaneK]) {
    int ex[kLaneK], E = kZeroExp;
#pragma unroll
    for (int i = 0; i < kLaneK; ++i) {
        ex[i] = scaled_exponent(v[i], SIGN * s[i]);
        E = max(E, ex[i]);
    }
#pragma unroll
    for (int w = 1; w < 8; w <<= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, w));
    if (stage_q() == 0) e[row] = common_exponent<T>(E);
    const int kend = (kn + 15) & ~15;
#pragma unroll
    for (int i = 0; i < kLaneK; i += 2) {
        if (8 * i >= kend) break;
        unsigned d[S];
        digit_pair<S>(v[i], v[i + 1], E - ex[i], E - ex[i + 1], d);
#pragma unroll
        for (int j = 0; j < S; ++j) *reinterpret_cast<unsigned*>(&dst[j][row][swizzled(row, lane_k(i))]) = d[j];
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

// The digit products of the staged chunk: acc[l][mt] += level l of the warp's
// 16 x 8 tile mt.
template <int S>
__device__ __forceinline__ void chunk_mma(const SplitSmem<S>& sm, int kn, float (&acc)[S][2][4]) {
    const int lane = threadIdx.x & 31;
    const int arow = warp_m0() + (lane & 15), brow = warp_n0() + (lane & 7);
#pragma unroll
    for (int l = 0; l < S; ++l)
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[l][mt][r] = 0.f;
#pragma unroll 1
    for (int k0 = 0; k0 < kn; k0 += 16) {
        const int ak = swizzled(arow, k0 + (lane >> 4) * 8), bk = swizzled(brow, k0 + ((lane >> 3) & 1) * 8);
        unsigned b[S / 2][4];                     // two digits of B per load
#pragma unroll
        for (int j = 0; j < S / 2; ++j) ldmatrix_x4(b[j], &sm.B[2 * j + (lane >> 4)][brow][bk]);
#pragma unroll
        for (int i = 0; i < S; ++i) {
            unsigned a[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) ldmatrix_x4(a[mt], &sm.A[i][arow + 16 * mt][ak]);
#pragma unroll
            for (int j = 0; j < S - i; ++j)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
                    mma_f16(acc[i + j][mt], a[mt], b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]);
        }
    }
}

// One output of a chunk in FP64 from its level sums and the exponents of its
// row and column: v + w 2^-14 in units of 2^-42 of a leading digit product,
// both exact integers; v is moved up by as many bits (at most 14) as it
// leaves free, so that w enters where it matters, and the sum is rounded once.
__device__ __forceinline__ double combine_levels(const float (&n)[8], int ea, int eb) {
    const int w = (__float2int_rn(n[6]) << 8) + __float2int_rn(n[7]);
    const int m = (__float2int_rn(n[4]) << 8) + __float2int_rn(n[5]);
    const int h = (__float2int_rn(n[2]) << 8) + __float2int_rn(n[3]);
    const int t = (__float2int_rn(n[0]) << 8) + __float2int_rn(n[1]);
    const long long v = ((long long)(t << 2) << 32) + (long long)h * 262144 + (long long)m * 4;    // |v| < 2^63
    const int up = min(14, max(__clzll((long long)((unsigned long long)v ^ (unsigned long long)(v >> 63))) - 2, 0));
    const long long x = (long long)((unsigned long long)v << up) + (w >> (14 - up));
    const unsigned long long s = (unsigned long long)(x >> 63), u = ((unsigned long long)x ^ s) - s;
    const int lz = __clzll((long long)u);
    // leading bit to bit 62, rounded at bit 10; the carry of the rounding
    // moves into the exponent field
    const unsigned long long mant = ((u << ((lz - 1) & 63)) + 0x200ull) >> 10;
    const int be = ea + eb - lz - 1014 - up;
    unsigned long long bits = ((unsigned long long)(be - 1) << 52) + mant;
    if (u == 0 || be <= 0) bits = 0;                                          // zero or underflow
    if (be >= 2047) bits = 0x7ff0000000000000ull;                             // overflow
    if (max(ea, eb) >= kNonFiniteExp) bits = 0x7ff8000000000000ull;           // an infinity or NaN among the entries
    return __longlong_as_double((long long)(bits | (s & 0x8000000000000000ull)));
}
// The same for S = 4 in FP32 (the levels are exact integers; one rounding
// per step of the Horner sum).
__device__ __forceinline__ float pow2f(int e) {         // 2^e, kept within the normal FP32 range, 0 below it
    return __int_as_float(e < -126 ? 0 : (min(e, 127) + 127) << 23);
}
__device__ __forceinline__ float combine_levels(const float (&n)[4], int ea, int eb) {
    const float v = fmaf(fmaf(fmaf(n[0], 256.f, n[1]), 256.f, n[2]), 256.f, n[3]);
    const int e = ea + eb - 2082;
    if ((unsigned)(e + 126) <= 253u) return v * __int_as_float((e + 127) << 23);
    // 2^e as two factors, so that v 2^e itself decides whether it leaves the range
    // (a row of zeros: e far below); beyond that an infinity or NaN in a row
    if (max(ea, eb) >= kNonFiniteExp) return __int_as_float(0x7fc00000);
    const int h = max(e, 2 * kZeroExp) >> 1;
    return v * pow2f(h) * pow2f(max(e, 2 * kZeroExp) - h);
}
// x as a double by integer operations (a conversion instruction holds the
// FP64 pipe like an FP64 instruction); FP32 subnormals count as zero.
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    const unsigned hi = e == 0 ? 0u : (e == 255 ? 0x7ff00000u : (e + 896u) << 20) | ((b & 0x7fffffu) >> 3);
    return __hiloint2double((int)(hi | (b & 0x80000000u)), e == 0 ? 0 : (int)(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }
template <int S> struct SplitAcc { using T = double; };
template <> struct SplitAcc<4> { using T = float; };

// This lane's entries of a row from p on (nullptr: zeros), through the index
// registers ix when the row is gathered.
template <bool GATHER, class T>
__device__ __forceinline__ void load_row(T (&v)[kLaneK], const T* p, const int (&ix)[kLaneK], int kn) {
#pragma unroll
    for (int i = 0; i < kLaneK; ++i) v[i] = (p && lane_k(i) < kn) ? p[GATHER ? ix[i] : lane_k(i)] : (T)0;
}
template <bool ON>
__device__ __forceinline__ void load_index(int (&ix)[kLaneK], const int* idx, int kn) {
#pragma unroll
    for (int i = 0; i < kLaneK; ++i) ix[i] = (ON && lane_k(i) < kn) ? idx[lane_k(i)] : 0;
}

// The powers of this lane's entries of the chunk.
__device__ __forceinline__ void load_scale(int (&s)[kLaneK], const int* sk) {
#pragma unroll
    for (int i = 0; i < kLaneK; i += 2) {
        const int2 x = *reinterpret_cast<const int2*>(sk + lane_k(i));
        s[i] = x.x;
        s[i + 1] = x.y;
    }
}

// The warp's part of sum_k A(row, k) B(col, k), k < K (K >= 1), at row
// out_row(mt, r), column out_col(r).  arow(row) / brow(col): pointer to the
// operand's row (nullptr: zeros), entry k at [k], or at [idx[k]] where AG /
// BG say that the operand is gathered.  sc(k): A's column k is cut as
// A 2^sc(k), B's as B 2^-sc(k).
template <int S, class T, bool AG, bool BG, class ASrc, class BSrc, class Scale>
__device__ __forceinline__ void split_product(SplitSmem<S>& sm, int K, const int* idx, ASrc&& arow, BSrc&& brow,
                                              Scale&& sc, typename SplitAcc<S>::T (&sum)[2][4]) {
    const int row = stage_slot();
    const T *pa[2] = {arow(row), arow(row + kPassRows)}, *pb = brow(row);
#pragma unroll 1
    for (int k0 = 0; k0 < K; k0 += kChunkK) {
        const int kn = min(kChunkK, K - k0);
        {
            int ix[kLaneK], s[kLaneK];
            load_index<AG || BG>(ix, idx + k0, kn);
            const int power = threadIdx.x < kn ? sc(k0 + (int)threadIdx.x) : 0;
            // every row's entries in flight together
            T va[2][kLaneK], vb[kLaneK];
#pragma unroll
            for (int p = 0; p < 2; ++p) load_row<AG>(va[p], pa[p] ? pa[p] + (AG ? 0 : k0) : nullptr, ix, kn);
            load_row<BG>(vb, pb ? pb + (BG ? 0 : k0) : nullptr, ix, kn);
            if (threadIdx.x < kChunkK) sm.sk[threadIdx.x] = power;
            __syncthreads();                          // the previous chunk's digits are read
            load_scale(s, sm.sk);
#pragma unroll
            for (int p = 0; p < 2; ++p) stage_row<S, 1>(sm.A, sm.ea, row + p * kPassRows, kn, va[p], s);
            stage_row<S, -1>(sm.B, sm.eb, row, kn, vb, s);
        }
        __syncthreads();
        float acc[S][2][4];
        chunk_mma<S>(sm, kn, acc);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float n[S];
#pragma unroll
                for (int l = 0; l < S; ++l) n[l] = acc[l][mt][r];
                const auto c = combine_levels(n, sm.ea[out_row(mt, r)], sm.eb[out_col(r)]);
                sum[mt][r] = k0 ? sum[mt][r] + c : c;
            }
    }
}

// The same for a strip of the product with K <= kChunkK: 64 rows of A, whose
// digits are cut once, by the 32-column tiles t0 <= t < t1.  A tile's rows of
// B and the values pre(t, row, column) that its epilogue needs are loaded
// while the products of the tile before run; epi(t, row, column, product,
// pre) receives every entry.
template <int S, bool AG, bool BG, class ASrc, class BSrc, class Scale, class Pre, class Epi>
__device__ __forceinline__ void strip_product(SplitSmem<S>& sm, int K, const int* idx, int t0, int t1, ASrc&& arow,
                                              BSrc&& brow, Scale&& sc, Pre&& pre, Epi&& epi) {
    const int row = stage_slot();
    const int power = threadIdx.x < K ? sc(threadIdx.x) : 0;          // in flight with the rows
    int ix[kLaneK];
    load_index<AG || BG>(ix, idx, K);
    double vb[kLaneK];
    load_row<BG>(vb, brow(t0, row), ix, K);
    {
        double va[2][kLaneK];
#pragma unroll
        for (int p = 0; p < 2; ++p) load_row<AG>(va[p], arow(row + p * kPassRows), ix, K);
        if (threadIdx.x < kChunkK) sm.sk[threadIdx.x] = power;
        __syncthreads();
        int s[kLaneK];
        load_scale(s, sm.sk);
#pragma unroll
        for (int p = 0; p < 2; ++p) stage_row<S, 1>(sm.A, sm.ea, row + p * kPassRows, K, va[p], s);
    }
    for (int t = t0; t < t1; ++t) {
        if (t > t0) __syncthreads();                  // the tile before is done with sm.B
        {
            int s[kLaneK];
            load_scale(s, sm.sk);
            stage_row<S, -1>(sm.B, sm.eb, row, K, vb, s);
        }
        __syncthreads();
        if (t + 1 < t1) load_row<BG>(vb, brow(t + 1, row), ix, K);
        double old[2][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int r = 0; r < 4; ++r) old[mt][r] = pre(t, out_row(mt, r), out_col(r));
        float acc[S][2][4];
        chunk_mma<S>(sm, K, acc);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float n[S];
#pragma unroll
                for (int l = 0; l < S; ++l) n[l] = acc[l][mt][r];
                const int i = out_row(mt, r), j = out_col(r);
                epi(t, i, j, widen(combine_levels(n, sm.ea[i], sm.eb[j])), old[mt][r]);
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
__device__ __forceinline__ int quad_exponent(const T (&v)[4], const int (&s)[4], int sign, int (&ex)[4]) {
    int E = kZeroExp;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        ex[i] = scaled_exponent(v[i], sign * s[i]);
        E = max(E, ex[i]);
    }
    E = max(E, __shfl_xor_sync(0xffffffffu, E, 1));
    return max(E, __shfl_xor_sync(0xffffffffu, E, 2));
}
// k of a lane's four entries of a fragment row
__device__ __forceinline__ int frag_k(int i) { return 2 * (threadIdx.x & 3) + (i & 1) + 8 * (i >> 1); }
// at(row, k): the operand's entry; entries i times 2^(sign s[i])
template <int S, class T, class At>
__device__ __forceinline__ void load_frag_a(FragA<S>& f, const int (&s)[4], int sign, At&& at) {
    const int g = (threadIdx.x & 31) >> 2;
    T v[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[h][i] = at(g + 8 * h, frag_k(i));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        int ex[4];
        const int E = quad_exponent(v[h], s, sign, ex);
        (h ? f.e1 : f.e0) = common_exponent<T>(E);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            unsigned d[S];
            digit_pair<S>(v[h][2 * p], v[h][2 * p + 1], E - ex[2 * p], E - ex[2 * p + 1], d);
#pragma unroll
            for (int j = 0; j < S; ++j) f.d[j][h + 2 * p] = d[j];
        }
    }
}
// at(col, k)
template <int S, class T, class At>
__device__ __forceinline__ void load_frag_b(FragB<S>& f, const int (&s)[4], int sign, At&& at) {
    const int g = (threadIdx.x & 31) >> 2;
    T v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = at(g, frag_k(i));
    int ex[4];
    const int E = quad_exponent(v, s, sign, ex);
    f.e = common_exponent<T>(E);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        unsigned d[S];
        digit_pair<S>(v[2 * p], v[2 * p + 1], E - ex[2 * p], E - ex[2 * p + 1], d);
#pragma unroll
        for (int j = 0; j < S; ++j) f.d[j][p] = d[j];
    }
}
// out[r]: row g + 8 (r / 2), column 2 t + r % 2 of the 16 x 8 product, of whose
// rows the first `rows` are wanted (0 past the eighth where there are no more)
template <int S>
__device__ __forceinline__ void frag_product(const FragA<S>& a, const FragB<S>& b, typename SplitAcc<S>::T (&out)[4],
                                             int rows = 16) {
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
    const int eb[2] = {__shfl_sync(0xffffffffu, b.e, 8 * t), __shfl_sync(0xffffffffu, b.e, 8 * t + 4)};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        out[r] = 0;
        if (r >= 2 && rows <= 8) continue;
        float n[S];
#pragma unroll
        for (int l = 0; l < S; ++l) n[l] = acc[l][r];
        out[r] = combine_levels(n, r < 2 ? a.e0 : a.e1, eb[r & 1]);
    }
}

}  // namespace
}  // namespace mrcm
