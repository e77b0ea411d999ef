// Inverses of small symmetric matrices inside a CTA: up to 16 x 16 by the
// lanes of one warp on the FP64 pipe, up to 64 x 64 by four or eight warps, 16
// rows at a time, with the products on the tensor cores (split_gemm.cuh).
//
// Both use the symmetric sweep operator: sweeping the indices K turns A_KK
// into -A_KK^-1, A_xK into A_xK A_KK^-1 and A_xy into A_xy - A_xK A_KK^-1 A_Ky
// (x, y outside K), symmetric throughout; all indices swept, -A^-1 is left.
// Only the lower triangle is kept.  No pivot search: the matrices are
// positive definite or quasi-definite, and the caller's test knows the sign
// every pivot must have.
#pragma once
#include "mrcm_internal.h"
#include "split_gemm.cuh"

namespace mrcm {
namespace {

constexpr int kPlane = 16;        // largest block swept by one warp

// Distribution of the lower triangle of a 16 x 16 block over GL lanes (8 or
// 16): lane l of 8 owns rows l and 15 - l, 17 entries, split over two lanes
// where there are 16.
template <int GL>
struct BlockSlots {
    static constexpr int kN = GL == 8 ? 17 : 9;
    int l, s0;
    __device__ __forceinline__ BlockSlots() {
        const int lane = threadIdx.x & (GL - 1);
        l = lane & 7;
        s0 = (lane >> 3) * kN;
    }
    __device__ __forceinline__ bool valid(int j) const { return s0 + j < 17; }
    __device__ __forceinline__ bool low(int j) const { return s0 + j <= l; }      // on row l (else row 15 - l)
    __device__ __forceinline__ int row(int j) const { return low(j) ? l : 15 - l; }
    __device__ __forceinline__ int colm(int j) const { return low(j) ? s0 + j : s0 + j - l - 1; }
};

// Sweeps every index of up to 32 / GL blocks at once (one warp, GL lanes per
// block).  e[]: the lane's entries on entry and exit; those that hold the next
// pivot's column go to shared memory as they are made (col: by pivot parity,
// the pivot itself in the last place; entries of no interest to a place past
// the block, so that no lane branches).  Per pivot 3 FP64 instructions for
// the reciprocal, 2 to scale the lane's rows and one per entry (an FP64
// instruction holds its scheduler's pipe for 64 cycles: these are the cost).
// nb: the lane's block (0: none), steps: the largest block of the warp;
// pivot_ok(p, k): the caller's test.
constexpr int kColPivot = kPlane, kColNone = kPlane + 1, kColSize = kPlane + 2;
template <int GL, class T, class Ok>
__device__ __forceinline__ bool sweep_block(T (&e)[BlockSlots<GL>::kN], const BlockSlots<GL>& B, T (*col)[kColSize],
                                            int nb, int steps, Ok&& pivot_ok) {
    constexpr int kN = BlockSlots<GL>::kN;
    int rr[kN], cc[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j) {
        rr[j] = B.valid(j) ? B.row(j) : kColNone;          // (matches no pivot)
        cc[j] = B.valid(j) ? B.colm(j) : kColNone;
    }
    auto publish = [&](int k) {
        T* c = col[k & 1];
#pragma unroll
        for (int j = 0; j < kN; ++j) {
            const int at = cc[j] == k ? (rr[j] == k ? kColPivot : rr[j]) : (rr[j] == k ? cc[j] : kColNone);
            c[at] = e[j];
        }
    };
    bool ok = true;
    publish(0);
#pragma unroll 1
    for (int k = 0; k < steps; ++k) {
        __syncwarp();
        if (k >= nb) continue;                  // a smaller block than the warp's largest
        const T* a = col[k & 1];
        const T p = a[kColPivot], a1 = a[B.l], a2 = a[15 - B.l];
        T ac[kN];
#pragma unroll
        for (int j = 0; j < kN; ++j) ac[j] = a[min(cc[j], kColNone)];
        const T rp = rcp_nr(p);
        ok &= pivot_ok(p, k);
        // row factor: -T_rk / p, or 1 / p on the pivot's row
        const T x1 = B.l == k ? rp : neg_bits(a1) * rp;
        const T x2 = 15 - B.l == k ? rp : neg_bits(a2) * rp;
#pragma unroll
        for (int j = 0; j < kN; ++j) {
            const T y = (rr[j] == k || cc[j] == k) ? (T)0 : e[j];
            e[j] = fma(B.low(j) ? x1 : x2, cc[j] == k ? (T)-1 : ac[j], y);
        }
        publish(k + 1);
    }
    __syncwarp();
    return ok;
}

// ---------------------------------------------------------------------------
// Up to 64 x 64 by the NT threads of a CTA.
constexpr int kInvert = 64;
template <class T>
struct InvertSmem {
    T A[kInvert][kInvert + 1];      // lower triangle (zero outside the matrix)
    T U[kInvert][kPlane + 1];       // A_xK A_KK^-1 of the current 16 columns
    T P[kPlane][kPlane + 1];        // A_KK^-1 (full, zero outside)
    T col[2][kColSize], rp[2];
    int bad;
};

// The 16 x 16 diagonal block from row k0 on (n rows) into S.P, by NT threads.
// Warp 0 runs the chain of pivots one step ahead of the others: while they
// apply pivot k - 1 to the lower triangle (one entry per thread, two with
// NT = 128), it forms pivot k itself,
//     p_k = T_kk - T_k,k-1^2 / p_(k-1)   (entries before pivot k - 1),
// and its reciprocal.  One CTA barrier per pivot hands the reciprocal to the
// update and the fresh entries to warp 0.
template <int NT, class T, class Ok>
__device__ __forceinline__ void invert16(InvertSmem<T>& S, int k0, int n, Ok&& pivot_ok) {
    constexpr int kTri = kPlane * (kPlane + 1) / 2, kOwn = (kTri + NT - 33) / (NT - 32);
    const int tid = threadIdx.x, u = tid - 32;
    int r[kOwn], c[kOwn];
    T e[kOwn];
#pragma unroll
    for (int j = 0; j < kOwn; ++j) {
        const int idx = u + (NT - 32) * j;
        r[j] = c[j] = kColNone;                            // (matches no pivot)
        e[j] = (T)0;
        if (u >= 0 && idx < kTri) {
            r[j] = (int)((sqrtf(8.0f * idx + 1.0f) - 1.0f) * 0.5f);
            while ((r[j] + 1) * (r[j] + 2) / 2 <= idx) ++r[j];
            while (r[j] * (r[j] + 1) / 2 > idx) --r[j];
            c[j] = idx - r[j] * (r[j] + 1) / 2;
            e[j] = S.A[k0 + r[j]][k0 + c[j]];
        }
    }
    // column k off its diagonal, and the next diagonal entry (last place)
    auto publish = [&](int k) {
#pragma unroll
        for (int j = 0; j < kOwn; ++j) {
            int at = c[j] == k ? r[j] : (r[j] == k ? c[j] : kColNone);
            if (r[j] == c[j]) at = r[j] == k + 1 ? kColPivot : kColNone;
            S.col[k & 1][at] = e[j];
        }
    };
    bool ok = true;
    T rp = (T)0;
    if (u >= 0) publish(0);
    if (u == 0) S.col[1][kColPivot] = e[0];                // T_00, where pivot 0 looks for it
    __syncthreads();
#pragma unroll 1
    for (int k = 0; k <= n; ++k) {
        // column k - 1 and entry (k, k) as they stand before pivot k - 1
        const T* a = S.col[(k + 1) & 1];
        if (u < 0) {
            if (k < n) {
                T p = a[kColPivot];
                if (k > 0) p = fma(neg_bits(a[k]) * a[k], rp, p);
                rp = rcp_nr(p);
                ok &= pivot_ok(p, k);
                if (tid == 0) S.rp[k & 1] = rp;
            }
        } else if (k > 0) {
            const int s = k - 1;
            const T q = S.rp[s & 1];
#pragma unroll
            for (int j = 0; j < kOwn; ++j) {
                const T m = (r[j] == s ? (T)-1 : a[r[j]]) * (c[j] == s ? (T)-1 : a[c[j]]);
                e[j] = fma(neg_bits(m), q, (r[j] == s || c[j] == s) ? (T)0 : e[j]);
            }
            publish(k);
        }
        __syncthreads();
    }
    if (u < 0) {
        if (!ok) S.bad = 1;
    } else {
#pragma unroll
        for (int j = 0; j < kOwn; ++j)
            if (r[j] < kPlane) S.P[r[j]][c[j]] = S.P[c[j]][r[j]] = r[j] < n ? neg_bits(e[j]) : (T)0;
    }
    __syncthreads();
}

// Sweeps all nb rows of S.A (-inverse in its lower triangle).  False (all
// threads) when pivot_ok(p, row) fails.
template <int NT, class T, class Ok>
__device__ bool invert_block(InvertSmem<T>& S, int nb, Ok&& pivot_ok) {
    constexpr int SL = Slices<T>::S, NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int nblk = (nb + kPlane - 1) / kPlane;
    if (tid == 0) S.bad = 0;
    __syncthreads();
    for (int kb = 0; kb < nblk; ++kb) {
        const int k0 = kb * kPlane;
        invert16<NT>(S, k0, min(kPlane, nb - k0), [&](T p, int k) { return pivot_ok(p, k0 + k); });
        // C(x, k) of row x of block bx against the block's columns
        auto c_entry = [&](int bx, int r, int k) -> T {
            return bx > kb ? S.A[bx * kPlane + r][k0 + k] : S.A[k0 + k][bx * kPlane + r];
        };
        // the powers of two that level the products over this block's columns
        int sk[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) sk[i] = half_exponent(S.P[frag_k(i)][frag_k(i)]);
        // U = C P, A_KK = -P
        for (int item = warp; item < 2 * (nblk - 1); item += NW) {
            const int q = item >> 1, nt = item & 1, bx = q < kb ? q : q + 1;
            FragA<SL> a;
            FragB<SL> b;
            load_frag_a<SL, T>(a, sk, 1, [&](int r, int k) { return c_entry(bx, r, k); });
            load_frag_b<SL, T>(b, sk, -1, [&](int n, int k) { return S.P[8 * nt + n][k]; });
            typename SplitAcc<SL>::T out[4];
            frag_product(a, b, out);
#pragma unroll
            for (int r = 0; r < 4; ++r) S.U[bx * kPlane + g + 8 * (r >> 1)][8 * nt + 2 * t + (r & 1)] = (T)out[r];
        }
        if (warp == NW - 1)
            for (int i = lane; i < kPlane * kPlane; i += 32) {
                const int r = i / kPlane, c = i % kPlane;
                if (r >= c) S.A[k0 + r][k0 + c] = neg_bits(S.P[r][c]);
            }
        __syncthreads();
        // A_xy -= C_x U_y^T by 16 x 8 tiles, each warp a run of them in row
        // order (the digits of C_x are kept from one to the next)
        const int nitem = (nblk - 1) * nblk, per = (nitem + NW - 1) / NW;
        const int lo = warp * per, hi = min(lo + per, nitem);
        int item = 0, have = -1;
        FragA<SL> a;
        for (int bx = 0; bx < nblk; ++bx)
            for (int by = 0; by <= bx; ++by) {
                if (bx == kb || by == kb) continue;
                for (int nt = 0; nt < 2; ++nt, ++item) {
                    if (item < lo || item >= hi) continue;
                    if (have != bx) load_frag_a<SL, T>(a, sk, 1, [&](int r, int k) { return c_entry(bx, r, k); });
                    have = bx;
                    FragB<SL> b;
                    load_frag_b<SL, T>(b, sk, -1, [&](int n, int k) { return S.U[by * kPlane + 8 * nt + n][k]; });
                    typename SplitAcc<SL>::T out[4];
                    frag_product(a, b, out);
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int x = bx * kPlane + g + 8 * (r >> 1), y = by * kPlane + 8 * nt + 2 * t + (r & 1);
                        if (y <= x) S.A[x][y] -= (T)out[r];
                    }
                }
            }
        __syncthreads();
        for (int i = tid; i < nblk * kPlane * kPlane; i += NT) {
            const int x = i / kPlane, c = i % kPlane, bx = x / kPlane;
            if (bx > kb) S.A[x][k0 + c] = S.U[x][c];
            else if (bx < kb) S.A[k0 + c][x] = S.U[x][c];
        }
    }
    __syncthreads();
    return S.bad == 0;
}

}  // namespace
}  // namespace mrcm
