"""The split products by themselves (csrc/split_gemm.cuh in a small library that
this test compiles): 64 x 32 products over k against extended precision, on
rows that are level, graded, of far exponents, zero, or hold an infinity or a NaN.

Bound.  With peak = max_k |a_k 2^s_k| max_k |b_k 2^-s_k| of a chunk of 64 k and the
row and column of an output, each of the chunk's terms loses two cut-off parts
and the dropped levels: (2 + 8) 2^-62 peak with eight digits (FP64), (2 + 4) 2^-30
peak with four (FP32).  FP64 rounds the chunk's sum c once and each addition of
chunks, 2^-53 of the values; FP32 rounds three times before (on |c| and the
levels still missing, below 2^-8 of all terms at their peak), 2^-24 of the values.
With one digit fewer the dropped levels alone are 2^8 times as large.

The reciprocal of the pivots over every seed argument there is (the upper 23
bits of the significand): within an ulp, so that no seed leaves [0.5, 1].
"""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "split_gemm.cuh"
namespace mrcm {
namespace {
template <int S, class T>
__global__ void product(const T* A, const T* B, const int* sk, int K, double* C) {
    extern __shared__ __align__(16) unsigned char raw[];
    SplitSmem<S>& sm = *reinterpret_cast<SplitSmem<S>*>(raw);
    typename SplitAcc<S>::T sum[2][4];
    split_product<S, T, false, false>(
        sm, K, nullptr, [&](int r) { return A + r * K; }, [&](int c) { return B + c * K; },
        [&](int k) { return sk[k]; }, sum);
    for (int mt = 0; mt < 2; ++mt)
        for (int q = 0; q < 4; ++q) C[out_row(mt, q) * kTileN + out_col(q)] = (double)sum[mt][q];
}
template <int S, class T>
int run(const void* A, const void* B, const int* sk, int K, double* C) {
    const int bytes = (int)sizeof(SplitSmem<S>);
    auto* kern = product<S, T>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return 1;
    kern<<<1, kGemmThreads, bytes>>>(static_cast<const T*>(A), static_cast<const T*>(B), sk, K, C);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 2;
}
}
}
using mrcm::run;
extern "C" int split64(const void* A, const void* B, const int* sk, int K, double* C) { return run<8, double>(A, B, sk, K, C); }
extern "C" int split32(const void* A, const void* B, const int* sk, int K, double* C) { return run<4, float>(A, B, sk, K, C); }
extern "C" int split64as32(const void* A, const void* B, const int* sk, int K, double* C) { return run<4, double>(A, B, sk, K, C); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2009_07965_gb300 import build
    d = tmp_path_factory.mktemp("split")
    (d / "split.cu").write_text(SOURCE)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-cudart", "shared", "-shared", "-I" + build.CSRC,
                    "-o", str(d / "split.so"), str(d / "split.cu")], check=True)
    return ctypes.CDLL(str(d / "split.so"))


def _product(lib, fn, A, B, sk):
    import torch
    a, b = torch.from_numpy(np.ascontiguousarray(A)).cuda(), torch.from_numpy(np.ascontiguousarray(B)).cuda()
    s = torch.from_numpy(np.asarray(sk, np.int32)).cuda()
    C = torch.empty(64, 32, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    P = ctypes.c_void_p
    assert getattr(lib, fn)(P(a.data_ptr()), P(b.data_ptr()), P(s.data_ptr()), A.shape[1], P(C.data_ptr())) == 0
    return C.cpu().numpy()


def _data(kind, K, rng, fn):
    dtype = np.float32 if fn == "split32" else np.float64
    A, B = rng.standard_normal((64, K)), rng.standard_normal((32, K))
    A *= 2.0 ** rng.integers(-3, 4, (64, 1))
    sk = np.zeros(K, int)
    span = 40 if fn == "split64" else 12
    if kind == "graded":                     # column k of A as d_k, of B as 1 / d_k: levelled by sk
        sk = -rng.integers(-span, span + 1, K)
        A, B = A * 2.0 ** -sk, B * 2.0 ** sk
    if kind == "uneven":                     # entries of one row far apart, nothing to level them
        A *= 2.0 ** rng.integers(-span, 1, A.shape)
        B *= 2.0 ** rng.integers(-span, 1, B.shape)
    if kind == "far":                        # rows of far exponents
        A *= 2.0 ** (rng.integers(-250, 251, (64, 1)) if fn == "split64" else rng.integers(-30, 31, (64, 1)))
    if kind == "zeros":
        A[::3] = 0
        B[::5] = 0
        A[1, :K // 2] = 0
        B[:, 0] = 0
    return A.astype(dtype), B.astype(dtype), sk


@pytest.mark.parametrize("K", [1, 15, 16, 17, 63, 64, 65, 130, 333])
@pytest.mark.parametrize("kind", ["level", "graded", "uneven", "far", "zeros"])
@pytest.mark.parametrize("fn", ["split64", "split32", "split64as32"])
def test_split_product_against_extended_precision(lib, fn, kind, K):
    rng = np.random.default_rng(K)
    A, B, sk = _data(kind, K, rng, fn)
    C = _product(lib, fn, A, B, sk)
    LD = np.longdouble
    unit, cut = (2.0 ** -53, 10 * 2.0 ** -62) if fn == "split64" else (3 * 2.0 ** -24, 6 * 2.0 ** -30)
    exact, bound, mag = np.zeros((64, 32), LD), np.zeros((64, 32)), np.zeros((64, 32))
    for k0 in range(0, K, 64):
        a, b, s = (x[..., k0:k0 + 64] for x in (A.astype(LD), B.astype(LD), np.asarray(sk)))
        c = np.zeros((64, 32), LD)
        for k in range(a.shape[1]):
            c += np.outer(a[:, k], b[:, k])
        exact += c
        peak = np.outer(np.max(np.abs(a * LD(2.0) ** s), 1), np.max(np.abs(b * LD(2.0) ** -s), 1)).astype(float)
        mag += np.abs(c).astype(float) + (2.0 ** -8 * peak * a.shape[1] if fn != "split64" else 0)
        bound += peak * cut * a.shape[1]
    bound += (1 + (K + 63) // 64) * unit * mag
    assert np.all(np.abs(C - exact).astype(float) <= bound)
    if kind == "zeros":
        assert np.all(C[::3] == 0) and np.all(C[:, ::5] == 0)


@pytest.mark.parametrize("fn", ["split64", "split32", "split64as32"])
def test_infinities_and_nan_reach_their_rows_and_columns_only(lib, fn):
    rng = np.random.default_rng(7)
    A, B, sk = _data("graded", 70, rng, fn)
    clean = _product(lib, fn, A, B, sk)
    A[5, 66], A[9, 2], B[3, 1] = np.inf, np.nan, -np.inf
    C = _product(lib, fn, A, B, sk)
    hit = np.zeros((64, 32), bool)
    hit[[5, 9]] = True
    hit[:, 3] = True
    assert not np.isfinite(C[hit]).any() and np.array_equal(C[~hit], clean[~hit])


def test_reciprocal_over_every_seed_argument(mrcm_lib):
    import torch
    import paper_2009_07965_gb300 as mr
    head = torch.arange(1 << 23, dtype=torch.int64, device="cuda") << 29
    for low in (0, 1, (1 << 29) - 1):
        for be in (1, 1023, 2044):
            x = ((be << 52) | head | low).view(torch.float64)
            r, t = mr.mrcm_check_reciprocal(x), 1.0 / x
            assert (r.view(torch.int64) - t.view(torch.int64)).abs().max().item() <= 1, (low, be)
