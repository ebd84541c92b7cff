// Small t-products straight from Definition 2.1 (the circular convolution of
// the tubes), in one launch:
//   C(i, j, k) = sum_q sum_{k'} op(A)(i, q, (k - k') mod n) op(B)(q, j, k').
//
// The Fourier form of a small product is four launches (two transforms, the
// slice products, the inverse) of a few microseconds each, most of it launch
// latency on the host and the device; the sums themselves are l kk m n^2
// multiply-adds, about 10^6 for a 32^3 operator and one column.  A CTA takes
// one row i of op(A) and up to four columns of op(B): the row's n x kk entries
// and the columns' go to shared memory once (row stride kk + 1: the threads of
// a warp read neighbouring k, that is neighbouring rows of op(A), at the same q,
// on distinct banks), thread (k, share) sums every P-th k', and the shares meet
// in shared memory in a fixed order.
//
// Float32 only: the sums are as exact as the Fourier form's there (1.2e-7 to
// 1.8e-7 relative against 1.0e-7 to 1e-6 over the sizes below), in float64 they
// would be up to twice as far off (3e-16).  The limit on l kk m n^2: at 8e6
// multiply-adds in CTAs of some size the kernel takes at most 10 us against 15 to 23 us
// of the four launches (32 x 32 x 32 by one column, 1e6: 4.3 against 13 us on the device,
// 19 against 27 us a call); from 1.7e7 on it is no longer always the faster one (n =
// 128, 32 x 32 by 1: 30 against 20 us).  The limit on the CTAs: one costs 2 ns whatever
// it does, so many rows or columns of short tubes belong to the Fourier form, 32 tubes
// a CTA there (n = 2: 1,216 CTAs 5.1 against 10.3 us, 5,000 13.6 against 10.8, 60,000
// 124 against 45; n = 8: 5,000 11.5 against 13.5; n = 32: 7,000 18 against 47).  It also
// keeps both dimensions of the grid in range.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace tp {

constexpr int TD_THREADS = 256;
constexpr int TD_COLS = 4;      // columns of op(B) per CTA
constexpr int TD_MAX_N = 128;

__global__ void __launch_bounds__(TD_THREADS)
k_tprod_direct(const float* __restrict__ A, const float* __restrict__ B, float* __restrict__ C, int l, int kk, int m, int n,
               int tA, int tB) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int ld = kk + 1, tid = threadIdx.x;
    const int i = blockIdx.x, j0 = blockIdx.y * TD_COLS, nc = min(TD_COLS, m - j0);
    float* as = (float*)smraw;                  // n x ld: op(A)(i, q, k)
    float* bs = as + (size_t)n * ld;        // n x kk x TD_COLS: op(B)(q, j0 + c, k)
    float* part = bs + (size_t)n * kk * TD_COLS;  // shares x n x TD_COLS
    for (int e = tid; e < n * kk; e += TD_THREADS) {
        const int k = e / kk, q = e - k * kk, r = k ? n - k : 0;  // the t-transpose reverses slices 1 .. n - 1
        as[k * ld + q] = tA ? A[((long)r * kk + q) * l + i] : A[((long)k * l + i) * kk + q];
#pragma unroll
        for (int c = 0; c < TD_COLS; ++c) {
            const int j = j0 + c;
            bs[e * TD_COLS + c] =
                c < nc ? (tB ? B[((long)r * m + j) * kk + q] : B[((long)k * kk + q) * m + j]) : 0.f;
        }
    }
    __syncthreads();
    const int P = TD_THREADS / n, share = tid / n, k = tid - share * n;
    if (share < P) {
        float acc[TD_COLS];
#pragma unroll
        for (int c = 0; c < TD_COLS; ++c) acc[c] = 0.f;
        for (int k2 = share; k2 < n; k2 += P) {
            const float* a = as + (size_t)(k >= k2 ? k - k2 : k - k2 + n) * ld;
            const float* b = bs + (size_t)k2 * kk * TD_COLS;
            float sum[TD_COLS];  // kk terms at a time: shorter chains of roundings
#pragma unroll
            for (int c = 0; c < TD_COLS; ++c) sum[c] = 0.f;
            if (nc == 1) {
#pragma unroll 4
                for (int q = 0; q < kk; ++q) sum[0] = fmaf(a[q], b[q * TD_COLS], sum[0]);
            } else {
#pragma unroll 4
                for (int q = 0; q < kk; ++q) {
                    const float x = a[q];
#pragma unroll
                    for (int c = 0; c < TD_COLS; ++c) sum[c] = fmaf(x, b[q * TD_COLS + c], sum[c]);
                }
            }
#pragma unroll
            for (int c = 0; c < TD_COLS; ++c) acc[c] += sum[c];
        }
#pragma unroll
        for (int c = 0; c < TD_COLS; ++c) part[(share * n + k) * TD_COLS + c] = acc[c];
    }
    __syncthreads();
    for (int e = tid; e < n * nc; e += TD_THREADS) {
        const int k1 = e / nc, c = e - k1 * nc;
        float v = part[k1 * TD_COLS + c];
        for (int s = 1; s < P; ++s) v += part[(s * n + k1) * TD_COLS + c];
        C[((long)k1 * l + i) * m + j0 + c] = v;
    }
}

static size_t td_smem(int kk, int n) {
    return ((size_t)n * (kk + 1) + (size_t)n * kk * TD_COLS + (size_t)TD_THREADS * TD_COLS) * sizeof(float);
}

bool tprod_direct_fits(int l, int kk, int m, int n) {
    const double work = (double)l * kk * m * n * n, ctas = (double)l * ((m + TD_COLS - 1) / TD_COLS);
    return n <= TD_MAX_N && work <= 8e6 && ctas <= 608.0 * (n + 1) && td_smem(kk, n) <= 100 * 1024;
}

tp_status tprod_direct(const float* A, const float* B, float* C, int l, int kk, int m, int n, int trans,
                       cudaStream_t st) {
    const size_t smem = td_smem(kk, n);
    if (smem_optin((const void*)k_tprod_direct, smem) != TP_OK) return TP_ERR_CUDA;
    prof_begin(TP_KC_GEMM, st);
    k_tprod_direct<<<dim3((unsigned)l, (unsigned)((m + TD_COLS - 1) / TD_COLS)), TD_THREADS, smem, st>>>(
        A, B, C, l, kk, m, n, trans & 1, trans >> 1);
    return launched(TP_KC_GEMM, st);
}

}  // namespace tp
