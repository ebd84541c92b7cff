// Mode-3 DFT along the tubes of a frontal-slice-major tensor (Section 2:
// fft(A,[],3) and its inverse), real data <-> half spectrum, any n.
//
// One CTA owns 32 neighbouring tubes as 16 packed complex sequences (tube 2p
// the real, tube 2p + 1 the imaginary part of sequence p), so that a row of a
// slice is one 8-byte load per lane and a row of the spectrum one 16-byte
// store.  n = r_1 r_2 .. r_np D: the transform is an in-place
// decimation-in-frequency FFT in shared memory, one pass per radix r_i <= 16
// (the register DFTs below), followed by direct DFTs of length D, the part of
// n made of primes above 13 (D = 1 for most n).  The passes leave the
// spectrum in digit-reversed order.
//   forward: the first pass reads its r_1 rows straight from global memory
//     (r_1 loads in flight per thread); the last pass writes shared memory, from
//     which the two tubes of a sequence are separated by conjugate symmetry;
//   inverse: the half spectrum becomes the packed full spectrum in shared
//     memory (re and im swapped: the inverse DFT is the swapped DFT of the
//     swapped data); the last pass writes its rows straight to global memory.
// So n = r_1 r_2 moves every element through shared memory two (inverse) or
// three (forward) times.
//
// What bounds it: HBM (12 bytes per element and direction), short of it the
// issue rate (62 % of the issue slots at 256 x 256 x 256, register DFTs,
// twiddles and shared-memory addresses) with 50 % occupancy.  Measured from a
// flushed L2 (CUDA events, forward / inverse), before: the direct sums over n
// that every n but the powers of two took, a radix-2 kernel for those, and
// kernels written for n = 256 and 512:
//   n    tubes      now                     before
//   96   256 x 256   21 / 23 us              116 / 140 us   (direct)
//   128  256 x 256   21 / 23 us              54 / 38 us     (radix 2)
//   256  256 x 256   36 / 40 us (3.8 TB/s)   38 / 43 us     (16 x 16)
//   331  256 x 256   322 / 289 us            1169 / 1484 us (direct; 331 is prime)
//   384  384 x 384   118 / 118 us (3.9 TB/s) 3392 / 4326 us (direct)
//   512  512 x 512   275 / 283 us (3.9 TB/s) 274 / 436 us   (16 x 32; radix 2)
//   1000 256 x 256   219 / 184 us            18654 / 19093 us (direct)
//
// Two tubes share a sequence, so a NaN or infinity in one would reach the
// other.  A CTA that meets one (or squares that overflow) evaluates the
// defining sums tube by tube instead (rare, slow, correct).
//
// The forward kernel can also emit one float64 partial sum of squares per CTA
// (used for ||A||_F^2); squares are summed per thread in the working precision
// and combined in float64 across the CTA.
#include <limits.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace tp {

constexpr int DFT_TILE = 32;   // tubes per CTA
constexpr int DFT_SEQ = 16;    // packed sequences per CTA
constexpr int DFT_MAX_THREADS = 256;
constexpr int DFT_MAX_PASS = 10;

template <typename T> __device__ __forceinline__ void sincospi_t(T x, T* s, T* c);
template <> __device__ __forceinline__ void sincospi_t<float>(float x, float* s, float* c) { sincospif(x, s, c); }
template <> __device__ __forceinline__ void sincospi_t<double>(double x, double* s, double* c) { sincospi(x, s, c); }

// ---- register DFTs ------------------------------------------------------------
// cos and sin of 2 pi m / R at compile time: the angle is brought to the first
// octant by symmetry, where the Taylor series converge to double precision.
constexpr double trig_pi = 3.14159265358979323846;
constexpr double taylor_cos(double x) {
    double t = 1.0, s = 1.0;
    for (int i = 1; i < 12; ++i) {
        t *= -x * x / ((2 * i - 1) * (2 * i));
        s += t;
    }
    return s;
}
constexpr double taylor_sin(double x) {
    double t = x, s = x;
    for (int i = 1; i < 12; ++i) {
        t *= -x * x / ((2 * i) * (2 * i + 1));
        s += t;
    }
    return s;
}
// num / den of a turn, 0 <= num / den <= 1/4
constexpr double cos_quarter(int num, int den) {
    return 8 * num <= den ? taylor_cos(2 * trig_pi * num / den) : taylor_sin(2 * trig_pi * (den - 4 * num) / (4.0 * den));
}
constexpr double root_cos(int m, int R) {
    m = ((m % R) + R) % R;
    if (2 * m > R) m = R - m;                                  // cos(2 pi - x) = cos x
    return 4 * m > R ? -cos_quarter(R - 2 * m, 2 * R) : cos_quarter(m, R);  // cos(pi - x) = -cos x
}
// sin x = cos(x - pi / 2), the angle in units of 1 / (4 R) of a turn
constexpr double root_sin(int m, int R) { return root_cos(4 * m - R, 4 * R); }

// a exp(-2 pi i m / R), m and R known at compile time
template <typename T, int M, int R> __device__ __forceinline__ cplx<T> turn(cplx<T> a) {
    constexpr int m = ((M % R) + R) % R;
    if constexpr (m == 0) {
        return a;
    } else if constexpr (4 * m == R) {
        return mk<T>(a.y, -a.x);
    } else if constexpr (2 * m == R) {
        return mk<T>(-a.x, -a.y);
    } else if constexpr (4 * m == 3 * R) {
        return mk<T>(-a.y, a.x);
    } else {
        constexpr double cd = root_cos(m, R), sd = root_sin(m, R);
        const T c = (T)cd, s = (T)sd;
        return mk<T>(a.x * c + a.y * s, a.y * c - a.x * s);
    }
}

// Forward R-point DFT of v in place, natural order in and out:
// X_k = sum_t x_t exp(-2 pi i t k / R).
template <typename T, int R> struct RDft;
template <typename T> struct RDft<T, 1> {
    static __device__ __forceinline__ void run(cplx<T> (&)[1]) {}
};
template <typename T> struct RDft<T, 2> {
    static __device__ __forceinline__ void run(cplx<T> (&v)[2]) {
        const cplx<T> a = v[0];
        v[0] = cadd(a, v[1]);
        v[1] = csub(a, v[1]);
    }
};
template <typename T> struct RDft<T, 4> {
    static __device__ __forceinline__ void run(cplx<T> (&v)[4]) {
        const cplx<T> t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]), t2 = cadd(v[1], v[3]), t3 = csub(v[1], v[3]);
        v[0] = cadd(t0, t2);
        v[2] = csub(t0, t2);
        v[1] = mk<T>(t1.x + t3.y, t1.y - t3.x);  // t1 - i t3
        v[3] = mk<T>(t1.x - t3.y, t1.y + t3.x);  // t1 + i t3
    }
};
// odd prime R: with e_q = x_q + x_{R-q} and o_q = x_q - x_{R-q},
// X_k, X_{R-k} = (x_0 + sum e_q cos(2 pi q k / R)) -+ i sum o_q sin(2 pi q k / R)
template <typename T, int R> struct RDftOdd {
    template <int K, int Q> static __device__ __forceinline__ void terms(const cplx<T> (&e)[R / 2], const cplx<T> (&o)[R / 2],
                                                                         cplx<T>& a, cplx<T>& b) {
        if constexpr (Q <= R / 2) {
            constexpr double cd = root_cos(K * Q, R), sd = root_sin(K * Q, R);
            const T c = (T)cd, s = (T)sd;
            a.x = fma(e[Q - 1].x, c, a.x);
            a.y = fma(e[Q - 1].y, c, a.y);
            b.x = fma(o[Q - 1].x, s, b.x);
            b.y = fma(o[Q - 1].y, s, b.y);
            terms<K, Q + 1>(e, o, a, b);
        }
    }
    template <int K> static __device__ __forceinline__ void outputs(const cplx<T> (&e)[R / 2], const cplx<T> (&o)[R / 2],
                                                                    cplx<T> x0, cplx<T> (&v)[R]) {
        if constexpr (K <= R / 2) {
            cplx<T> a = x0, b = mk<T>(0, 0);
            terms<K, 1>(e, o, a, b);
            v[K] = mk<T>(a.x + b.y, a.y - b.x);      // a - i b
            v[R - K] = mk<T>(a.x - b.y, a.y + b.x);  // a + i b
            outputs<K + 1>(e, o, x0, v);
        }
    }
    static __device__ __forceinline__ void run(cplx<T> (&v)[R]) {
        cplx<T> e[R / 2], o[R / 2], x0 = v[0], s = v[0];
#pragma unroll
        for (int q = 1; q <= R / 2; ++q) {
            e[q - 1] = cadd(v[q], v[R - q]);
            o[q - 1] = csub(v[q], v[R - q]);
            s = cadd(s, e[q - 1]);
        }
        v[0] = s;
        outputs<1>(e, o, x0, v);
    }
};
template <typename T> struct RDft<T, 3> : RDftOdd<T, 3> {};
template <typename T> struct RDft<T, 5> : RDftOdd<T, 5> {};
template <typename T> struct RDft<T, 7> : RDftOdd<T, 7> {};
template <typename T> struct RDft<T, 11> : RDftOdd<T, 11> {};
template <typename T> struct RDft<T, 13> : RDftOdd<T, 13> {};
// R = A B: t = B t1 + t2, k = k1 + A k2
template <typename T, int A, int B> struct RDftComp {
    static constexpr int R = A * B;
    template <int T2> static __device__ __forceinline__ void columns(cplx<T> (&v)[R]) {
        if constexpr (T2 < B) {
            cplx<T> u[A];
#pragma unroll
            for (int i = 0; i < A; ++i) u[i] = v[B * i + T2];
            RDft<T, A>::run(u);
            twiddles<T2, 0>(u, v);
            columns<T2 + 1>(v);
        }
    }
    template <int T2, int K1> static __device__ __forceinline__ void twiddles(cplx<T> (&u)[A], cplx<T> (&v)[R]) {
        if constexpr (K1 < A) {
            v[B * K1 + T2] = turn<T, T2 * K1, R>(u[K1]);
            twiddles<T2, K1 + 1>(u, v);
        }
    }
    static __device__ __forceinline__ void run(cplx<T> (&v)[R]) {
        columns<0>(v);
        cplx<T> o[R];
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            cplx<T> u[B];
#pragma unroll
            for (int i = 0; i < B; ++i) u[i] = v[B * k1 + i];
            RDft<T, B>::run(u);
#pragma unroll
            for (int i = 0; i < B; ++i) o[k1 + A * i] = u[i];
        }
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = o[i];
    }
};
template <typename T> struct RDft<T, 6> : RDftComp<T, 2, 3> {};
template <typename T> struct RDft<T, 8> : RDftComp<T, 2, 4> {};
template <typename T> struct RDft<T, 9> : RDftComp<T, 3, 3> {};
template <typename T> struct RDft<T, 10> : RDftComp<T, 2, 5> {};
template <typename T> struct RDft<T, 12> : RDftComp<T, 4, 3> {};
template <typename T> struct RDft<T, 15> : RDftComp<T, 3, 5> {};
template <typename T> struct RDft<T, 16> : RDftComp<T, 4, 4> {};

constexpr int DFT_RADICES[] = {16, 15, 13, 12, 11, 10, 9, 8, 7, 6, 5, 4, 3, 2, 1};

// ---- the plan -------------------------------------------------------------------
struct DftPlan {
    int n = 0, np, D;         // n = r[0] .. r[np-1] D
    int r[DFT_MAX_PASS];
    unsigned rr[DFT_MAX_PASS], rm[DFT_MAX_PASS];  // ceil(2^20 / r) and ceil(2^20 / M) of each pass (M: see pass_smem)
    int lns;                  // log2 of the sequences per sub-tile
    int nt;                   // threads per CTA
    int kb;                   // direct part: pairs (k, D - k) per thread
    int cls;                  // dft_class
    bool split;               // one CTA per sub-tile
    size_t smem;
};

// Fewest passes, then the smallest sum of radices, largest radix first.
static void best_radices(int m, int max_idx, int depth, int sum, int* cur, int* best, int* best_np, int* best_sum) {
    if (m == 1) {
        if (depth < *best_np || (depth == *best_np && sum < *best_sum)) {
            *best_np = depth;
            *best_sum = sum;
            for (int i = 0; i < depth; ++i) best[i] = cur[i];
        }
        return;
    }
    if (depth + 1 > *best_np || depth + 1 > DFT_MAX_PASS) return;
    for (int i = max_idx; DFT_RADICES[i] > 1; ++i)
        if (m % DFT_RADICES[i] == 0) {
            cur[depth] = DFT_RADICES[i];
            best_radices(m / DFT_RADICES[i], i, depth + 1, sum + DFT_RADICES[i], cur, best, best_np, best_sum);
        }
}

// sequences per sub-tile: all 16 while two CTAs fit on an SM (the direct part
// needs a second buffer in the forward kernel), else 8 or 4, one after another
static size_t dft_smem(const DftPlan& P, size_t elem, bool fwd) {
    const size_t c = 2 * elem, buf = ((size_t)P.n << P.lns) * c;
    return (P.D > 1 && fwd ? 2 : 1) * buf + (size_t)P.n * c + (((size_t)P.n * 2 + 15) & ~(size_t)15);
}

// Class of a plan: 0 = powers of two, 1 = radices up to 10, 2 = the other
// products of small primes, 3 = plans with a direct part or whose tiles are
// split (the others have the sequence count as a compile-time constant).
static int dft_class(const DftPlan& P) {
    if (P.lns != 4 || P.D > 1) return 3;
    int cls = 0;
    for (int i = 0; i < P.np; ++i) {
        const int r = P.r[i];
        if (r > 10 && r != 16) return 2;
        if (r & (r - 1)) cls = 1;
    }
    for (int i = 0; i < P.np; ++i)
        if (cls == 1 && P.r[i] > 10) return 2;
    return cls;
}
// split: a CTA per sub-tile of four sequences instead of per tile
static DftPlan make_plan(int n, size_t elem, bool fwd, bool split) {
    DftPlan P;
    P.n = n;
    P.split = split;
    int m = n;
    P.D = 1;
    for (int q = 17; q <= m; ++q)
        while (m % q == 0) {
            bool prime = true;
            for (int d = 2; d * d <= q; ++d) prime = prime && q % d != 0;
            if (!prime) break;
            m /= q;
            P.D *= q;
        }
    int cur[DFT_MAX_PASS], sum = 1 << 30;
    P.np = DFT_MAX_PASS + 1;
    best_radices(m, 0, 0, 0, cur, P.r, &P.np, &sum);
    if (P.np == 0 && P.D == 1) {  // n = 1
        P.np = 1;
        P.r[0] = 1;
    }
    // x / d = x ceil(2^20 / d) >> 20 for x <= 1024, d <= 1024
    for (int i = 0, L = n; i < P.np; ++i) {
        P.rr[i] = ((1u << 20) + P.r[i] - 1) / P.r[i];
        L /= P.r[i];
        P.rm[i] = ((1u << 20) + L - 1) / L;
    }
    P.lns = split ? 2 : 4;
    while (P.lns > 2 && dft_smem(P, elem, fwd) > 112 * 1024) --P.lns;
    // a thread per item of the pass with the fewest items
    const int items = (n / (P.np ? P.r[0] : 1)) << P.lns;
    P.nt = std::min(DFT_MAX_THREADS, std::max(64, (items + 31) & ~31));
    // The direct part: groups of kb pairs on sequences / 2 lanes each, about 12 kb + 4 instructions per entry.
    // Up to about 370 points one round of some width does (17 .. 61 points on 64 or 128 threads, 331 on 256):
    // the cheapest of those, counting no fewer than three warps (fewer leave the SM waiting).  Beyond, 256 threads
    // and the fewest rounds, about kb + 1/2 units of time each.
    if (P.D > 1) {
        int cost1 = INT_MAX, cost2 = INT_MAX, nt1 = 0, kb1 = 0, kb2 = 4;
        for (int nt = DFT_MAX_THREADS; nt >= 64; nt /= 2)
            for (int kb : {2, 3, 4, 6}) {
                const int slots = nt >> (P.lns - 1), groups = n / P.D * ((P.D / 2 + kb) / kb);
                const int rounds = (groups + slots - 1) / slots;
                const int c1 = std::max(nt, 96) * (12 * kb + 4), c2 = rounds * (2 * kb + 1);
                if (rounds == 1 && c1 < cost1) {
                    cost1 = c1;
                    nt1 = nt;
                    kb1 = kb;
                }
                if (nt == DFT_MAX_THREADS && c2 < cost2) {
                    cost2 = c2;
                    kb2 = kb;
                }
            }
        P.nt = nt1 ? nt1 : DFT_MAX_THREADS;
        P.kb = nt1 ? kb1 : kb2;
    } else {
        P.kb = 0;
    }
    P.smem = dft_smem(P, elem, fwd);
    P.cls = dft_class(P);
    return P;
}

// The plans of the last lengths that a thread used (the search takes about a
// microsecond, which a small transform would notice).
static const DftPlan& dft_plan(int n, size_t elem, bool fwd, bool split) {
    struct Slot {
        DftPlan P;
        size_t elem = 0;
        bool fwd = false;
    };
    thread_local Slot slots[16];
    Slot& s = slots[((n * 4) ^ (elem == 4 ? 2 : 0) ^ (fwd ? 1 : 0)) & 15];
    if (s.elem != elem || s.fwd != fwd || s.P.n != n || s.P.split != split) {
        s.P = make_plan(n, elem, fwd, split);
        s.elem = elem;
        s.fwd = fwd;
    }
    return s.P;
}

constexpr int DFT_CTAS[4] = {4, 4, 3, 2};  // CTAs per SM that the registers of each class allow (float32)

// ---- kernels ----------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void store_partial(T v, double* sumsq) {
    __shared__ double red[33];
    const double t = block_sum_t(v, red);
    if (threadIdx.x == 0) sumsq[blockIdx.x] = t;
}

__device__ __forceinline__ long tube_off(long t, int cols, long ld) {
    if (ld == cols) return t;  // a uniform branch: no 64-bit division
    const long r = t / cols;
    return r * ld + (t - r * cols);
}

// n roots exp(-2 pi i m / n), and the digit reversal of the passes: table[pos]
// = frequency index of shared position pos (inverse) or table[s] = position
// of frequency s (forward).  Position digits (most significant first) are k_1
// (weight n / r_1), k_2 (n / (r_1 r_2)), ..., the last one, of the direct part,
// of weight 1; the frequency is k_1 + r_1 (k_2 + r_2 (k_3 + ...)).
template <typename T>
__device__ __forceinline__ void fill_tables(const DftPlan& P, cplx<T>* tw, unsigned short* table, bool by_pos) {
    const int n = P.n;
    const T step = (T)2 / (T)n;
    const bool pow2 = (n & (n - 1)) == 0;  // 2 m / n without a division then
    for (int m = threadIdx.x; m < n; m += blockDim.x) {
        T s, c;
        sincospi_t<T>(pow2 ? (T)m * step : (T)(2 * m) / (T)n, &s, &c);
        tw[m] = mk<T>(c, -s);
        int rest = m, pos = 0, w = n;
        for (int i = 0; i < P.np; ++i) {  // m as a frequency: its digits, lowest first
            const int r = P.r[i], q = (int)((rest * P.rr[i]) >> 20);
            w = (int)((w * P.rr[i]) >> 20);
            pos += (rest - q * r) * w;
            rest = q;
        }
        pos += rest;
        if (by_pos) table[pos] = (unsigned short)m;
        else table[m] = (unsigned short)pos;
    }
}

// One pass over shared memory: blocks of length L, radix R, M = L / R.
// LAST: M = 1, no twiddles.  MR = ceil(2^20 / M) divides item numbers by M.
template <typename T, int R, bool LAST>
__device__ __forceinline__ void pass_smem(cplx<T>* z, const cplx<T>* tw, int n, int L, int tstep, unsigned MR, int lns) {
    const int p = threadIdx.x & ((1 << lns) - 1), ust = blockDim.x >> lns, items = n / R;
    const int M = LAST ? 1 : L / R;
    for (int u = threadIdx.x >> lns; u < items; u += ust) {
        const int b = LAST ? u : (int)((u * MR) >> 20), j = LAST ? 0 : u - b * M;
        cplx<T>* zp = z + ((size_t)(b * L + j) << lns) + p;
        cplx<T> v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = zp[(q * M) << lns];
        RDft<T, R>::run(v);
        zp[0] = v[0];
#pragma unroll
        for (int k = 1; k < R; ++k) zp[(k * M) << lns] = LAST ? v[k] : cmul(v[k], tw[j * k * tstep]);
    }
}

// The radices of a kernel's class (dft_class): the registers of a kernel are
// those of its largest radix, and fewer registers keep more CTAs on an SM.
#define DFT_SWITCH(r, GO)                                    \
    if constexpr (CLS == 0) {                                \
        switch (r) {                                         \
            case 1: GO(1); break;                            \
            case 2: GO(2); break;                            \
            case 4: GO(4); break;                            \
            case 8: GO(8); break;                            \
            default: GO(16); break;                          \
        }                                                    \
    } else if constexpr (CLS == 1) {                         \
        switch (r) {                                         \
            case 2: GO(2); break;                            \
            case 3: GO(3); break;                            \
            case 4: GO(4); break;                            \
            case 5: GO(5); break;                            \
            case 6: GO(6); break;                            \
            case 7: GO(7); break;                            \
            case 8: GO(8); break;                            \
            case 9: GO(9); break;                            \
            default: GO(10); break;                          \
        }                                                    \
    } else {                                                 \
        switch (r) {                                         \
            case 1: GO(1); break;                            \
            case 2: GO(2); break;                            \
            case 3: GO(3); break;                            \
            case 4: GO(4); break;                            \
            case 5: GO(5); break;                            \
            case 6: GO(6); break;                            \
            case 7: GO(7); break;                            \
            case 8: GO(8); break;                            \
            case 9: GO(9); break;                            \
            case 10: GO(10); break;                          \
            case 11: GO(11); break;                          \
            case 12: GO(12); break;                          \
            case 13: GO(13); break;                          \
            case 15: GO(15); break;                          \
            default: GO(16); break;                          \
        }                                                    \
    }

// First forward pass: rows j, j + M, ... of the real tubes, packed.
template <typename T, int R>
__device__ __forceinline__ void pass_load(cplx<T>* z, const cplx<T>* tw, int n, int lns, const T* xa, const T* xb,
                                          bool la, bool lb, bool vec, long ss, T& acc) {
    const int p = threadIdx.x & ((1 << lns) - 1), M = n / R, ust = blockDim.x >> lns;
    for (int j = threadIdx.x >> lns; j < M; j += ust) {
        cplx<T> v[R];
        if (vec) {
#pragma unroll
            for (int q = 0; q < R; ++q)
                v[q] = la ? __ldcs((const cplx<T>*)(xa + (long)(j + q * M) * ss)) : mk<T>(0, 0);
        } else {
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const long off = (long)(j + q * M) * ss;
                v[q] = mk<T>(la ? __ldcs(xa + off) : (T)0, lb ? __ldcs(xb + off) : (T)0);
            }
        }
#pragma unroll
        for (int q = 0; q < R; ++q) acc = fma(v[q].x, v[q].x, fma(v[q].y, v[q].y, acc));
        RDft<T, R>::run(v);
        cplx<T>* zp = z + ((size_t)j << lns) + p;
        zp[0] = v[0];
#pragma unroll
        for (int k = 1; k < R; ++k) zp[(k * M) << lns] = cmul(v[k], tw[j * k]);
    }
}

// Last inverse pass: block u's outputs are the rows low + (n / R) k of the
// tubes (low = the frequency of the block's first position), swapped back and
// scaled.
template <typename T, int R>
__device__ __forceinline__ void pass_store(const cplx<T>* z, const unsigned short* freq, int n, int lns, T* xa, T* xb,
                                           bool la, bool lb, bool vec, long ss) {
    const int p = threadIdx.x & ((1 << lns) - 1), M = n / R, ust = blockDim.x >> lns;
    const T inv = (T)1 / (T)n;
    for (int u = threadIdx.x >> lns; u < M; u += ust) {
        const cplx<T>* zp = z + ((size_t)(u * R) << lns) + p;
        cplx<T> v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = zp[q << lns];
        RDft<T, R>::run(v);
        const long row = freq[u * R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const long off = (row + (long)k * M) * ss;
            if (vec) {
                if (la) *(cplx<T>*)(xa + off) = mk<T>(v[k].y * inv, v[k].x * inv);
            } else {
                if (la) xa[off] = v[k].y * inv;
                if (lb) xb[off] = v[k].x * inv;
            }
        }
    }
}

// The direct part: DFTs of the n / D contiguous blocks of odd length D, whose
// entries q and D - q first become e_q = x_q + x_{D-q} and o_q = x_q - x_{D-q}.
// (direct_fold.)  A thread forms KB pairs (k, D - k) of two neighbouring sequences, so each
// twiddle and each (e, o) read serves several products (about two thirds of
// the issue slots are multiply-adds).  put(block, k, sequence, value).
template <typename T>
__device__ __forceinline__ void direct_fold(cplx<T>* z, int n, int D, int lns) {
    typedef cplx<T> V;
    const int H = D / 2, nb = n / D, ns = 1 << lns;
    for (int e = threadIdx.x; e < nb * H * ns; e += blockDim.x) {
        const int p = e & (ns - 1), bq = e >> lns, b = bq / H, q = bq - b * H + 1;
        V* x = z + ((size_t)(b * D + q) << lns) + p;
        V* y = z + ((size_t)(b * D + D - q) << lns) + p;
        const V u = *x, v = *y;
        *x = cadd(u, v);
        *y = csub(u, v);
    }
    __syncthreads();
}
template <typename T, int KB, typename Put>
__device__ __forceinline__ void direct_part(const cplx<T>* z, const cplx<T>* tw, int n, int D, int lns, Put put) {
    typedef cplx<T> V;
    const int H = D / 2, nb = n / D, ts = n / D;  // twiddles exp(-2 pi i m / D) = tw[m n / D]
    const int lhs = lns - 1, sp = threadIdx.x & ((1 << lhs) - 1), gst = blockDim.x >> lhs;
    const int ng = (H + KB) / KB;  // groups of KB values of k in 0 .. H
    for (int it = threadIdx.x >> lhs; it < nb * ng; it += gst) {
        const int b = it / ng, k0 = (it - b * ng) * KB;
        const V* zb = z + ((size_t)(b * D) << lns) + 2 * sp;
        V A[KB][2], B[KB][2];
        int idx[KB], kk[KB];
#pragma unroll
        for (int t = 0; t < KB; ++t) {
            kk[t] = min(k0 + t, H);
            idx[t] = 0;
            A[t][0] = zb[0];
            A[t][1] = zb[1];
            B[t][0] = B[t][1] = mk<T>(0, 0);
        }
#pragma unroll 2
        for (int q = 1; q <= H; ++q) {
            const V e0 = zb[(size_t)q << lns], e1 = zb[((size_t)q << lns) + 1];
            const V o0 = zb[(size_t)(D - q) << lns], o1 = zb[((size_t)(D - q) << lns) + 1];
#pragma unroll
            for (int t = 0; t < KB; ++t) {
                const unsigned nx = (unsigned)(idx[t] + kk[t]);
                idx[t] = (int)min(nx, nx - (unsigned)D);  // (q k) mod D
                const V w = tw[idx[t] * ts];
                A[t][0].x = fma(e0.x, w.x, A[t][0].x);
                A[t][0].y = fma(e0.y, w.x, A[t][0].y);
                A[t][1].x = fma(e1.x, w.x, A[t][1].x);
                A[t][1].y = fma(e1.y, w.x, A[t][1].y);
                B[t][0].x = fma(o0.x, w.y, B[t][0].x);
                B[t][0].y = fma(o0.y, w.y, B[t][0].y);
                B[t][1].x = fma(o1.x, w.y, B[t][1].x);
                B[t][1].y = fma(o1.y, w.y, B[t][1].y);
            }
        }
        // tw holds cos - i sin: X_k, X_{D-k} = A +- i B
#pragma unroll
        for (int t = 0; t < KB; ++t) {
            const int k = k0 + t;
            if (k > H) break;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const V a = A[t][c], bb = B[t][c];
                put(b, k, 2 * sp + c, mk<T>(a.x - bb.y, a.y + bb.x));
                if (k > 0) put(b, D - k, 2 * sp + c, mk<T>(a.x + bb.y, a.y - bb.x));
            }
        }
    }
}

// Entries of two neighbouring tubes in one row of the spectrum.
template <typename T>
__device__ __forceinline__ void store_pair(cplx<T>* dst, cplx<T> a, cplx<T> b, bool lb, bool vec) {
    if (sizeof(T) == 4 && vec) {
        *(float4*)dst = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
    } else {
        dst[0] = a;
        if (lb) dst[1] = b;
    }
}
template <typename T>
__device__ __forceinline__ void load_pair(const cplx<T>* src, cplx<T>& a, cplx<T>& b, bool lb, bool vec) {
    if (sizeof(T) == 4 && vec) {
        const float4 v = *(const float4*)src;
        a = mk<T>((T)v.x, (T)v.y);
        b = mk<T>((T)v.z, (T)v.w);
    } else {
        a = src[0];
        if (lb) b = src[1];
    }
}

template <typename T, int CLS>
__global__ void __launch_bounds__(DFT_MAX_THREADS, sizeof(T) == 4 ? DFT_CTAS[CLS] : 1)
k_rdft(const __grid_constant__ DftPlan P, const T* __restrict__ X, cplx<T>* __restrict__ Xh, long tubes, int cols,
       long ld, long ss, int vin, int vout, double* sumsq, const int* skip) {
    if (skip && *skip) return;
    typedef cplx<T> V;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int n = P.n, lns = CLS == 3 ? P.lns : 4, ns = 1 << lns, h = n / 2 + 1;
    V* z = (V*)smraw;
    V* z2 = CLS == 3 && P.D > 1 ? z + ((size_t)n << lns) : z;
    V* tw = z2 + ((size_t)n << lns);
    unsigned short* pos = (unsigned short*)(tw + n);
    fill_tables<T>(P, tw, pos, false);
    __syncthreads();
    T total = 0;
    // all sub-tiles of tile blockIdx.x, or (split) one
    const int nsub = DFT_SEQ >> lns;
    const long tile = CLS == 3 && P.split ? blockIdx.x / nsub : blockIdx.x;
    const int sub0 = CLS == 3 && P.split ? (blockIdx.x % nsub) << lns : 0;
    const int sub1 = CLS == 3 && P.split ? sub0 + ns : DFT_SEQ;
    for (int sub = sub0; sub < sub1; sub += ns) {
        const long t0 = tile * DFT_TILE + 2 * (sub + (threadIdx.x & (ns - 1)));
        const bool la = t0 < tubes, lb = t0 + 1 < tubes;
        const T* xa = X + (la ? tube_off(t0, cols, ld) : 0);
        const T* xb = X + (lb ? tube_off(t0 + 1, cols, ld) : 0);
        T acc = 0;
        int L = n, tstep = 1;
        if (CLS < 3 || P.np > 0) {
#define GO(R) pass_load<T, R>(z, tw, n, lns, xa, xb, la, lb, vin, ss, acc)
            DFT_SWITCH(P.r[0], GO)
#undef GO
            tstep = P.r[0];
            L = (int)((n * P.rr[0]) >> 20);
        } else {  // n is all direct part: a plain copy
            for (int k = threadIdx.x >> lns; k < n; k += blockDim.x >> lns) {
                const V v = mk<T>(la ? __ldcs(xa + (long)k * ss) : (T)0, lb ? __ldcs(xb + (long)k * ss) : (T)0);
                acc = fma(v.x, v.x, fma(v.y, v.y, acc));
                z[((size_t)k << lns) + (threadIdx.x & (ns - 1))] = v;
            }
        }
        const bool finite = !__syncthreads_or(!isfinite(acc));
        total += acc;
        if (!finite) {
            // the defining sum, tube by tube
            const long f0 = tile * DFT_TILE + 2 * sub;
            for (int e = threadIdx.x; e < h * 2 * ns; e += blockDim.x) {
                const int s = e / (2 * ns), tt = e - s * 2 * ns;
                const long t = f0 + tt;
                if (t >= tubes) continue;
                const T* x = X + tube_off(t, cols, ld);
                V o = mk<T>(0, 0);
                int idx = 0;
                for (int k = 0; k < n; ++k) {
                    const T v = x[(long)k * ss];
                    o.x = fma(v, tw[idx].x, o.x);
                    o.y = fma(v, tw[idx].y, o.y);
                    idx += s;
                    if (idx >= n) idx -= n;
                }
                Xh[(long)s * tubes + t] = o;
            }
            __syncthreads();
            continue;
        }
        for (int i = 1; i < P.np; ++i) {
            if (L == P.r[i]) {
#define GO(R) pass_smem<T, R, true>(z, tw, n, L, tstep, 0u, lns)
                DFT_SWITCH(P.r[i], GO)
#undef GO
            } else {
#define GO(R) pass_smem<T, R, false>(z, tw, n, L, tstep, P.rm[i], lns)
                DFT_SWITCH(P.r[i], GO)
#undef GO
            }
            tstep *= P.r[i];
            L = (int)((L * P.rr[i]) >> 20);
            __syncthreads();
        }
        if (CLS == 3 && P.D > 1) {
            direct_fold<T>(z, n, P.D, lns);
            auto put = [&](int b, int k, int q, V v) { z2[((size_t)(b * P.D + k) << lns) + q] = v; };
            if (P.kb == 2) direct_part<T, 2>(z, tw, n, P.D, lns, put);
            else if (P.kb == 3) direct_part<T, 3>(z, tw, n, P.D, lns, put);
            else if (P.kb == 4) direct_part<T, 4>(z, tw, n, P.D, lns, put);
            else direct_part<T, 6>(z, tw, n, P.D, lns, put);
            __syncthreads();
        }
        // the two tubes of a sequence: (Z_s + conj Z_{n-s}) / 2 and (Z_s - conj Z_{n-s}) / 2i
        const int p = threadIdx.x & (ns - 1);
        if (la) {
            const int hp = (n + 1) / 2, sst = blockDim.x >> lns;
            V* dst = Xh + t0;
            auto out = [&](int s, int m) {  // m: n - s, or s when they are the same slice
                const V zs = z2[((size_t)pos[s] << lns) + p], zc = z2[((size_t)pos[m] << lns) + p];
                const V a = mk<T>((zs.x + zc.x) * (T)0.5, (zs.y - zc.y) * (T)0.5);
                const V b = mk<T>((zs.y + zc.y) * (T)0.5, (zc.x - zs.x) * (T)0.5);
                store_pair<T>(dst + (long)s * tubes, a, b, lb, vout);
            };
#pragma unroll 2
            for (int s = threadIdx.x >> lns; s < hp; s += sst) out(s, s ? n - s : 0);
            if (2 * hp == n && (int)(threadIdx.x >> lns) == sst - 1) out(hp, hp);
        }
        if (ns < DFT_SEQ) __syncthreads();
    }
    if (sumsq) store_partial<T>(total, sumsq);
}

template <typename T, int CLS>
__global__ void __launch_bounds__(DFT_MAX_THREADS, sizeof(T) == 4 ? DFT_CTAS[CLS] : 1)
k_irdft(const __grid_constant__ DftPlan P, const cplx<T>* __restrict__ Xh, T* __restrict__ X, long tubes, int cols,
        long ld, long ss, int vin, int vout, const int* skip) {
    if (skip && *skip) return;
    typedef cplx<T> V;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int n = P.n, lns = CLS == 3 ? P.lns : 4, ns = 1 << lns, h = n / 2 + 1;
    V* z = (V*)smraw;
    V* tw = z + ((size_t)n << lns);
    unsigned short* freq = (unsigned short*)(tw + n);
    fill_tables<T>(P, tw, freq, true);
    const int nsub = DFT_SEQ >> lns;
    const long tile = CLS == 3 && P.split ? blockIdx.x / nsub : blockIdx.x;
    const int sub0 = CLS == 3 && P.split ? (blockIdx.x % nsub) << lns : 0;
    const int sub1 = CLS == 3 && P.split ? sub0 + ns : DFT_SEQ;
    for (int sub = sub0; sub < sub1; sub += ns) {
        const int p = threadIdx.x & (ns - 1), sst = blockDim.x >> lns;
        const long t0 = tile * DFT_TILE + 2 * (sub + p);
        const bool la = t0 < tubes, lb = t0 + 1 < tubes;
        T* xa = X + (la ? tube_off(t0, cols, ld) : 0);
        T* xb = X + (lb ? tube_off(t0 + 1, cols, ld) : 0);
        T bad = 0;  // stays 0 for finite data
        constexpr int LB = sizeof(T) == 4 ? 8 : 4;  // pairs of spectrum entries in flight per thread
        const int hp = (n + 1) / 2;  // slices 0 .. hp - 1, then slice n / 2 of an even n
        auto put = [&](int s, V x, V y, bool self) {
            if (self) x.y = y.y = 0;  // the imaginary parts of slices 0 and n / 2 are ignored
            bad = fma(x.x, (T)0, fma(x.y, (T)0, fma(y.x, (T)0, fma(y.y, (T)0, bad))));
            // Z_s = x + i y and Z_{n-s} = conj(x) + i conj(y), re and im swapped
            z[((size_t)s << lns) + p] = mk<T>(x.y + y.x, x.x - y.y);
            if (!self) z[((size_t)(n - s) << lns) + p] = mk<T>(y.x - x.y, x.x + y.y);
        };
        const V* src = Xh + t0;
        for (int s0 = threadIdx.x >> lns; s0 < hp; s0 += LB * sst) {
            V a[LB], b[LB];
#pragma unroll
            for (int u = 0; u < LB; ++u) {
                a[u] = b[u] = mk<T>(0, 0);
                if (la && s0 + u * sst < hp) load_pair<T>(src + (long)(s0 + u * sst) * tubes, a[u], b[u], lb, vin);
            }
#pragma unroll
            for (int u = 0; u < LB; ++u)
                if (s0 + u * sst < hp) put(s0 + u * sst, a[u], b[u], s0 + u * sst == 0);
        }
        if (2 * hp == n && (int)(threadIdx.x >> lns) == sst - 1) {
            V a = mk<T>(0, 0), b = mk<T>(0, 0);
            if (la) load_pair<T>(src + (long)hp * tubes, a, b, lb, vin);
            put(hp, a, b, true);
        }
        const bool finite = !__syncthreads_or(bad != (T)0 || isnan(bad));
        if (!finite) {
            // the defining sum, tube by tube
            const long f0 = tile * DFT_TILE + 2 * sub;
            const T inv = (T)1 / (T)n;
            for (int e = threadIdx.x; e < n * 2 * ns; e += blockDim.x) {
                const int k = e / (2 * ns), tt = e - k * 2 * ns;
                const long t = f0 + tt;
                if (t >= tubes) continue;
                T acc = Xh[t].x;
                int idx = k;
                for (int s = 1; s < h; ++s) {
                    V v = Xh[(long)s * tubes + t];
                    if (2 * s == n) v.y = 0;
                    const T w = (2 * s == n) ? (T)1 : (T)2;
                    acc += w * (v.x * tw[idx].x + v.y * tw[idx].y);  // tw holds cos - i sin
                    idx += k;
                    if (idx >= n) idx -= n;
                }
                X[tube_off(t, cols, ld) + (long)k * ss] = acc * inv;
            }
            __syncthreads();
            continue;
        }
        int L = n, tstep = 1;
        const int last = P.D > 1 ? P.np : P.np - 1;
        for (int i = 0; i < last; ++i) {
            if (L == P.r[i]) {
#define GO(R) pass_smem<T, R, true>(z, tw, n, L, tstep, 0u, lns)
                DFT_SWITCH(P.r[i], GO)
#undef GO
            } else {
#define GO(R) pass_smem<T, R, false>(z, tw, n, L, tstep, P.rm[i], lns)
                DFT_SWITCH(P.r[i], GO)
#undef GO
            }
            tstep *= P.r[i];
            L = (int)((L * P.rr[i]) >> 20);
            __syncthreads();
        }
        if (CLS == 3 && P.D > 1) {
            const T inv = (T)1 / (T)n;
            const int nb = n / P.D;
            const long f0 = tile * DFT_TILE + 2 * sub;
            direct_fold<T>(z, n, P.D, lns);
            auto put = [&](int b, int k, int q, V v) {
                const long t = f0 + 2 * q, off = (long)(freq[b * P.D] + nb * k) * ss;
                if (t < tubes) X[tube_off(t, cols, ld) + off] = v.y * inv;
                if (t + 1 < tubes) X[tube_off(t + 1, cols, ld) + off] = v.x * inv;
            };
            if (P.kb == 2) direct_part<T, 2>(z, tw, n, P.D, lns, put);
            else if (P.kb == 3) direct_part<T, 3>(z, tw, n, P.D, lns, put);
            else if (P.kb == 4) direct_part<T, 4>(z, tw, n, P.D, lns, put);
            else direct_part<T, 6>(z, tw, n, P.D, lns, put);
        } else {
#define GO(R) pass_store<T, R>(z, freq, n, lns, xa, xb, la, lb, vout, ss)
            DFT_SWITCH(P.r[last], GO)
#undef GO
        }
        if (ns < DFT_SEQ) __syncthreads();
    }
}

int rdft_parts(int rows, int cols) { return (int)(((long)rows * cols + DFT_TILE - 1) / DFT_TILE); }

// Tubes t and t + 1 (t even) are neighbours in every slice and 2-element
// aligned: one load or store serves both.
template <typename T> static int pair_ok(const void* X, long tubes, int cols, long ld, long ss) {
    return ld == cols && (ss & 1) == 0 && (tubes & 1) == 0 && ((size_t)X & (2 * sizeof(T) - 1)) == 0;
}
// the same for the spectrum's (h, tubes) rows, 16 bytes a store in float32
template <typename T> static int hat_pair_ok(const void* Xh, long tubes) {
    return (tubes & 1) == 0 && ((size_t)Xh & 15) == 0;
}

// Float64 transforms of few tubes take a CTA per sub-tile: the time is that of
// one SM's float64 units on its 16 sequences (n = 73, 1600 tubes in 50 tiles:
// 41 -> 31 us), and most SMs would be idle.  Not where the norm
// partials are wanted, which are one per tile.
template <typename T> static bool dft_split(unsigned tiles, const double* sumsq) {
    return sizeof(T) == 8 && !sumsq && tiles <= 76;
}

template <typename T>
tp_status rdft(const T* X, void* Xh, int n, int rows, int cols, long ld, long ss, double* sumsq,
               const int* skip, cudaStream_t st) {
    const long tubes = (long)rows * cols;
    if (tubes == 0) return TP_OK;
    const unsigned tiles = (unsigned)((tubes + DFT_TILE - 1) / DFT_TILE);
    const DftPlan& P = dft_plan(n, sizeof(T), true, dft_split<T>(tiles, sumsq));
    auto kern = P.cls == 0 ? k_rdft<T, 0> : (P.cls == 1 ? k_rdft<T, 1> : (P.cls == 2 ? k_rdft<T, 2> : k_rdft<T, 3>));
    if (smem_optin((const void*)kern, P.smem) != TP_OK) return TP_ERR_CUDA;
    prof_begin(TP_KC_DFT, st);
    kern<<<tiles * (P.split ? DFT_SEQ >> P.lns : 1), P.nt, P.smem, st>>>(
        P, X, (cplx<T>*)Xh, tubes, cols, ld, ss, pair_ok<T>(X, tubes, cols, ld, ss), hat_pair_ok<T>(Xh, tubes), sumsq,
        skip);
    return launched(TP_KC_DFT, st);
}

template <typename T>
tp_status irdft(const void* Xh, T* X, int n, int rows, int cols, long ld, long ss, const int* skip,
                cudaStream_t st) {
    const long tubes = (long)rows * cols;
    if (tubes == 0) return TP_OK;
    const unsigned tiles = (unsigned)((tubes + DFT_TILE - 1) / DFT_TILE);
    const DftPlan& P = dft_plan(n, sizeof(T), false, dft_split<T>(tiles, nullptr));
    auto kern =
        P.cls == 0 ? k_irdft<T, 0> : (P.cls == 1 ? k_irdft<T, 1> : (P.cls == 2 ? k_irdft<T, 2> : k_irdft<T, 3>));
    if (smem_optin((const void*)kern, P.smem) != TP_OK) return TP_ERR_CUDA;
    prof_begin(TP_KC_DFT, st);
    kern<<<tiles * (P.split ? DFT_SEQ >> P.lns : 1), P.nt, P.smem, st>>>(
        P, (const cplx<T>*)Xh, X, tubes, cols, ld, ss, hat_pair_ok<T>(Xh, tubes), pair_ok<T>(X, tubes, cols, ld, ss),
        skip);
    return launched(TP_KC_DFT, st);
}

// ||X||_F^2 from a half spectrum (h = n/2 + 1 slices of rows x cols), in the
// same rdft_parts(rows, cols) partial sums the forward transform writes:
// Parseval, (1/n) sum_s w_s ||X-hat_s||^2.  Partial b covers the entries
// DFT_TILE b .. DFT_TILE (b+1) - 1 of every slice; the 256 threads of its CTA
// take the 32 entries of eight slices at a time (their loads independent), and
// the sum runs in a fixed order (per thread in the working precision, across
// threads in float64).
template <typename T>
__global__ void __launch_bounds__(256) k_norm2_hat(const cplx<T>* __restrict__ Xh, int n, int h, long rc, int nparts,
                                                   double* parts) {
    __shared__ double red[33];
    const int b = blockIdx.x, t = threadIdx.x & (DFT_TILE - 1), g = threadIdx.x / DFT_TILE;
    const int ng = blockDim.x / DFT_TILE;
    const long e = (long)b * DFT_TILE + t;
    double acc = 0.0;
    if (e < rc)
#pragma unroll 4
        for (int s = g; s < h; s += ng) acc += parseval_w(s, n) * (double)cabs2(__ldg(Xh + (long)s * rc + e));
    acc = block_sum_t(acc, red);
    if (threadIdx.x == 0) parts[b] = acc / (double)n;
}

template <typename T>
tp_status norm2_hat(const void* Xh, int n, int rows, int cols, double* parts, cudaStream_t st) {
    const int np = rdft_parts(rows, cols), h = n / 2 + 1;
    prof_begin(TP_KC_DFT, st);
    k_norm2_hat<T><<<np, 256, 0, st>>>((const cplx<T>*)Xh, n, h, (long)rows * cols, np, parts);
    return launched(TP_KC_DFT, st);
}
template tp_status norm2_hat<float>(const void*, int, int, int, double*, cudaStream_t);
template tp_status norm2_hat<double>(const void*, int, int, int, double*, cudaStream_t);

template tp_status rdft<float>(const float*, void*, int, int, int, long, long, double*, const int*, cudaStream_t);
template tp_status rdft<double>(const double*, void*, int, int, int, long, long, double*, const int*, cudaStream_t);
template tp_status irdft<float>(const void*, float*, int, int, int, long, long, const int*, cudaStream_t);
template tp_status irdft<double>(const void*, double*, int, int, int, long, long, const int*, cudaStream_t);

}  // namespace tp
