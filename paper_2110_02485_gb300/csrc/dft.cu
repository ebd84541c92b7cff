// Mode-3 DFT along the tubes of a frontal-slice-major tensor (Section 2:
// fft(A,[],3) and its inverse), real data <-> half spectrum, any n.
//
// Every tube is transformed by itself: no sum or product takes entries of two
// tubes, so a tube's error is relative to its own norm whatever lies beside it
// (lateral slices of very different scale, zeros, a NaN).  Two tubes as the real
// and imaginary part of one complex sequence halve the work too, but carry the
// larger one's rounding into the smaller: a slice 1e-6 of its neighbour came out
// with a relative error of 6e-2.
//
// One CTA owns 32 neighbouring tubes, a lane each: a row of a slice is 128 bytes a
// warp, a row of the spectrum 256.  n = first M, M = r_0 r_1 ..: decimation in
// frequency, whose first step is a real DFT of `first` points over the rows j, j + M,
// .., j < M; only its outputs k <= first / 2 are kept (the others are conjugates),
// times exp(-2 pi i j k / n): blocks of M complex words, whose DFTs are the frequencies
// k + first k2, one pass per radix r_i <= 16 (the register DFTs below).
//   forward: the first pass reads its rows straight from global memory, the last
//     one writes its frequencies straight to the spectrum (the conjugate where
//     one is above n / 2);
//   inverse: the transpose: the first pass reads the blocks from the half spectrum
//     (re and im swapped: the inverse DFT is the swapped DFT of the swapped data),
//     the last one is the real inverse of `first` points, whose rows go to global
//     memory.
// So n = first r_0 moves every element through shared memory once.  Where n has
// primes above 13, their product is `first` and its real DFTs are direct sums
// (e_q, o_q below), formed on pairs of tubes part by part.
//
// What bounds it: HBM (about 4 bytes per element to read and 4 to write, in
// either direction), short of it the issue rate and, at n near 256, the loads in
// flight.  Measured on 256 x 256 tubes with buffers that exceed the L2 (CUDA events
// over a graph of launches, forward / inverse), and before: the direct sums over n
// that every n but the powers of two took (1), a radix-2 kernel for those and
// 16 x 16 and 16 x 32 forms for n = 256 and 512, and two tubes as one complex sequence (2):
//   n     now                      (1)              (2)
//   96    15.2 / 16.3 us           111 / 135        14.6 / 15.0
//   128   14.2 / 16.5 us           49 / 32          14.2 / 16.6
//   256   29.7 / 32.8 us (4.5 TB/s) 31 / 37         29.9 / 34.1
//   331   280 / 267 us             1166 / 1480      324 / 283   (prime)
//   384   49.0 / 49.9 us (4.1 TB/s) 1571 / 1980     53.5 / 55.2
//   512   62.0 / 67.3 us (4.3 TB/s) 73 / 123        73.0 / 77.8
//   1000  210 / 182 us             18651 / 19087    215 / 178
// The forward's root mean square error at 256 and 384 is 0.90e-7 and 0.95e-7 (0.99e-7 and
// 1.19e-7 in the form (2)): the first sums and differences are taken on exact data.
//
// A tile with a NaN, an infinity or squares that overflow evaluates the defining
// sums instead (rare, slow): an infinity stays in the entries it reaches.
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
constexpr int DFT_MAX_THREADS = 256;
constexpr int DFT_MAX_PASS = 10;
constexpr unsigned DFT_FULL = 4 * 152;  // tiles from which on every SM holds several CTAs

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

// R reals: X_k, k <= R / 2, and back, from e_q = x_q + x_{R-q} and o_q = x_q - x_{R-q}
// (formed first: exact, or nearly, on the symmetric tubes that blurs have).
//   R odd: X_k = (x_0 + sum e_q cos(2 pi q k / R), -sum o_q sin(2 pi q k / R)); the same sums,
//     with (Re X_k, Im X_k) for (e, o), give the outputs q and R - q as their sum and difference.
//   R even, H = R / 2: the even X_k are the DFT of length H of x_t + x_{t+H}, whose pairs are
//     e_q + e_{H-q} and o_q - o_{H-q}; the odd ones are the sums over e_q - e_{H-q} and o_q + o_{H-q}
//     (cos changes its sign from q to H - q, sin does not).  The inverse is the transpose.
template <typename T, int R> struct RealDft {
    static constexpr int H = R / 2;                            // the last k
    static constexpr int E = R % 2 ? R / 2 : (R / 2 - 1) / 2;  // pairs (q, R - q), or (t, R / 2 - t)
    // v += (sum e_q cos(2 pi q k / R), -sum o_q sin(2 pi q k / R)), q = 1 .. E
    template <int K, int Q> static __device__ __forceinline__ void terms(const T (&e)[E + 1], const T (&o)[E + 1], cplx<T>& v) {
        if constexpr (Q <= E) {
            constexpr double cd = root_cos(K * Q, R), sd = root_sin(K * Q, R);
            const T c = (T)cd, s = (T)sd;
            v.x = fma(e[Q], c, v.x);
            v.y = fma(-o[Q], s, v.y);
            terms<K, Q + 1>(e, o, v);
        }
    }
    template <int K, int STEP> static __device__ __forceinline__ void outputs(const T (&e)[E + 1], const T (&o)[E + 1],
                                                                              T mid, cplx<T> (&v)[H + 1]) {
        if constexpr (K <= H) {
            v[K] = mk<T>(e[0], K % 4 == 3 ? mid : -mid);
            terms<K, 1>(e, o, v[K]);
            if constexpr (2 * K == R) v[K].y = 0;
            outputs<K + STEP, STEP>(e, o, mid, v);
        }
    }
    // P = (R - 1) / 2 pairs e, o (entries 1 .. P), x_0 and, R even, x_{R/2}
    static constexpr int P = (R - 1) / 2;
    static __device__ __forceinline__ void from_pairs(T x0, T xh, const T (&e)[P + 1], const T (&o)[P + 1],
                                                      cplx<T> (&v)[H + 1]) {
        if constexpr (R % 2) {
            T a[P + 1], s = x0;
            a[0] = x0;
#pragma unroll
            for (int q = 1; q <= P; ++q) {
                a[q] = e[q];
                s += e[q];
            }
            outputs<1, 1>(a, o, (T)0, v);
            v[0] = mk<T>(s, 0);
        } else {
            typedef RealDft<T, H> Half;
            T e2[Half::P + 1], o2[Half::P + 1], a[E + 1], b[E + 1];
            cplx<T> u[H / 2 + 1];
            e2[0] = o2[0] = b[0] = 0;
#pragma unroll
            for (int q = 1; q <= Half::P; ++q) {
                e2[q] = e[q] + e[H - q];
                o2[q] = o[q] - o[H - q];
            }
            Half::from_pairs(x0 + xh, H % 2 ? (T)0 : e[H / 2], e2, o2, u);
#pragma unroll
            for (int k = 0; k <= H / 2; ++k) v[2 * k] = u[k];
            a[0] = x0 - xh;
#pragma unroll
            for (int q = 1; q <= E; ++q) {
                a[q] = e[q] - e[H - q];
                b[q] = o[q] + o[H - q];
            }
            outputs<1, 2>(a, b, H % 2 ? (T)0 : o[H / 2], v);
        }
    }
    static __device__ __forceinline__ void forward(const T (&x)[R], cplx<T> (&v)[H + 1]) {
        T e[P + 1], o[P + 1];
        e[0] = o[0] = 0;
#pragma unroll
        for (int q = 1; q <= P; ++q) {
            e[q] = x[q] + x[R - q];
            o[q] = x[q] - x[R - q];
        }
        from_pairs(x[0], R % 2 ? (T)0 : x[H], e, o, v);
    }
    // odd k of the inverse, the transposed sums: z += (sum a_k cos(2 pi t k / R), -sum b_k sin(2 pi t k / R))
    template <int TT, int K> static __device__ __forceinline__ void odd_terms(const cplx<T> (&v)[H + 1], cplx<T>& z) {
        if constexpr (K <= H) {
            constexpr double cd = root_cos(K * TT, R), sd = root_sin(K * TT, R);
            const T c = (T)cd, s = (T)sd;
            z.x = fma(v[K].x, c, z.x);
            z.y = fma(-v[K].y, s, z.y);
            odd_terms<TT, K + 2>(v, z);
        }
    }
    template <int TT> static __device__ __forceinline__ void odd_outputs(const cplx<T> (&v)[H + 1], T (&z)[H > 0 ? H : 1]) {
        if constexpr (TT <= E) {
            cplx<T> c = mk<T>(0, 0);
            odd_terms<TT, 1>(v, c);
            z[TT] = c.x + c.y;
            z[H - TT] = c.y - c.x;
            odd_outputs<TT + 1>(v, z);
        }
    }
    // x_q = sum_k v_k.x cos(2 pi q k / R) - v_k.y sin(2 pi q k / R): the caller has doubled the k that stand for two
    static __device__ __forceinline__ void inverse(const cplx<T> (&v)[H + 1], T (&x)[R]) {
        if constexpr (R % 2) {
            T e[E + 1], o[E + 1], s = v[0].x;
            cplx<T> w[H + 1];
#pragma unroll
            for (int k = 0; k <= E; ++k) {
                e[k] = v[k].x;
                o[k] = v[k].y;
                if (k > 0) s += e[k];
            }
            outputs<1, 1>(e, o, (T)0, w);
            x[0] = s;
#pragma unroll
            for (int q = 1; q <= E; ++q) {
                x[q] = w[q].x + w[q].y;
                x[R - q] = w[q].x - w[q].y;
            }
        } else {
            cplx<T> u[H / 2 + 1];
            T y[H], z[H];
#pragma unroll
            for (int k = 0; k <= H / 2; ++k) u[k] = v[2 * k];
            RealDft<T, H>::inverse(u, y);
            z[0] = 0;
            if constexpr (H % 2 == 0) z[H / 2] = 0;
#pragma unroll
            for (int k = 1; k <= H; k += 2) {
                z[0] += v[k].x;
                if constexpr (H % 2 == 0) z[H / 2] += k % 4 == 3 ? v[k].y : -v[k].y;
            }
            odd_outputs<1>(v, z);
#pragma unroll
            for (int t = 0; t < H; ++t) {
                x[t] = y[t] + z[t];
                x[t + H] = y[t] - z[t];
            }
        }
    }
};
template <typename T> struct RealDft<T, 1> {
    static constexpr int P = 0;
    static __device__ __forceinline__ void from_pairs(T x0, T, const T (&)[1], const T (&)[1], cplx<T> (&v)[1]) {
        v[0] = mk<T>(x0, 0);
    }
    static __device__ __forceinline__ void forward(const T (&x)[1], cplx<T> (&v)[1]) { v[0] = mk<T>(x[0], 0); }
    static __device__ __forceinline__ void inverse(const cplx<T> (&v)[1], T (&x)[1]) { x[0] = v[0].x; }
};

constexpr int DFT_FIRST[] = {32, 24, 20, 18, 16, 15, 14, 13, 12, 11, 10, 9, 8, 7, 6, 5, 4, 3, 2, 1};  // real
constexpr int DFT_RADICES[] = {16, 15, 13, 12, 11, 10, 9, 8, 7, 6, 5, 4, 3, 2, 1};

// ---- the plan -------------------------------------------------------------------
struct DftPlan {
    int n = 0, first, M;      // n = first M: the real radix (or direct part), and the length of its blocks
    int D, np;                // direct part (the primes above 13); M = r[0] .. r[np-1]
    int r[DFT_MAX_PASS];
    unsigned ff, fm, rr[DFT_MAX_PASS], rm[DFT_MAX_PASS];  // ceil(2^20 / first), / M, / r and / (r's M, see pass_smem)
    int len;                  // complex words per tube: blocks 0 .. first / 2
    int lns;                  // log2 of the tubes per sub-tile
    int nt;                   // threads per CTA
    int kb;                   // direct part: pairs (k, D - k) per thread
    int cls;                  // dft_class
    bool split, full;         // one CTA per sub-tile; tiles for several CTAs on every SM
    size_t smem;
};
enum { DFT_GENERAL = 3, DFT_DIRECT = 4, DFT_CLASSES = 5 };

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

// Tubes per sub-tile: a whole tile while two CTAs fit on an SM, else a half or
// a quarter, one after another.  A direct part works on pairs of tubes (n words
// of two reals each) beside the blocks, where there are any.
static size_t dft_smem(const DftPlan& P, size_t elem) {
    const size_t c = 2 * elem;
    size_t words = (size_t)P.len << P.lns;
    if (P.cls == DFT_DIRECT) words = ((size_t)P.n << (P.lns - 1)) + (P.M > 1 ? words : 0);
    return (words + P.n) * c + (((size_t)P.n * 2 + 15) & ~(size_t)15);
}

// Class of a plan: 0 = powers of two, 1 = radices up to 10, 2 = the other
// products of small primes, 3 = those whose tiles are split (the others have
// the tube count as a compile-time constant), 4 = lengths with a direct part (and 1).
static int dft_class(const DftPlan& P) {
    if (P.D > 1 || P.n == 1) return DFT_DIRECT;
    if (P.lns != 5) return DFT_GENERAL;
    int cls = 0;
    for (int i = -1; i < P.np; ++i) {
        const int r = i < 0 ? P.first : P.r[i];
        if (r > 10 && r != 16) return 2;
        if (r & (r - 1)) cls = 1;
    }
    for (int i = -1; i < P.np; ++i)
        if (cls == 1 && (i < 0 ? P.first : P.r[i]) > 10) return 2;
    return cls;
}
// split: a CTA per sub-tile of eight tubes instead of per tile; full: tiles for
// several CTAs on every SM
static DftPlan make_plan(int n, size_t elem, bool split, bool full) {
    DftPlan P;
    P.n = n;
    P.split = split;
    P.full = full;
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
    int cur[DFT_MAX_PASS];
    if (P.D > 1 || n == 1) {
        int sum = INT_MAX;
        P.first = P.D;
        P.np = DFT_MAX_PASS;
        best_radices(m, 0, 0, 0, cur, P.r, &P.np, &sum);
    } else {
        // Fewest passes, then the least arithmetic, about W words times the radix of a complex pass and 0.3 n times the
        // real one (fitted to n = 96 .. 384; float32 radices above 10 take more registers: a tenth more).  A single pass of a wide radix counts as
        // two: most lanes of a small tile would idle (n = 32 in float64, one pass of 32 and 8 x 4: 15.8 and 6.7 us for
        // 32 x 32 tubes; n = 24 in float32, 256 x 256 tubes: 8.2 and 5.3 us).
        int passes = INT_MAX;
        double cost = 0.0;
        for (int i = 0; DFT_FIRST[i] > 1; ++i) {
            const int f = DFT_FIRST[i], rest = m / f;
            if (m % f) continue;
            int r[DFT_MAX_PASS], np = DFT_MAX_PASS, sum = INT_MAX;
            best_radices(rest, 0, 0, 0, cur, r, &np, &sum);
            const int total = np + 1 + (np == 0 && f >= 8 ? 1 : 0);
            double c = (double)(f / 2 + 1) * rest * (np ? sum : 0) + 0.3 * n * f;
            if (elem == 4 && (f > 10 || (np && r[0] > 10)) && (n & (n - 1))) c *= 1.1;
            if (total < passes || (total == passes && c < cost)) {
                passes = total;
                cost = c;
                P.first = f;
                P.np = np;
                std::copy(r, r + np, P.r);
            }
        }
    }
    P.M = n / P.first;
    P.len = (P.first / 2 + 1) * P.M;
    // x / d = x ceil(2^20 / d) >> 20 for x <= 1024, d <= 1024
    auto inverse = [](int d) { return ((1u << 20) + d - 1) / d; };
    P.ff = inverse(P.first);
    P.fm = inverse(P.M);
    for (int i = 0, L = P.M; i < P.np; ++i) {
        P.rr[i] = inverse(P.r[i]);
        L /= P.r[i];
        P.rm[i] = inverse(L);
    }
    P.lns = split ? 3 : 5;
    P.cls = dft_class(P);
    while (P.lns > 3 && dft_smem(P, elem) > 112 * 1024) --P.lns;
    P.cls = dft_class(P);
    P.smem = dft_smem(P, elem);
    // a thread per item of the first pass
    const int items = P.M << P.lns;
    P.nt = std::min(DFT_MAX_THREADS, std::max(64, (items + 31) & ~31));
    // where tiles fill the SMs, fewer threads keep more tiles (and loads) in flight (n = 128, 256 x 256 tubes, 256 and
    // 128 threads: 18.0 and 14.4 us; with 200 tiles in all 4.1 and 4.3 us), more so beside three CTAs of 256 than four
    // (n = 240: 34.3 and 30.7 us; n = 256: 30.5 and 33.9)
    const int want = (P.len << P.lns) / 24;
    if (full && P.cls < 2) P.nt = std::min(P.nt, want <= 64 ? 64 : (want <= 144 ? 128 : DFT_MAX_THREADS));
    if (full && P.cls >= 2) P.nt = std::min(P.nt, want <= 64 ? 64 : (want <= 224 ? 128 : (want <= 250 ? 192 : DFT_MAX_THREADS)));
    // The direct part: M columns of groups of kb pairs on a quarter as many lanes as tubes, about 12 kb + 4 instructions
    // per entry.  Up to about 370 points one round of some width does (17 .. 61 points on 64 or 128 threads, 331 on
    // 256): the cheapest of those, counting no fewer than three warps (fewer leave the SM waiting).  Beyond, 256 threads
    // and the fewest rounds, about kb + 1/2 units of time each.
    P.kb = 2;
    if (P.D > 1) {
        int cost1 = INT_MAX, cost2 = INT_MAX, nt1 = 0, kb1 = 0, kb2 = 4;
        for (int nt = DFT_MAX_THREADS; nt >= 64; nt /= 2)
            for (int kb : {2, 3, 4, 6}) {
                const int slots = nt >> (P.lns - 2), groups = P.M * ((P.D / 2 + kb) / kb);
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
    }
    return P;
}

// The plans of the last lengths that a thread used (the search takes some
// microseconds, which a small transform would notice).  A solve uses one length with
// few and with many tiles, split and not: a slot for each.
static const DftPlan& dft_plan(int n, size_t elem, bool split, bool full) {
    struct Slot {
        DftPlan P;
        size_t elem = 0;
    };
    thread_local Slot slots[64];
    Slot& s = slots[((n << 3) | (elem == 4 ? 4 : 0) | (split ? 2 : 0) | (full ? 1 : 0)) & 63];
    if (s.elem != elem || s.P.n != n || s.P.split != split || s.P.full != full) {
        s.P = make_plan(n, elem, split, full);
        s.elem = elem;
    }
    return s.P;
}

// CTAs per SM that the registers of each class allow (float32)
constexpr int DFT_CTAS[DFT_CLASSES] = {4, 4, 3, 2, 2};

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

// Digits of x < M in the mixed radix r_0, r_1, .., lowest first, read in the other
// direction (weights M / r_0, M / (r_0 r_1), ..): the position in a block of its
// frequency x after the passes.
__device__ __forceinline__ int dft_reverse(const DftPlan& P, int x) {
    int pos = 0, w = P.M;
    for (int i = 0; i < P.np; ++i) {
        const int q = (int)((x * P.rr[i]) >> 20);
        w = (int)((w * P.rr[i]) >> 20);
        pos += (x - q * P.r[i]) * w;
        x = q;
    }
    return pos;
}

// n roots exp(-2 pi i m / n), and what the passes do to the order:
//   forward: table[position] = its frequency,
//   inverse: table[position in a block] = time index in the block.
template <typename T, bool FWD>
__device__ __forceinline__ void fill_tables(const DftPlan& P, cplx<T>* tw, unsigned short* table) {
    const int n = P.n, M = P.M;
    const T step = (T)2 / (T)n;
    const bool pow2 = (n & (n - 1)) == 0;  // 2 m / n without a division then
    for (int m = threadIdx.x; m < n; m += blockDim.x) {
        T s, c;
        sincospi_t<T>(pow2 ? (T)m * step : (T)(2 * m) / (T)n, &s, &c);
        tw[m] = mk<T>(c, -s);
        const int k2 = (int)((m * P.ff) >> 20), k1 = m - k2 * P.first;
        if (FWD && 2 * k1 <= P.first) table[k1 * M + dft_reverse(P, k2)] = (unsigned short)m;
        if (!FWD && m < M) table[dft_reverse(P, m)] = (unsigned short)m;
    }
}

// One pass over shared memory (len words per tube): blocks of length L, radix R,
// M = L / R.  MR = ceil(2^20 / M) divides item numbers by M.
template <typename T, int R>
__device__ __forceinline__ void pass_smem(cplx<T>* z, const cplx<T>* tw, int len, int L, int tstep, unsigned MR, int lns) {
    const int p = threadIdx.x & ((1 << lns) - 1), ust = blockDim.x >> lns, items = len / R, M = L / R;
    for (int u = threadIdx.x >> lns; u < items; u += ust) {
        const int b = (int)((u * MR) >> 20), j = u - b * M;
        cplx<T>* zp = z + ((size_t)(b * L + j) << lns) + p;
        cplx<T> v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = zp[(q * M) << lns];
        RDft<T, R>::run(v);
        zp[0] = v[0];
#pragma unroll
        for (int k = 1; k < R; ++k) zp[(k * M) << lns] = M == 1 ? v[k] : cmul(v[k], tw[j * k * tstep]);
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

// the first radix
#define DFT_SWITCH_FIRST(r, GO)                              \
    if constexpr (CLS >= 2) {                                \
        switch (r) {                                         \
            case 14: GO(14); break;                          \
            case 18: GO(18); break;                          \
            case 20: GO(20); break;                          \
            case 24: GO(24); break;                          \
            case 32: GO(32); break;                          \
            default: DFT_SWITCH(r, GO)                       \
        }                                                    \
    } else {                                                 \
        DFT_SWITCH(r, GO)                                    \
    }

// Items of a first pass whose R entries a thread loads before it uses any.
constexpr int dft_batch(int R) { return R >= 12 ? 1 : (R >= 6 ? 2 : (R > 1 ? 4 : 8)); }

// First forward pass: rows j, j + M, .. of a tube (M = n / R); blocks k <= R / 2 of
// length M.
template <typename T, int R>
__device__ __forceinline__ void pass_load(cplx<T>* z, const cplx<T>* tw, int n, int lns, const T* x, bool live, long ss,
                                          T& acc) {
    constexpr int U = (R == 16 || R == 8 ? 2 : 1) * dft_batch(R);  // powers of two: 32 loads (30.5 -> 29.7 us at n = 256)
    const int p = threadIdx.x & ((1 << lns) - 1), M = n / R, ust = blockDim.x >> lns;
    for (int j0 = threadIdx.x >> lns; j0 < M; j0 += U * ust) {
        T a[U][R];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int j = j0 + u * ust;
                a[u][q] = live && j < M ? __ldcs(x + (long)(j + q * M) * ss) : (T)0;
            }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = j0 + u * ust;
            if (j >= M) break;
            cplx<T> v[R / 2 + 1];
#pragma unroll
            for (int q = 0; q < R; ++q) acc = fma(a[u][q], a[u][q], acc);
            RealDft<T, R>::forward(a[u], v);
            cplx<T>* zp = z + ((size_t)j << lns) + p;
            zp[0] = v[0];
#pragma unroll
            for (int k = 1; k <= R / 2; ++k) zp[(k * M) << lns] = cmul(v[k], tw[j * k]);
        }
    }
}

// Frequency f of a tube (dst: its column of the spectrum), or, above n / 2, its
// conjugate to n - f; blocks 0 and first / 2 hold n - f themselves (twice: not one of
// those).
template <typename T>
__device__ __forceinline__ void put_hat(cplx<T>* dst, long tubes, int n, int f, bool twice, cplx<T> v) {
    if (f == 0 || 2 * f == n) v.y = 0;
    if (2 * f <= n) dst[(long)f * tubes] = v;
    else if (twice) dst[(long)(n - f) * tubes] = cconj(v);
}

// Last forward pass: block u's frequencies low + (n / R) k to the spectrum.
template <typename T, int R>
__device__ __forceinline__ void pass_out(const cplx<T>* z, const unsigned short* freq, int n, int len, int lns, int lo,
                                         int hi, cplx<T>* dst, bool live, long tubes) {
    const int p = threadIdx.x & ((1 << lns) - 1), ust = blockDim.x >> lns, items = len / R, M = n / R;
    for (int u = threadIdx.x >> lns; u < items; u += ust) {
        const cplx<T>* zp = z + ((size_t)(u * R) << lns) + p;
        cplx<T> v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = zp[q << lns];
        RDft<T, R>::run(v);
        const int low = freq[u * R];  // the last digit is 0
        const bool twice = u * R >= lo && u * R < hi;
        if (live)
#pragma unroll
            for (int k = 0; k < R; ++k) put_hat<T>(dst, tubes, n, low + k * M, twice, v[k]);
    }
}

// First inverse pass over the blocks k1 <= r0 / 2 of length M = n / r0: word k2 of block
// k1 is frequency f = k1 + r0 k2, the conjugate of n - f above n / 2 (blocks 0 and r0 / 2
// read theirs twice), re and im swapped.  R = 1: a copy.
template <typename T, int R, typename Note>
__device__ __forceinline__ void pass_load_hat(cplx<T>* z, const cplx<T>* tw, int n, int r0, int M, int len, unsigned MR,
                                              int lns, const cplx<T>* src, bool live, long tubes, Note note) {
    const int p = threadIdx.x & ((1 << lns) - 1), ust = blockDim.x >> lns, items = len / R, Q = M / R;
    constexpr int U = dft_batch(R);
    for (int u0 = threadIdx.x >> lns; u0 < items; u0 += U * ust) {
        cplx<T> v[U][R];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int u = u0 + i * ust, k1 = (int)((u * MR) >> 20), j = u - k1 * Q;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int f = k1 + r0 * (j + q * Q);
                v[i][q] = live && u < items ? src[(long)(2 * f <= n ? f : n - f) * tubes] : mk<T>(0, 0);
            }
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int u = u0 + i * ust, k1 = (int)((u * MR) >> 20), j = u - k1 * Q;
            if (u >= items) break;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int f = k1 + r0 * (j + q * Q);
                if (f == 0 || 2 * f == n) v[i][q].y = 0;  // the imaginary parts of slices 0 and n / 2 are ignored
                note(v[i][q]);
                v[i][q] = mk<T>(2 * f <= n ? v[i][q].y : -v[i][q].y, v[i][q].x);
            }
            RDft<T, R>::run(v[i]);
            cplx<T>* zp = z + ((size_t)(k1 * M + j) << lns) + p;
            zp[0] = v[i][0];
#pragma unroll
            for (int k = 1; k < R; ++k) zp[(k * Q) << lns] = Q == 1 ? v[i][k] : cmul(v[i][k], tw[j * k * r0]);
        }
    }
}

// Last inverse pass: the blocks' entries at one position, times exp(2 pi i j k / n) (j
// its time index), to the rows j + M q of the tube.
template <typename T, int R>
__device__ __forceinline__ void pass_store(const cplx<T>* z, const cplx<T>* tw, const unsigned short* time, int n, int lns,
                                           T* x, bool live, long ss, T inv) {
    const int p = threadIdx.x & ((1 << lns) - 1), M = n / R, ust = blockDim.x >> lns;
    for (int u = threadIdx.x >> lns; u < M; u += ust) {
        const cplx<T>* zp = z + ((size_t)u << lns) + p;
        const int j = time[u];
        T o[R];
        cplx<T> a[R / 2 + 1];
        a[0] = mk<T>(zp[0].y * inv, 0);
#pragma unroll
        for (int k = 1; k <= R / 2; ++k) {
            const cplx<T> v = zp[(k * M) << lns], w = tw[j * k];  // (im, re); cos - i sin
            const T g = 2 * k == R ? inv : 2 * inv;
            a[k] = mk<T>((v.y * w.x + v.x * w.y) * g, (v.x * w.x - v.y * w.y) * g);
        }
        RealDft<T, R>::inverse(a, o);
        if (live)
#pragma unroll
            for (int q = 0; q < R; ++q) x[(long)(j + q * M) * ss] = o[q];
    }
}

// The direct part: real DFTs of odd length D over the rows j, j + M, .. of each column
// j < M, on pairs of tubes (a word holds an entry of tube 2 p and one of tube 2 p + 1, which
// never meet: every sum is formed part by part).  The rows j + M q and j + M (D - q)
// hold e_q and o_q; a thread forms KB pairs (k, D - k) of two neighbouring pairs of
// tubes, so each twiddle and each (e, o) read serves several products (about two thirds of
// the issue slots are multiply-adds).  put(j, k, pair, A, B) takes A = x_0 + sum e_q
// cos(2 pi q k / D) and B = -sum o_q sin(2 pi q k / D).
template <typename T, int KB, typename Put>
__device__ __forceinline__ void direct_sums(const cplx<T>* z, const cplx<T>* tw, int M, int D, int lnp, Put put) {
    typedef cplx<T> V;
    const int H = D / 2;  // twiddles exp(-2 pi i m / D) = tw[m M]
    const int lhs = lnp - 1, sp = threadIdx.x & ((1 << lhs) - 1), gst = blockDim.x >> lhs;
    const int ng = (H + KB) / KB;  // groups of KB values of k in 0 .. H
    const size_t row = (size_t)M << lnp;
    for (int it = threadIdx.x >> lhs; it < M * ng; it += gst) {
        const int j = it / ng, k0 = (it - j * ng) * KB;
        const V* zj = z + ((size_t)j << lnp) + 2 * sp;
        V A[KB][2], B[KB][2];
        int idx[KB], kk[KB];
#pragma unroll
        for (int t = 0; t < KB; ++t) {
            kk[t] = min(k0 + t, H);
            idx[t] = 0;
            A[t][0] = zj[0];
            A[t][1] = zj[1];
            B[t][0] = B[t][1] = mk<T>(0, 0);
        }
        const V *ze = zj + row, *zo = zj + (D - 1) * row;
#pragma unroll 2
        for (int q = 1; q <= H; ++q, ze += row, zo -= row) {
            const V e0 = ze[0], e1 = ze[1], o0 = zo[0], o1 = zo[1];
#pragma unroll
            for (int t = 0; t < KB; ++t) {
                const unsigned nx = (unsigned)(idx[t] + kk[t]);
                idx[t] = (int)min(nx, nx - (unsigned)D);  // (q k) mod D
                const V w = tw[idx[t] * M];
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
#pragma unroll
        for (int t = 0; t < KB; ++t) {
            const int k = k0 + t;
            if (k > H) break;
#pragma unroll
            for (int c = 0; c < 2; ++c) put(j, k, 2 * sp + c, A[t][c], B[t][c]);
        }
    }
}
template <typename T, typename Put>
__device__ __forceinline__ void direct_part(const DftPlan& P, const cplx<T>* z, const cplx<T>* tw, int lnp, Put put) {
    if (P.kb == 2) direct_sums<T, 2>(z, tw, P.M, P.D, lnp, put);
    else if (P.kb == 3) direct_sums<T, 3>(z, tw, P.M, P.D, lnp, put);
    else if (P.kb == 4) direct_sums<T, 4>(z, tw, P.M, P.D, lnp, put);
    else direct_sums<T, 6>(z, tw, P.M, P.D, lnp, put);
}

// Rows of a pair of tubes to shared memory as e and o (rows j of q = 0 as they are).
template <typename T>
__device__ __forceinline__ void direct_load(cplx<T>* z, int M, int D, unsigned FM, int lnp, const T* x, const T* y, bool la, bool lb,
                                            long ss, T& acc) {
    typedef cplx<T> V;
    constexpr int U = 4;  // row pairs in flight per thread
    const int p = threadIdx.x & ((1 << lnp) - 1), ust = blockDim.x >> lnp, items = M * (D / 2 + 1);
    for (int u0 = threadIdx.x >> lnp; u0 < items; u0 += U * ust) {
        V a[U], b[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int u = u0 + i * ust, q = (int)((u * FM) >> 20), r = u - q * M + M * (q ? D - q : 0);  // rows u = j + M q and j + M (D - q)
            const bool ok = u < items;
            a[i] = mk<T>(ok && la ? __ldcs(x + (long)u * ss) : (T)0, ok && lb ? __ldcs(y + (long)u * ss) : (T)0);
            b[i] = mk<T>(ok && la && q ? __ldcs(x + (long)r * ss) : (T)0, ok && lb && q ? __ldcs(y + (long)r * ss) : (T)0);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int u = u0 + i * ust, q = (int)((u * FM) >> 20), r = u - q * M + M * (q ? D - q : 0);
            if (u >= items) break;
            acc = fma(a[i].x, a[i].x, fma(a[i].y, a[i].y, acc));
            acc = fma(b[i].x, b[i].x, fma(b[i].y, b[i].y, acc));
            z[((size_t)u << lnp) + p] = cadd(a[i], b[i]);
            if (q) z[((size_t)r << lnp) + p] = csub(a[i], b[i]);
        }
    }
}

template <typename T, int CLS>
__global__ void __launch_bounds__(DFT_MAX_THREADS, sizeof(T) == 4 ? DFT_CTAS[CLS] : 1)
k_rdft(const __grid_constant__ DftPlan P, const T* __restrict__ X, cplx<T>* __restrict__ Xh, long tubes, int cols,
       long ld, long ss, double* sumsq, const int* skip) {
    if (skip && *skip) return;
    typedef cplx<T> V;
    constexpr bool ANY = CLS >= DFT_GENERAL;  // any sub-tile
    extern __shared__ __align__(16) unsigned char smraw[];
    const int n = P.n, M = P.M, len = P.len, lns = ANY ? P.lns : 5, nts = 1 << lns, h = n / 2 + 1;
    V* zp = (V*)smraw;  // DIRECT: the pairs of tubes
    V* z = CLS == DFT_DIRECT ? zp + ((size_t)n << (lns - 1)) : zp;
    V* tw = CLS == DFT_DIRECT && M == 1 ? z : z + ((size_t)len << lns);
    unsigned short* freq = (unsigned short*)(tw + n);
    fill_tables<T, true>(P, tw, freq);
    __syncthreads();
    T total = 0;
    // all sub-tiles of tile blockIdx.x, or (split) one
    const int nsub = DFT_TILE >> lns;
    const long tile = ANY && P.split ? blockIdx.x / nsub : blockIdx.x;
    const int sub0 = ANY && P.split ? (blockIdx.x % nsub) << lns : 0;
    const int sub1 = ANY && P.split ? sub0 + nts : DFT_TILE;
    for (int sub = sub0; sub < sub1; sub += nts) {
        const long f0 = tile * DFT_TILE + sub, t0 = f0 + (threadIdx.x & (nts - 1));
        const bool live = t0 < tubes;
        T acc = 0;
        if constexpr (CLS == DFT_DIRECT) {
            const long t = f0 + 2 * (threadIdx.x & ((nts >> 1) - 1));
            const bool la = t < tubes, lb = t + 1 < tubes;
            direct_load<T>(zp, M, P.D, P.fm, lns - 1, X + (la ? tube_off(t, cols, ld) : 0), X + (lb ? tube_off(t + 1, cols, ld) : 0), la,
                           lb, ss, acc);
        } else {
            const T* x = X + (live ? tube_off(t0, cols, ld) : 0);
#define GO(R) pass_load<T, R>(z, tw, n, lns, x, live, ss, acc)
            DFT_SWITCH_FIRST(P.first, GO)
#undef GO
        }
        const bool finite = !__syncthreads_or(!isfinite(acc));
        total += acc;
        if (!finite) {
            // the defining sum, tube by tube
            for (int e = threadIdx.x; e < h * nts; e += blockDim.x) {
                const int s = e >> lns;
                const long t = f0 + (e & (nts - 1));
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
        if constexpr (CLS == DFT_DIRECT) {
            direct_part<T>(P, zp, tw, lns - 1, [&](int j, int k, int q, V a, V b) {
                const V u = mk<T>(a.x, b.x), v = mk<T>(a.y, b.y);  // the two tubes
                if (M == 1) {
                    const long t = f0 + 2 * q;
                    V* dst = Xh + (long)k * tubes + t;
                    if (t < tubes) dst[0] = u;
                    if (t + 1 < tubes) dst[1] = v;
                } else {
                    const V w = tw[j * k];
                    V* dst = z + ((size_t)(k * M + j) << lns) + 2 * q;
                    dst[0] = cmul(u, w);
                    dst[1] = cmul(v, w);
                }
            });
            if (M > 1) __syncthreads();
        }
        int L = M, tstep = P.first;
        for (int i = 0; i < P.np - 1; ++i) {
#define GO(R) pass_smem<T, R>(z, tw, len, L, tstep, P.rm[i], lns)
            DFT_SWITCH(P.r[i], GO)
#undef GO
            tstep *= P.r[i];
            L = (int)((L * P.rr[i]) >> 20);
            __syncthreads();
        }
        const int lo = M, hi = (P.first + 1) / 2 * M;  // words of frequencies and of conjugates
        V* dst = Xh + t0;
        if (P.np > 0) {
#define GO(R) pass_out<T, R>(z, freq, n, len, lns, lo, hi, dst, live, tubes)
            DFT_SWITCH(P.r[P.np - 1], GO)
#undef GO
        } else if (CLS != DFT_DIRECT) {
            pass_out<T, 1>(z, freq, n, len, lns, lo, hi, dst, live, tubes);
        }
        if (nts < DFT_TILE) __syncthreads();
    }
    if (sumsq) store_partial<T>(total, sumsq);
}

template <typename T, int CLS>
__global__ void __launch_bounds__(DFT_MAX_THREADS, sizeof(T) == 4 ? DFT_CTAS[CLS] : 1)
k_irdft(const __grid_constant__ DftPlan P, const cplx<T>* __restrict__ Xh, T* __restrict__ X, long tubes, int cols,
        long ld, long ss, const int* skip) {
    if (skip && *skip) return;
    typedef cplx<T> V;
    constexpr bool ANY = CLS >= DFT_GENERAL;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int n = P.n, M = P.M, len = P.len, lns = ANY ? P.lns : 5, nts = 1 << lns, h = n / 2 + 1;
    V* zp = (V*)smraw;
    V* z = CLS == DFT_DIRECT ? zp + ((size_t)n << (lns - 1)) : zp;
    V* tw = CLS == DFT_DIRECT && M == 1 ? z : z + ((size_t)len << lns);
    unsigned short* time = (unsigned short*)(tw + n);
    fill_tables<T, false>(P, tw, time);
    __syncthreads();
    const T inv = (T)1 / (T)n;
    const int nsub = DFT_TILE >> lns;
    const long tile = ANY && P.split ? blockIdx.x / nsub : blockIdx.x;
    const int sub0 = ANY && P.split ? (blockIdx.x % nsub) << lns : 0;
    const int sub1 = ANY && P.split ? sub0 + nts : DFT_TILE;
    for (int sub = sub0; sub < sub1; sub += nts) {
        const long f0 = tile * DFT_TILE + sub, t0 = f0 + (threadIdx.x & (nts - 1));
        const bool live = t0 < tubes;
        const V* src = Xh + t0;
        T bad = 0;  // stays 0 for finite data
        auto note = [&](V v) { bad = fma(v.x, (T)0, fma(v.y, (T)0, bad)); };
        if (P.np > 0) {
#define GO(R) pass_load_hat<T, R>(z, tw, n, P.first, M, len, P.rm[0], lns, src, live, tubes, note)
            DFT_SWITCH(P.r[0], GO)
#undef GO
        } else if constexpr (CLS == DFT_DIRECT) {
            // straight to the pairs of tubes: e = 2 Re X_s, o = 2 Im X_s
            const int np = nts >> 1, p = threadIdx.x & (np - 1);
            const long t = f0 + 2 * p;
            for (int s = threadIdx.x >> (lns - 1); s < h; s += blockDim.x >> (lns - 1)) {
                const V* x = Xh + (long)s * tubes + t;
                V a = t < tubes ? x[0] : mk<T>(0, 0), b = t + 1 < tubes ? x[1] : mk<T>(0, 0);
                if (s == 0) a.y = b.y = 0;  // the imaginary part of slice 0 is ignored
                note(a);
                note(b);
                const T g = s ? (T)2 : (T)1;
                zp[s * np + p] = mk<T>(g * a.x, g * b.x);
                if (s) zp[(n - s) * np + p] = mk<T>(g * a.y, g * b.y);
            }
        } else {
            pass_load_hat<T, 1>(z, tw, n, P.first, M, len, P.fm, lns, src, live, tubes, note);
        }
        const bool finite = !__syncthreads_or(bad != (T)0 || isnan(bad));
        if (!finite) {
            // the defining sum, tube by tube
            for (int e = threadIdx.x; e < n * nts; e += blockDim.x) {
                const int k = e >> lns;
                const long t = f0 + (e & (nts - 1));
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
        int L = M, tstep = P.first;
        for (int i = 0; i < P.np; ++i) {
            if (i > 0) {
#define GO(R) pass_smem<T, R>(z, tw, len, L, tstep, P.rm[i], lns)
                DFT_SWITCH(P.r[i], GO)
#undef GO
                __syncthreads();
            }
            tstep *= P.r[i];
            L = (int)((L * P.rr[i]) >> 20);
        }
        if constexpr (CLS == DFT_DIRECT) {
            if (M > 1) {
                // the blocks' entries at a position, times exp(2 pi i j k / n): e = 2 Re, o = 2 Im at row j + M k of the pairs
                T* zr = (T*)zp;
                for (int e = threadIdx.x >> lns; e < len; e += blockDim.x >> lns) {
                    const int k = (int)((e * P.fm) >> 20), j = time[e - k * M], t = threadIdx.x & (nts - 1);
                    const V v = z[((size_t)e << lns) + t], w = tw[j * k];  // (im, re); cos - i sin
                    const T g = k ? (T)2 : (T)1;
                    zr[((size_t)(j + M * k) << lns) + t] = (v.y * w.x + v.x * w.y) * g;
                    if (k) zr[((size_t)(j + M * (P.D - k)) << lns) + t] = (v.x * w.x - v.y * w.y) * g;
                }
                __syncthreads();
            }
            direct_part<T>(P, zp, tw, lns - 1, [&](int j, int k, int q, V a, V b) {
                const long t = f0 + 2 * q, up = (long)(j + M * k) * ss, down = (long)(j + M * (P.D - k)) * ss;
                if (t < tubes) {
                    T* o = X + tube_off(t, cols, ld);
                    o[up] = (a.x + b.x) * inv;
                    if (k > 0) o[down] = (a.x - b.x) * inv;
                }
                if (t + 1 < tubes) {
                    T* o = X + tube_off(t + 1, cols, ld);
                    o[up] = (a.y + b.y) * inv;
                    if (k > 0) o[down] = (a.y - b.y) * inv;
                }
            });
        } else {
            T* x = X + (live ? tube_off(t0, cols, ld) : 0);
#define GO(R) pass_store<T, R>(z, tw, time, n, lns, x, live, ss, inv)
            DFT_SWITCH_FIRST(P.first, GO)
#undef GO
        }
        if (nts < DFT_TILE) __syncthreads();
    }
}

int rdft_parts(int rows, int cols) { return (int)(((long)rows * cols + DFT_TILE - 1) / DFT_TILE); }

// Float64 transforms of few tubes take a CTA per sub-tile: the time is that of
// one SM's float64 units on its tile (n = 73, 1600 tubes in 50 tiles:
// 41 -> 31 us), and most SMs would be idle.  Not where the norm
// partials are wanted, which are one per tile.
template <typename T> static bool dft_split(unsigned tiles, const double* sumsq) {
    return sizeof(T) == 8 && !sumsq && tiles <= 76;
}

static unsigned dft_grid(const DftPlan& P, unsigned tiles) { return P.split ? tiles * (unsigned)(DFT_TILE >> P.lns) : tiles; }

template <typename T>
tp_status rdft(const T* X, void* Xh, int n, int rows, int cols, long ld, long ss, double* sumsq,
               const int* skip, cudaStream_t st) {
    const long tubes = (long)rows * cols;
    if (tubes == 0) return TP_OK;
    const unsigned tiles = (unsigned)((tubes + DFT_TILE - 1) / DFT_TILE);
    const DftPlan& P = dft_plan(n, sizeof(T), dft_split<T>(tiles, sumsq), tiles >= DFT_FULL);
    static constexpr decltype(&k_rdft<T, 0>) forms[DFT_CLASSES] = {k_rdft<T, 0>, k_rdft<T, 1>, k_rdft<T, 2>, k_rdft<T, 3>,
                                                                   k_rdft<T, 4>};
    const auto kern = forms[P.cls];
    if (smem_optin((const void*)kern, P.smem) != TP_OK) return TP_ERR_CUDA;
    prof_begin(TP_KC_DFT, st);
    kern<<<dft_grid(P, tiles), P.nt, P.smem, st>>>(P, X, (cplx<T>*)Xh, tubes, cols, ld, ss, sumsq, skip);
    return launched(TP_KC_DFT, st);
}

template <typename T>
tp_status irdft(const void* Xh, T* X, int n, int rows, int cols, long ld, long ss, const int* skip,
                cudaStream_t st) {
    const long tubes = (long)rows * cols;
    if (tubes == 0) return TP_OK;
    const unsigned tiles = (unsigned)((tubes + DFT_TILE - 1) / DFT_TILE);
    const DftPlan& P = dft_plan(n, sizeof(T), dft_split<T>(tiles, nullptr), tiles >= DFT_FULL);
    static constexpr decltype(&k_irdft<T, 0>) forms[DFT_CLASSES] = {k_irdft<T, 0>, k_irdft<T, 1>, k_irdft<T, 2>,
                                                                    k_irdft<T, 3>, k_irdft<T, 4>};
    const auto kern = forms[P.cls];
    if (smem_optin((const void*)kern, P.smem) != TP_OK) return TP_ERR_CUDA;
    prof_begin(TP_KC_DFT, st);
    kern<<<dft_grid(P, tiles), P.nt, P.smem, st>>>(P, (const cplx<T>*)Xh, X, tubes, cols, ld, ss, skip);
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
