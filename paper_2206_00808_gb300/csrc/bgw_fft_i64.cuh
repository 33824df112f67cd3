// FFT lines of FP64 data in 64-bit block fixed point.
//
// GB300 issues two FP64 operations per clock per SM: a warp's DFMA takes 64
// issue cycles of its scheduler, against 2 for a 32 x 32 + 64 bit multiply-add
// and 2 for a 64-bit add (measured).  A transform is nothing but sums of its
// inputs times roots of unity, so every value of it is bounded by a known
// multiple of the largest input component: one power of two per line is
// enough, and 64-bit integers hold more bits of it than FP64 does.
//
// A line of FP64 values is scaled by 2^s so that its largest component lies in
// [2^(T-1), 2^T), T = fix_top(N) = 57 or 58, and transformed in integers.  A
// twiddle product is
//   x w / 2 = xh wh + ((xh wl + xl wh) >> 32),   w in units of 2^-63, x = xh 2^32 + xl,
// with xl and wl signed, so that the dropped xl wl (below half a unit) has no
// bias; the halving takes back part of the growth of the radix that follows and
// saves the shifts of a full product (the factors that carry no twiddle are
// halved as well).  A line of N = R1 R2 ... leaves as DFT / 2^levels.  Against
// long double the error of a line is 0.3 to 0.5 of the FP64 transform's.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

#include "bgw_fft.cuh"

namespace bgw {

using i64c = cpx<long long>;

// Longest line held by one thread: 4 registers a point.
constexpr int kFixMaxN = 40;

// Twiddle levels of a length (each halves).
__host__ __device__ constexpr int fix_levels(int n) {
    const int m = n / first_radix(n);
    return m == 1 ? 0 : 1 + fix_levels(m);
}
// Growth of a component over the largest input component, in 2^-10, without
// the sqrt(2) of its rotation.
__host__ __device__ constexpr long fix_growth(int n) {
    const int r = first_radix(n), m = n / r;
    return m == 1 ? 1024L * r : fix_growth(m) * r / 2;
}
// Smallest b with 2^b >= sqrt(2) g / 1024.
__host__ __device__ constexpr int fix_bits(long g) {
    int b = 0;
    while ((1024L * 1024L << (2 * b)) < 2 * g * g) ++b;
    return b;
}
// Input components stay below 2^fix_top(n): the inputs of every twiddle then
// stay below 2^61 and the results below 2^62.
__host__ __device__ constexpr int fix_top(int n, int limit = 62) {
    const int m = n / first_radix(n);
    const int own = limit - fix_bits(fix_growth(n)), sub = m == 1 ? own : fix_top(m, 61);
    return own < sub ? own : sub;
}

// Roots exp(-2 pi i j / N) in units of 2^-63, each component as hi 2^32 + lo
// with lo signed: {cos hi, cos lo, sin hi, sin lo}; and real constants.
enum { kQsin3, kQsqrt8, kQcos5a, kQsin5a, kQcos5b, kQsin5b, kQnsin5a, kQcount };
static __constant__ int4 c_twq[kTwTotal];
static __constant__ int2 c_consq[kQcount];

// Both tables from the host's long double cosine and sine.
inline void fix_tables(int4 *tw, int2 *cons) {
    auto parts = [](long double v, int &h, int &l) {
        const long long n = std::llrint(v * 9223372036854775808.0L);   // 2^63
        l = (int)(unsigned)n;
        h = (int)((n - l) >> 32);
    };
    const long double pi = 3.14159265358979323846264338327950288419716939937510L;
    for (int i = 0; i < kNumFftLens; ++i)
        for (int n = kFftLens[i], j = 0; j < n; ++j) {
            int4 &w = tw[tw_offset(n) + j];
            w = {0, 0, 0, 0};
            if (4 * j % n == 0) continue;          // 1, i, -1, -i are never multiplied by
            parts(std::cos(2 * pi * j / n), w.x, w.y);
            parts(-std::sin(2 * pi * j / n), w.z, w.w);
        }
    // sqrt(3)/2 - 1 times two, sqrt(1/2), cos and sin of 2 pi/5 and 4 pi/5, -sin 2 pi/5
    const long double c[kQcount] = {2 * (std::sqrt(0.75L) - 1), std::sqrt(0.5L),       std::cos(2 * pi / 5),
                                    std::sin(2 * pi / 5),       std::cos(4 * pi / 5),  std::sin(4 * pi / 5),
                                    -std::sin(2 * pi / 5)};
    for (int i = 0; i < kQcount; ++i) parts(c[i], cons[i].x, cons[i].y);
}

// ------------------------------------------------------------- products --
struct fix_parts { int h, l; };
__device__ __forceinline__ fix_parts fix_split(long long x) {
    return {(int)(x >> 32) + (int)((unsigned)x >> 31), (int)(unsigned)x};
}
__device__ __forceinline__ long long fix_mad(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (long long)a * b + c;
#endif
}
constexpr long long kFixHalf = 1LL << 31;
// p + q / 2^32 (q carries its rounding half)
__device__ __forceinline__ long long fix_join(long long p, long long q) { return p + (q >> 32); }
// 2 (p + q / 2^32)
__device__ __forceinline__ long long fix_join2(long long p, long long q) { return (p << 1) + (q >> 31); }
// x w / 2, |x| <= 2^61.5
__device__ __forceinline__ long long fix_mul(long long x, int2 w) {
    const fix_parts s = fix_split(x);
    return fix_join(fix_mad(s.h, w.x, 0), fix_mad(s.h, w.y, fix_mad(s.l, w.x, kFixHalf)));
}
// a u + b v, |a| + |b| <= 2^61
__device__ __forceinline__ long long fix_mul2(long long a, int2 u, long long b, int2 v) {
    const fix_parts s = fix_split(a), t = fix_split(b);
    return fix_join2(fix_mad(s.h, u.x, fix_mad(t.h, v.x, 0)),
                     fix_mad(s.h, u.y, fix_mad(s.l, u.x, fix_mad(t.h, v.y, fix_mad(t.l, v.x, kFixHalf >> 1)))));
}
// x / 2; an odd x goes up or down by its next bit, so there is no bias
__device__ __forceinline__ long long fix_halve(long long x) { return (x >> 1) | (x & 1); }

// a w_N^E / 2
template <int S, int N, int NTOP, int E>
__device__ __forceinline__ i64c fix_twiddle(i64c a) {
    constexpr int e = E % N;
    if constexpr (4 * e % N == 0) {
        const long long x = fix_halve(a.x), y = fix_halve(a.y);
        if constexpr (e == 0) return {x, y};
        if constexpr (2 * e == N) return {-x, -y};
        if constexpr (4 * e == N) return {-S * y, S * x};
        return {S * y, -S * x};
    } else if constexpr (8 * e % N == 0) {        // odd powers of w_8: two products instead of four
        constexpr int o = 8 * e / N;              // 1, 3, 5, 7
        const long long p = fix_mul(a.x - S * a.y, c_consq[kQsqrt8]), m = fix_mul(a.y + S * a.x, c_consq[kQsqrt8]);
        if constexpr (o == 1) return {p, m};
        if constexpr (o == 3) return {-S * m, S * p};
        if constexpr (o == 5) return {-p, -m};
        return {S * m, -S * p};
    } else {
        constexpr int j = (S < 0 ? e : N - e) * (NTOP / N);
        const int4 w = c_twq[tw_offset(NTOP) + j], c = c_twq[tw_offset(NTOP) + NTOP - j];   // w and conj(w)
        const fix_parts x = fix_split(a.x), y = fix_split(a.y);
        return {fix_join(fix_mad(x.h, w.x, fix_mad(y.h, c.z, 0)),
                         fix_mad(x.h, w.y, fix_mad(x.l, w.x, fix_mad(y.h, c.w, fix_mad(y.l, c.z, kFixHalf))))),
                fix_join(fix_mad(x.h, w.z, fix_mad(y.h, w.x, 0)),
                         fix_mad(x.h, w.w, fix_mad(x.l, w.z, fix_mad(y.h, w.y, fix_mad(y.l, w.x, kFixHalf)))))};
    }
}

// Length-R DFT in place, R in {2, 3, 4, 5}.
template <int S, int R>
__device__ __forceinline__ void fix_dft_small(i64c (&a)[R]) {
    if constexpr (R == 2) {
        const i64c t = a[0];
        a[0] = cadd(t, a[1]);
        a[1] = csub(t, a[1]);
    } else if constexpr (R == 4) {
        const i64c t0 = cadd(a[0], a[2]), t1 = csub(a[0], a[2]), t2 = cadd(a[1], a[3]), d = csub(a[1], a[3]);
        a[0] = cadd(t0, t2);
        a[2] = csub(t0, t2);
        a[1] = {t1.x - S * d.y, t1.y + S * d.x};
        a[3] = {t1.x + S * d.y, t1.y - S * d.x};
    } else if constexpr (R == 3) {
        const i64c t1 = cadd(a[1], a[2]), t2 = csub(a[1], a[2]);
        const i64c m = {a[0].x - fix_halve(t1.x), a[0].y - fix_halve(t1.y)};
        const i64c q = {t2.x + fix_mul(t2.x, c_consq[kQsin3]), t2.y + fix_mul(t2.y, c_consq[kQsin3])};
        a[0] = cadd(a[0], t1);
        a[1] = {m.x - S * q.y, m.y + S * q.x};
        a[2] = {m.x + S * q.y, m.y - S * q.x};
    } else {
        static_assert(R == 5, "radix");
        const int2 ca = c_consq[kQcos5a], sa = c_consq[kQsin5a], cb = c_consq[kQcos5b], sb = c_consq[kQsin5b];
        const int2 na = c_consq[kQnsin5a];
        const i64c t1 = cadd(a[1], a[4]), t2 = cadd(a[2], a[3]), t3 = csub(a[1], a[4]), t4 = csub(a[2], a[3]);
        const i64c m1 = {a[0].x + fix_mul2(t1.x, ca, t2.x, cb), a[0].y + fix_mul2(t1.y, ca, t2.y, cb)};
        const i64c m2 = {a[0].x + fix_mul2(t1.x, cb, t2.x, ca), a[0].y + fix_mul2(t1.y, cb, t2.y, ca)};
        const i64c n1 = {fix_mul2(t3.x, sa, t4.x, sb), fix_mul2(t3.y, sa, t4.y, sb)};
        const i64c n2 = {fix_mul2(t3.x, sb, t4.x, na), fix_mul2(t3.y, sb, t4.y, na)};
        a[0] = cadd(a[0], cadd(t1, t2));
        a[1] = {m1.x - S * n1.y, m1.y + S * n1.x};
        a[4] = {m1.x + S * n1.y, m1.y - S * n1.x};
        a[2] = {m2.x - S * n2.y, m2.y + S * n2.x};
        a[3] = {m2.x + S * n2.y, m2.y - S * n2.x};
    }
}

// DFT / 2^fix_levels(N) in place; the decomposition of Fft in bgw_fft.cuh.
template <int S, int N, int NTOP>
struct FixFft {
    static constexpr int R = first_radix(N);
    static constexpr int M = N / R;

    template <int N1, int K1>
    __device__ __forceinline__ static void stage_twiddle(i64c (&sub)[R][M]) {
        if constexpr (N1 < R) {
            if constexpr (K1 < M) {
                sub[N1][K1] = fix_twiddle<S, N, NTOP, N1 * K1>(sub[N1][K1]);
                stage_twiddle<N1, K1 + 1>(sub);
            } else {
                stage_twiddle<N1 + 1, 0>(sub);
            }
        }
    }

    __device__ __forceinline__ static void run(i64c (&a)[N]) {
        if constexpr (M == 1) {
            fix_dft_small<S, R>(a);
        } else {
            i64c sub[R][M];
#pragma unroll
            for (int n1 = 0; n1 < R; ++n1)
#pragma unroll
                for (int n2 = 0; n2 < M; ++n2) sub[n1][n2] = a[R * n2 + n1];
#pragma unroll
            for (int n1 = 0; n1 < R; ++n1) FixFft<S, M, NTOP>::run(sub[n1]);
            stage_twiddle<0, 0>(sub);
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) {
                i64c t[R];
#pragma unroll
                for (int n1 = 0; n1 < R; ++n1) t[n1] = sub[n1][k1];
                fix_dft_small<S, R>(t);
#pragma unroll
                for (int k2 = 0; k2 < R; ++k2) a[k1 + M * k2] = t[k2];
            }
        }
    }
};

// ---------------------------------------------------------- conversions --
// A line's scale: component = integer * 2^-(top - (E - 1022)), E the biased
// exponent of its largest component (0: all zero or subnormal; 0x7ff: some
// component is not finite).
template <int N>
__device__ __forceinline__ int fix_line_exponent(const cpx<double> (&a)[N]) {
    int m = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        m = max(m, __double2hiint(a[i].x) & 0x7fffffff);
        m = max(m, __double2hiint(a[i].y) & 0x7fffffff);
    }
    return m >> 20;
}

// v scaled to the integers of a line of exponent E, rounded to nearest.
template <int TOP>
__device__ __forceinline__ long long fix_in(double v, int E) {
    const int hi = __double2hiint(v);
    const int e = (hi >> 20) & 0x7ff;
    const unsigned long long m =
        (((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v)) << (TOP - 52);
    const int d = e ? min(E - e, 63) : 63;       // zeros and subnormals vanish
    const long long r = (long long)((m >> d) + 1) >> 1;
    const long long s = (long long)(hi >> 31);
    return (r ^ s) - s;
}

// The FP64 number nearest to v 2^(eb - 1086).
__device__ __forceinline__ double fix_out(long long v, int eb) {
    const unsigned long long s = (unsigned long long)(v >> 63);
    unsigned long long u = ((unsigned long long)v ^ s) - s;
    const int lz = __clzll((long long)u);
    u <<= lz & 63;                                // leading bit at 63 (u = 0: lz = 64)
    const int e = eb - lz;
    unsigned long long b = (u >> 11) + ((u >> 10) & 1ull);
    b += (unsigned long long)(long long)(e - 1) << 52;      // the implicit bit adds one to the exponent field
    if (lz >= 64 || e < 1) b = 0;                 // zero, and results below the normal range
    if (e >= 0x7ff) b = 0x7ff0000000000000ull;
    return __longlong_as_double((long long)(b | (s & 0x8000000000000000ull)));
}

// Unnormalised forward (S = -1) or inverse (S = +1) DFT of a line of FP64
// values through 64-bit fixed point.  A line with an infinity or a NaN leaves
// as NaN throughout.
template <int S, int N>
__device__ __forceinline__ void fft_line_fix(cpx<double> (&a)[N]) {
    static_assert(fft_len_supported(N) && N <= kFixMaxN, "unsupported FFT length");
    constexpr int TOP = fix_top(N);
    const int E = fix_line_exponent<N>(a);
    i64c v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = i64c{fix_in<TOP>(a[i].x, E), fix_in<TOP>(a[i].y, E)};
    FixFft<S, N, N>::run(v);
    const int eb = 1086 - (TOP - (E - 1022)) + fix_levels(N);
#pragma unroll
    for (int i = 0; i < N; ++i) a[i] = cpx<double>{fix_out(v[i].x, eb), fix_out(v[i].y, eb)};
    if (E == 0x7ff) {
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
        for (int i = 0; i < N; ++i) a[i] = cpx<double>{nan, nan};
    }
}

// ------------------------------------------------------- integer grids --
// Real-space grids of the FP64 contexts whose y-z planes are square and at
// most 40 wide are kept as integers of one scale per (band, spin component,
// x-plane): {re hi, re lo, im hi, im lo} with u = (hi 2^32 + lo) 2^scale,
// |u| 2^-scale <= 2^fix_grid_top(N).  16 bytes a value, as in FP64; the largest
// component of a plane keeps 60 bits.  The two spin components of a plane share
// the larger's scale unless one is more than 2^kFixApart smaller (a nearly
// spin-pure state, whose small component then keeps its own 60 bits).
constexpr int kFixBad = 1 << 24;      // scale of a plane with an infinity or a NaN
constexpr int kFixApart = 4;
// The scale a component with own scale s takes beside one with scale t.
__device__ __forceinline__ int fix_shared_scale(int s, int t) { return s < t && t - s <= kFixApart ? t : s; }
// Pair densities of two such planes stay below 2^fix_top(N).
__host__ __device__ constexpr int fix_grid_top(int n) { return fix_top(n) >= 58 ? 60 : 59; }

__device__ __forceinline__ int4 fix_pack(long long x, long long y) {
    fix_parts p = fix_split(x), q = fix_split(y);
    // -2^31 has no negative: one unit aside instead
    if (p.l == (int)0x80000000) p.l = -0x7fffffff;
    if (q.l == (int)0x80000000) q.l = -0x7fffffff;
    return make_int4(p.h, p.l, q.h, q.l);
}
__device__ __forceinline__ long long fix_unpack(int h, int l) { return ((long long)h << 32) + l; }

// |hi word| bits of a value, for the OR over many: all |v| < 2^(64 - clz(OR)).
__device__ __forceinline__ int fix_mag(i64c v) {
    const int x = (int)(v.x >> 32), y = (int)(v.y >> 32);
    return (x ^ (x >> 31)) | (y ^ (y >> 31));
}
// r in 1..63
__device__ __forceinline__ long long fix_shift_right(long long v, int r) { return (v + (1LL << (r - 1))) >> r; }

}  // namespace bgw
