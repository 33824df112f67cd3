// FFT lines of FP64 data in 64-bit block fixed point.
//
// GB300 issues two FP64 operations per clock per SM, against 64 32 x 32 -> 64
// bit multiply-adds and 64 32-bit adds with carry (measured: 64 issue cycles
// per warp for a DFMA, 2.05 for a mad.wide, 4.6 for a 64-bit add).  A
// transform is nothing but sums of its inputs times roots of unity, so every
// value of it is bounded by N sqrt(2) times the largest input component: one
// power of two per line is enough, and 64-bit integers carry more bits of it
// than FP64 does.
//
// A line enters as FP64, is scaled by 2^s so that its largest component lies
// in [2^(T-1), 2^T), T = 62 - ceil(log2(N sqrt 2)) (55..57: two to four bits
// more than FP64's 53), is transformed with integer adds and
//   x w = 4 xh wh + ((xh wl + xl wh) >> 30),   w in units of 2^-62, x = xh 2^32 + xl,
// with xl and wl signed (so the dropped xl wl, below one unit, has no bias),
// and leaves as FP64, rounded to nearest.  The rounding of a line is thus about
// 2^-56 of its largest component; FP64 butterflies round at 2^-53 of the
// running values.  A line with an infinity or a NaN leaves as NaN throughout.
#pragma once
#include "bgw_fft.cuh"

namespace bgw {

using i64c = cpx<long long>;

// Longest line held by one thread: 4 registers a point.
constexpr int kFixMaxN = 40;

// Bits of the growth bound N sqrt(2) (components of a sum of N terms).
__host__ __device__ constexpr int fix_growth_bits(int n) {
    int b = 0;
    while ((1L << (2 * b)) < 2L * n * n) ++b;
    return b;
}
// Largest input component is below 2^fix_top(n).
__host__ __device__ constexpr int fix_top(int n) { return 62 - fix_growth_bits(n); }

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

// The FP64 number nearest to v 2^(eb - 1086), eb = 1086 - (scale exponent).
__device__ __forceinline__ double fix_out(long long v, int eb) {
    const unsigned long long s = (unsigned long long)(v >> 63);
    unsigned long long u = ((unsigned long long)v ^ s) - s;
    const int lz = __clzll((long long)u);
    u <<= lz;                                     // leading bit at 63 (u = 0: lz = 64)
    const int e = eb - lz;
    unsigned long long b = (u >> 11) + ((u >> 10) & 1ull);
    b += (unsigned long long)(long long)(e - 1) << 52;      // the implicit bit adds one to the exponent field
    if (lz >= 64 || e < 1) b = 0;                 // zero, and results below the normal range
    if (e >= 0x7ff) b = 0x7ff0000000000000ull;
    return __longlong_as_double((long long)(b | (s & 0x8000000000000000ull)));
}

// Unnormalised forward (S = -1) or inverse (S = +1) DFT of a line of FP64
// values through 64-bit fixed point.  PRUNED inputs (known zeros) cost
// nothing but their butterflies.
template <int S, int N>
__device__ __forceinline__ void fft_line_fix(cpx<double> (&a)[N]) {
    constexpr int TOP = fix_top(N);
    const int E = fix_line_exponent<N>(a);
    i64c v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = i64c{fix_in<TOP>(a[i].x, E), fix_in<TOP>(a[i].y, E)};
    fft_line<long long, S, N>(v);
    const int eb = 1086 - (TOP - (E - 1022));
#pragma unroll
    for (int i = 0; i < N; ++i) a[i] = cpx<double>{fix_out(v[i].x, eb), fix_out(v[i].y, eb)};
    if (E == 0x7ff) {
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
        for (int i = 0; i < N; ++i) a[i] = cpx<double>{nan, nan};
    }
}

}  // namespace bgw
