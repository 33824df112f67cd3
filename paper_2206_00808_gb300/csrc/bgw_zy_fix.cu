// Pair density + z and y passes of the FP64 matrix elements in 64-bit fixed
// point, for boxes with N2 = N3 <= 40 (Eq. matrix_el of arXiv:2206.00808).
//
// k2_zy_fix reads integer grids (bgw_fft_i64.cuh) and takes one x-plane and a
// tile of TV x TC pairs per CTA:
//   1. rho = sum_alpha conj(u_v) u_c at every point of the plane, a thread per
//      point with the tile's TV + TC values in registers (24 multiply-adds and
//      two joins a pair and point), into shared memory [pair][y][z];
//   2. z lines, one per thread (fft_line of bgw_fft_i64.cuh), the kept outputs
//      written over the thread's own row;
//   3. y lines over the kept outputs, back to FP64, to Bs[pair][x][w1][w2].
// Nothing is converted or rescaled between the passes unless a pair's z
// outputs are too large for the y transform (the shift r below).
//
// Bound: integer issue (a multiply-add or a 64-bit add every two cycles of a
// scheduler).  The FP64 passes it replaces (k2_zpass, k2_ypass) ran at 0.9 of
// the FP64 pipe, whose operations cost 64 to 76 such cycles.
#include <cuda_runtime.h>

#include <type_traits>

#include "bgw_fft_i64.cuh"
#include "bgw_internal.h"

namespace bgw {
namespace {

constexpr int kWinF = 8;              // kept outputs within +-kWinF of 0 let the compiler drop butterflies

// Pairs per CTA, one z line per thread: as many as shared memory and the
// registers of a line leave room for.  Measured per shape: 24^3 (1600 pairs)
// 2 x 5 pairs at 128 registers 225 us, 2 x 4 at 168 240, 1 x 5 251, 4 x 4 253,
// 2 x 2 256; 32^3 (1782 pairs) 2 x 4 one CTA per SM 626 us, 2 x 3 656, 2 x 2
// 677, 1 x 4 730.
template <int N>
struct ZyTile {
    static constexpr int TV = 2;
    static constexpr int TC = N == 24 ? 5 : N <= 27 || N == 32 ? 4 : N == 30 ? 3 : 2;
    static constexpr int RS = N | 1;                                   // odd row: conflict-free 16-byte rows
    static constexpr int THREADS = (TV * TC * N + 31) / 32 * 32;
    static constexpr int MINB = N == 16 ? 4 : N <= 20 ? 3 : N == 32 ? 1 : 2;
    static constexpr size_t SMEM = (size_t)TV * TC * N * RS * 16;
};

template <int N, bool WIN>
__global__ void __launch_bounds__(ZyTile<N>::THREADS, ZyTile<N>::MINB)
k2_zy_fix(const int4 *__restrict__ Fv, const int *__restrict__ Sv, const int4 *__restrict__ Fc,
          const int *__restrict__ Sc, int nv, int nc, int ldc, int w1, int w2, int s1, int s2,
          double2 *__restrict__ Bs) {
    constexpr int TV = ZyTile<N>::TV, TC = ZyTile<N>::TC, RS = ZyTile<N>::RS, THREADS = ZyTile<N>::THREADS;
    constexpr int NN = N * N, TOP = fix_top(N);
    extern __shared__ int4 zy_raw[];
    i64c *R = reinterpret_cast<i64c *>(zy_raw);      // [TV*TC][N][RS]
    __shared__ int pbits[TV * TC];
    __shared__ int apart[TV * TC];     // exponent of the spin-up products over the spin-down ones
    const int x = blockIdx.x, n0 = gridDim.x;
    const int v0 = blockIdx.y * TV, c0 = blockIdx.z * TC;
    const int tv = min(TV, nv - v0), tc = min(TC, nc - c0);
    const auto scale_v = [&](int v, int al) { return Sv[(2L * (v0 + v) + al) * n0 + x]; };
    const auto scale_c = [&](int c, int al) { return Sc[(2L * (c0 + c) + al) * n0 + x]; };
    int ap = 0;
    if (threadIdx.x < TV * TC) {
        const int v = min((int)threadIdx.x / TC, tv - 1), c = min((int)threadIdx.x % TC, tc - 1);
        pbits[threadIdx.x] = 0;
        ap = scale_v(v, 0) + scale_c(c, 0) - scale_v(v, 1) - scale_c(c, 1);
        apart[threadIdx.x] = ap;
    }
    const bool any_apart = __syncthreads_or(ap != 0);
    // 1. pair densities (a tile's missing bands repeat its last one)
    const int4 *pv[TV], *pc[TC];
#pragma unroll
    for (int v = 0; v < TV; ++v) pv[v] = Fv + (2L * (v0 + min(v, tv - 1)) * n0 + x) * NN;
#pragma unroll
    for (int c = 0; c < TC; ++c) pc[c] = Fc + (2L * (c0 + min(c, tc - 1)) * n0 + x) * NN;
    const long spin = (long)n0 * NN;
    // in a loop of its own where a pair's spin components have scales apart (one
    // loop for both took 13 % longer at 32^3)
    auto densities = [&](auto slow) {
    for (int t = threadIdx.x; t < NN; t += THREADS) {
        int4 c[TC][2];
#pragma unroll
        for (int i = 0; i < TC; ++i) {
            c[i][0] = __ldg(pc[i] + t);
            c[i][1] = __ldg(pc[i] + spin + t);
        }
        i64c *r = R + (t / N) * RS + t % N;
#pragma unroll
        for (int v = 0; v < TV; ++v) {
            const int4 a = __ldg(pv[v] + t), b = __ldg(pv[v] + spin + t);
            const int nah = -a.z, nal = -a.w, nbh = -b.z, nbl = -b.w;      // minus the imaginary parts
#pragma unroll
            for (int i = 0; i < TC; ++i) {
                const int4 p = c[i][0], q = c[i][1];
                // (pair by pair, so that a pair's bits do not depend on its tile)
                if (decltype(slow)::value && apart[v * TC + i] != 0) {        // the spin components have scales of their own: join each, align the smaller
                    auto part = [&](const int4 &a4, int nh, int nl, const int4 &p4) {
                        const long long rh = fix_mad(a4.x, p4.x, fix_mad(a4.z, p4.z, 0));
                        const long long rl = fix_mad(a4.x, p4.y, fix_mad(a4.y, p4.x, fix_mad(a4.z, p4.w, fix_mad(a4.w, p4.z, kFixHalf))));
                        const long long ih = fix_mad(a4.x, p4.z, fix_mad(nh, p4.x, 0));
                        const long long il = fix_mad(a4.x, p4.w, fix_mad(a4.y, p4.z, fix_mad(nh, p4.y, fix_mad(nl, p4.x, kFixHalf))));
                        return i64c{fix_join(rh, rl), fix_join(ih, il)};
                    };
                    i64c up = part(a, nah, nal, p), dn = part(b, nbh, nbl, q);
                    const int d = apart[v * TC + i], r1 = min(d < 0 ? -d : d, 63);
                    if (d < 0) up = i64c{fix_shift_right(up.x, r1), fix_shift_right(up.y, r1)};
                    else dn = i64c{fix_shift_right(dn.x, r1), fix_shift_right(dn.y, r1)};
                    r[(v * TC + i) * N * RS] = cadd(up, dn);
                    continue;
                }
                const long long reh = fix_mad(a.x, p.x, fix_mad(a.z, p.z, fix_mad(b.x, q.x, fix_mad(b.z, q.z, 0))));
                long long rel = fix_mad(a.x, p.y, fix_mad(a.y, p.x, fix_mad(a.z, p.w, fix_mad(a.w, p.z, kFixHalf))));
                rel = fix_mad(b.x, q.y, fix_mad(b.y, q.x, fix_mad(b.z, q.w, fix_mad(b.w, q.z, rel))));
                const long long imh = fix_mad(a.x, p.z, fix_mad(nah, p.x, fix_mad(b.x, q.z, fix_mad(nbh, q.x, 0))));
                long long iml = fix_mad(a.x, p.w, fix_mad(a.y, p.z, fix_mad(nah, p.y, fix_mad(nal, p.x, kFixHalf))));
                iml = fix_mad(b.x, q.w, fix_mad(b.y, q.z, fix_mad(nbh, q.y, fix_mad(nbl, q.x, iml))));
                r[(v * TC + i) * N * RS] = i64c{fix_join(reh, rel), fix_join(imh, iml)};
            }
        }
    }
    };
    if (any_apart)
        densities(std::true_type());
    else
        densities(std::false_type());
    __syncthreads();
    // 2. z lines
    const int ns1 = N - s1, ns2 = N - s2;
    {
        const int pr = threadIdx.x / N, y = threadIdx.x % N;
        if (pr < TV * TC && pr / TC < tv && pr % TC < tc) {
            i64c *row = R + (pr * N + y) * RS;
            i64c a[N];
#pragma unroll
            for (int z = 0; z < N; ++z) a[z] = row[z];
            FixFft<-1, N, N>::run(a);
            int big = 0;
            constexpr int K = WIN ? 2 * kWinF + 1 : N;
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const int f = !WIN || i <= kWinF ? i : N - K + i;
                const int j = f + ns2 >= N ? f + ns2 - N : f + ns2;
                if (j < w2) {
                    row[j] = a[f];
                    big |= fix_mag(a[f]);
                }
            }
            atomicMax(&pbits[pr], 64 - __clz(big));      // every kept |value| <= 2^bits
        }
    }
    __syncthreads();
    // 3. y lines of the kept z outputs, back to FP64
    for (int t = threadIdx.x; t < TV * TC * w2; t += THREADS) {
        const int pr = t / w2, jz = t % w2;
        const int v = pr / TC, c = pr % TC;
        if (v >= tv || c >= tc) continue;
        const i64c *col = R + pr * N * RS + jz;
        const int r = max(0, pbits[pr] - TOP);
        i64c a[N];
#pragma unroll
        for (int y = 0; y < N; ++y) a[y] = col[y * RS];
        if (r > 0) {
#pragma unroll
            for (int y = 0; y < N; ++y) a[y] = i64c{fix_shift_right(a[y].x, r), fix_shift_right(a[y].y, r)};
        }
        FixFft<-1, N, N>::run(a);
        const int v0s = scale_v(v, 0), v1s = scale_v(v, 1), c0s = scale_c(c, 0), c1s = scale_c(c, 1);
        const bool bad = v0s == kFixBad || v1s == kFixBad || c0s == kFixBad || c1s == kFixBad;
        const int eb = 1086 + max(v0s + c0s, v1s + c1s) + 64 + 2 * fix_levels(N) + r;
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        double2 *o = Bs + (((long)(v0 + v) * ldc + c0 + c) * n0 + x) * w1 * (long)w2 + jz;
        constexpr int K = WIN ? 2 * kWinF + 1 : N;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const int f = !WIN || i <= kWinF ? i : N - K + i;
            const int j = f + ns1 >= N ? f + ns1 - N : f + ns1;
            if (j < w1) {
                double2 d = make_double2(fix_out(a[f].x, eb), fix_out(a[f].y, eb));
                if (bad) d = make_double2(nan, nan);
                o[j * w2] = d;
            }
        }
    }
}

bool in_window(const Axes &a, int ax) {
    for (int j = 0; j < a.w[ax]; ++j) {
        const int f = (a.s[ax] + j) % a.n[ax];
        if (f > kWinF && f < a.n[ax] - kWinF) return false;
    }
    return true;
}

template <int N>
cudaError_t zy_fix_n(const int4 *fv, const int *sv, const int4 *fc, const int *sc, int nv, int nc, const Axes &a,
                     double2 *Bs, cudaStream_t st) {
    using Tile = ZyTile<N>;
    auto kern = k2_zy_fix<N, false>;
    if (in_window(a, 1) && in_window(a, 2)) kern = k2_zy_fix<N, (N > 2 * kWinF + 1)>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile::SMEM);
    if (e != cudaSuccess) return e;
    // tiles of bands are a launch's y and z index: pieces of at most kMaxGridYZ tiles
    const long planes = 2L * a.n[0], vol = (long)N * N, out = (long)a.n[0] * a.w[1] * a.w[2];
    const int vmax = kMaxGridYZ * Tile::TV, cmax = kMaxGridYZ * Tile::TC;
    for (int v0 = 0; v0 < nv; v0 += vmax)
        for (int c0 = 0; c0 < nc; c0 += cmax) {
            const int v = nv - v0 < vmax ? nv - v0 : vmax, c = nc - c0 < cmax ? nc - c0 : cmax;
            const dim3 grid(a.n[0], (v + Tile::TV - 1) / Tile::TV, (c + Tile::TC - 1) / Tile::TC);
            kern<<<grid, Tile::THREADS, Tile::SMEM, st>>>(fv + v0 * planes * vol, sv + v0 * planes, fc + c0 * planes * vol,
                                                          sc + c0 * planes, v, c, nc, a.w[1], a.w[2], a.s[1], a.s[2],
                                                          Bs + ((long)v0 * nc + c0) * out);
        }
    return cudaGetLastError();
}

}  // namespace

cudaError_t zy_fix_tables_init() {
    int4 tq[kTwTotal];
    int2 cq[kQcount];
    fix_tables(tq, cq);
    const cudaError_t e = cudaMemcpyToSymbol(c_twq, tq, sizeof tq);
    return e == cudaSuccess ? cudaMemcpyToSymbol(c_consq, cq, sizeof cq) : e;
}

cudaError_t mtxel_zy_fix(const void *Fv, const int *Sv, const void *Fc, const int *Sc, int nv, int nc, const Axes &a,
                         void *Bs, cudaStream_t st) {
    const int4 *fv = static_cast<const int4 *>(Fv), *fc = static_cast<const int4 *>(Fc);
    double2 *b = static_cast<double2 *>(Bs);
    switch (a.n[1]) {
        case 16: return zy_fix_n<16>(fv, Sv, fc, Sc, nv, nc, a, b, st);
        case 18: return zy_fix_n<18>(fv, Sv, fc, Sc, nv, nc, a, b, st);
        case 20: return zy_fix_n<20>(fv, Sv, fc, Sc, nv, nc, a, b, st);
        case 24: return zy_fix_n<24>(fv, Sv, fc, Sc, nv, nc, a, b, st);
        case 27: return zy_fix_n<27>(fv, Sv, fc, Sc, nv, nc, a, b, st);
        case 30: return zy_fix_n<30>(fv, Sv, fc, Sc, nv, nc, a, b, st);
        case 32: return zy_fix_n<32>(fv, Sv, fc, Sc, nv, nc, a, b, st);
        case 36: return zy_fix_n<36>(fv, Sv, fc, Sc, nv, nc, a, b, st);
        case 40: return zy_fix_n<40>(fv, Sv, fc, Sc, nv, nc, a, b, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace bgw
