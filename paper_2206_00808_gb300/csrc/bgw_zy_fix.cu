// Pair density + z and y passes of the FP64 matrix elements in 64-bit fixed
// point, for boxes with N2 = N3 <= 40 (Eq. matrix_el of arXiv:2206.00808).
//
// k2_fix_planes writes every band's x-planes as integers of one scale per
// (band, x-plane), split for the multiplier: {re hi, re lo, im hi, im lo}.
// k2_zy_fix then takes one x-plane and a tile of TV x TC pairs per CTA:
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

#include "bgw_fft_i64.cuh"
#include "bgw_internal.h"

namespace bgw {
namespace {

constexpr int kFixBad = 1 << 24;      // scale of a plane with an infinity or a NaN
constexpr int kConvThreads = 256;
constexpr int kWinF = 8;              // kept outputs within +-kWinF of 0 let the compiler drop butterflies

// |u| of a plane below 2^kTopU: rho stays below fix_top(N).
__host__ __device__ constexpr int zy_top_u(int n) { return fix_top(n) >= 58 ? 60 : 59; }

// One CTA per (x-plane, band): both spin components.
template <int N>
__global__ void __launch_bounds__(kConvThreads)
k2_fix_planes(const double2 *__restrict__ U, int4 *__restrict__ F, int *__restrict__ scale) {
    constexpr int NN = N * N, IT = (2 * NN + kConvThreads - 1) / kConvThreads;
    const int x = blockIdx.x, n0 = gridDim.x;
    const long b = blockIdx.y;
    __shared__ int smax;
    if (threadIdx.x == 0) smax = 0;
    double2 v[IT];
    int m = 0;
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int t = i * kConvThreads + threadIdx.x;
        v[i] = make_double2(0.0, 0.0);
        if (t < 2 * NN) v[i] = U[((2 * b + t / NN) * n0 + x) * NN + t % NN];
        m = max(m, max(__double2hiint(v[i].x) & 0x7fffffff, __double2hiint(v[i].y) & 0x7fffffff));
    }
    __syncthreads();
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(&smax, m);
    __syncthreads();
    const int E = smax >> 20;
    constexpr int TOP = zy_top_u(N);
    if (threadIdx.x == 0) scale[b * n0 + x] = E == 0x7ff ? kFixBad : E - 1022 - TOP;
    int4 *o = F + (b * n0 + x) * 2L * NN;
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int t = i * kConvThreads + threadIdx.x;
        if (t < 2 * NN) {
            fix_parts p = fix_split(fix_in<TOP>(v[i].x, E)), q = fix_split(fix_in<TOP>(v[i].y, E));
            // -2^31 has no negative: one unit of 2^-60 aside instead
            if (p.l == (int)0x80000000) p.l = -0x7fffffff;
            if (q.l == (int)0x80000000) q.l = -0x7fffffff;
            o[t] = make_int4(p.h, p.l, q.h, q.l);
        }
    }
}

template <int N>
struct ZyTile {
    static constexpr int TV = 2;
    static constexpr int TC = N <= 27 ? 4 : N <= 32 ? 3 : 2;
    static constexpr int RS = N | 1;                                   // odd row: conflict-free 16-byte rows
    static constexpr int THREADS = (TV * TC * N + 31) / 32 * 32;       // one z line per thread
    static constexpr int MINB = N == 16 ? 4 : N <= 20 ? 3 : 2;
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
    const int x = blockIdx.x, n0 = gridDim.x;
    const int v0 = blockIdx.y * TV, c0 = blockIdx.z * TC;
    const int tv = min(TV, nv - v0), tc = min(TC, nc - c0);
    if (threadIdx.x < TV * TC) pbits[threadIdx.x] = 0;
    // 1. pair densities (a tile's missing bands repeat its last one)
    const int4 *pv[TV], *pc[TC];
#pragma unroll
    for (int v = 0; v < TV; ++v) pv[v] = Fv + ((long)(v0 + min(v, tv - 1)) * n0 + x) * 2 * NN;
#pragma unroll
    for (int c = 0; c < TC; ++c) pc[c] = Fc + ((long)(c0 + min(c, tc - 1)) * n0 + x) * 2 * NN;
    for (int t = threadIdx.x; t < NN; t += THREADS) {
        int4 c[TC][2];
#pragma unroll
        for (int i = 0; i < TC; ++i) {
            c[i][0] = __ldg(pc[i] + t);
            c[i][1] = __ldg(pc[i] + NN + t);
        }
        i64c *r = R + (t / N) * RS + t % N;
#pragma unroll
        for (int v = 0; v < TV; ++v) {
            const int4 a = __ldg(pv[v] + t), b = __ldg(pv[v] + NN + t);
            const int nah = -a.z, nal = -a.w, nbh = -b.z, nbl = -b.w;      // minus the imaginary parts
#pragma unroll
            for (int i = 0; i < TC; ++i) {
                const int4 p = c[i][0], q = c[i][1];
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
                    const int hx = (int)(a[f].x >> 32), hy = (int)(a[f].y >> 32);
                    big |= (hx ^ (hx >> 31)) | (hy ^ (hy >> 31));
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
            const long long half = 1LL << (r - 1);
#pragma unroll
            for (int y = 0; y < N; ++y) a[y] = i64c{(a[y].x + half) >> r, (a[y].y + half) >> r};
        }
        FixFft<-1, N, N>::run(a);
        const int ev = Sv[(long)(v0 + v) * n0 + x], ec = Sc[(long)(c0 + c) * n0 + x];
        const bool bad = ev == kFixBad || ec == kFixBad;
        const int eb = 1086 + ev + ec + 64 + 2 * fix_levels(N) + r;
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
cudaError_t zy_fix_n(const double2 *uv, const double2 *uc, int nv, int nc, const Axes &a, void *ws, double2 *Bs,
                     cudaStream_t st) {
    using Tile = ZyTile<N>;
    const int n0 = a.n[0];
    const long plane_vals = (long)n0 * 2 * N * N;
    int vcap, ccap;
    fix_band_caps(a, nv, nc, &vcap, &ccap);
    int4 *Fv = static_cast<int4 *>(ws), *Fc = Fv + (long)vcap * plane_vals;
    int *Sv = reinterpret_cast<int *>(Fc + (long)ccap * plane_vals), *Sc = Sv + (long)vcap * n0;
    auto kern = k2_zy_fix<N, false>;
    if (in_window(a, 1) && in_window(a, 2)) kern = k2_zy_fix<N, (N > 2 * kWinF + 1)>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile::SMEM);
    if (e != cudaSuccess) return e;
    for (int v = 0; v < nv; v += vcap) {
        const int kv = nv - v < vcap ? nv - v : vcap;
        k2_fix_planes<N><<<dim3(n0, kv), kConvThreads, 0, st>>>(uv + v * plane_vals, Fv, Sv);
        for (int c = 0; c < nc; c += ccap) {
            const int kc = nc - c < ccap ? nc - c : ccap;
            k2_fix_planes<N><<<dim3(n0, kc), kConvThreads, 0, st>>>(uc + c * plane_vals, Fc, Sc);
            const dim3 grid(n0, (kv + Tile::TV - 1) / Tile::TV, (kc + Tile::TC - 1) / Tile::TC);
            kern<<<grid, Tile::THREADS, Tile::SMEM, st>>>(
                Fv, Sv, Fc, Sc, kv, kc, nc, a.w[1], a.w[2], a.s[1], a.s[2],
                Bs + ((long)v * nc + c) * n0 * a.w[1] * (long)a.w[2]);
        }
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

cudaError_t mtxel_zy_fix(const void *Uv, const void *Uc, int nv, int nc, const Axes &a, void *ws, void *Bs,
                         cudaStream_t st) {
    const double2 *uv = static_cast<const double2 *>(Uv), *uc = static_cast<const double2 *>(Uc);
    double2 *b = static_cast<double2 *>(Bs);
    switch (a.n[1]) {
        case 16: return zy_fix_n<16>(uv, uc, nv, nc, a, ws, b, st);
        case 18: return zy_fix_n<18>(uv, uc, nv, nc, a, ws, b, st);
        case 20: return zy_fix_n<20>(uv, uc, nv, nc, a, ws, b, st);
        case 24: return zy_fix_n<24>(uv, uc, nv, nc, a, ws, b, st);
        case 27: return zy_fix_n<27>(uv, uc, nv, nc, a, ws, b, st);
        case 30: return zy_fix_n<30>(uv, uc, nv, nc, a, ws, b, st);
        case 32: return zy_fix_n<32>(uv, uc, nv, nc, a, ws, b, st);
        case 36: return zy_fix_n<36>(uv, uc, nv, nc, a, ws, b, st);
        case 40: return zy_fix_n<40>(uv, uc, nv, nc, a, ws, b, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace bgw
