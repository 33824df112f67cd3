// Sphere -> grid into integer grids (bgw_fft_i64.cuh): the y and z passes of
// wfn_to_grid for boxes with N2 = N3 <= 40 in 64-bit fixed point, and the
// conversions between integer and FP64 grids.
//
// k1_yz_fix: a CTA takes XP x-planes of one band, both spin components.  Their
// x-transformed cubes (FP64) are scaled by the planes' largest component once,
// then y lines and z lines run as integers in shared memory, one line per
// thread, and the z lines leave as integers scaled to fix_grid_top.  Bound:
// integer issue.  The single passes it replaces (k1_ypass, k1_zpass)
// converted every line to FP64 and back, and their rows, one per thread, were
// read and written 16 bytes at a time.
#include <cuda_runtime.h>

#include "bgw_fft_i64.cuh"
#include "bgw_internal.h"

namespace bgw {
namespace {

constexpr int kConvThreads = 256;

template <int N>
struct K1Tile {
    // x-planes per CTA: 2 N z lines each, one per thread, in whole warps as far as that goes
    static constexpr int XP = N == 16 ? 2 : N == 18 ? 3 : N == 20 ? 4 : N == 24 ? 2 : 1;
    static constexpr int THREADS = (2 * N * XP + 31) / 32 * 32;
    static constexpr int RS = N | 1;
    static size_t smem(int w1, int w2) {
        const size_t in = (size_t)w1 * w2 + (size_t)N * (w2 | 1), out = (size_t)N * RS;
        return 16 * (size_t)XP * 2 * (in > out ? in : out);
    }
};

template <int N>
__device__ __forceinline__ void k1_yz_fix_body(const double2 *__restrict__ S, int n0, int w1, int w2, int s1, int s2,
                                               int4 *__restrict__ U, int *__restrict__ scale, long b) {
    constexpr int XP = K1Tile<N>::XP, THREADS = K1Tile<N>::THREADS, RS = K1Tile<N>::RS;
    constexpr int NN = N * N, TOP = fix_top(N), GTOP = fix_grid_top(N);
    extern __shared__ int4 yz_raw[];
    __shared__ int smax[2 * XP], ybits[2 * XP], zbits[2 * XP];      // per (spin component, plane)
    const int x0 = blockIdx.x * XP, xp = min(XP, n0 - x0);
    const int cells = w1 * w2, w2p = w2 | 1;
    // A: [2][XP][w1][w2] inputs, Y: [2][XP][N][w2p] y outputs; C: [2][XP][N][RS]
    // z outputs, over both
    i64c *A = reinterpret_cast<i64c *>(yz_raw), *Y = A + 2 * XP * cells;
    int4 *Cc = yz_raw;
    if (threadIdx.x < 2 * XP) smax[threadIdx.x] = ybits[threadIdx.x] = zbits[threadIdx.x] = 0;
    __syncthreads();
    double2 *Ad = reinterpret_cast<double2 *>(yz_raw);
    for (int al = 0; al < 2; ++al)
        for (int xl = 0; xl < xp; ++xl) {
            const double2 *si = S + ((2 * b + al) * n0 + x0 + xl) * (long)cells;
            double2 *a = Ad + (al * XP + xl) * cells;
            int m = 0;
            for (int i = threadIdx.x; i < cells; i += THREADS) {
                const double2 v = si[i];
                a[i] = v;
                m = max(m, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
            }
            m = __reduce_max_sync(0xffffffffu, m);
            if ((threadIdx.x & 31) == 0) atomicMax(&smax[al * XP + xl], m);
        }
    __syncthreads();
    for (int al = 0; al < 2; ++al)
        for (int xl = 0; xl < xp; ++xl) {
            const int E = smax[al * XP + xl] >> 20;
            double2 *a = Ad + (al * XP + xl) * cells;
            for (int i = threadIdx.x; i < cells; i += THREADS) {       // each thread its own values
                const double2 v = a[i];
                reinterpret_cast<i64c *>(a)[i] = i64c{fix_in<TOP>(v.x, E), fix_in<TOP>(v.y, E)};
            }
        }
    __syncthreads();
    const int ns1 = N - s1, ns2 = N - s2;
    for (int l = threadIdx.x; l < 2 * XP * w2; l += THREADS) {
        const int q = l / w2, z = l % w2, xl = q % XP;
        if (xl >= xp) continue;
        const i64c *in = A + q * cells + z;
        i64c a[N];
#pragma unroll
        for (int f = 0; f < N; ++f) {
            const int j = f + ns1 >= N ? f + ns1 - N : f + ns1;
            a[f] = j < w1 ? in[j * w2] : i64c{0, 0};
        }
        FixFft<+1, N, N>::run(a);
        i64c *o = Y + q * N * w2p + z;
        int big = 0;
#pragma unroll
        for (int y = 0; y < N; ++y) {
            o[y * w2p] = a[y];
            big |= fix_mag(a[y]);
        }
        atomicMax(&ybits[q], 64 - __clz(big));
    }
    __syncthreads();
    const int q = threadIdx.x / N, y = threadIdx.x % N, xl = q % XP;
    const bool line = q < 2 * XP && xl < xp;
    const int r = line ? max(0, ybits[q] - TOP) : 0;
    i64c a[N];
    if (line) {
        const i64c *row = Y + (q * N + y) * w2p;
#pragma unroll
        for (int f = 0; f < N; ++f) {
            const int j = f + ns2 >= N ? f + ns2 - N : f + ns2;
            a[f] = j < w2 ? row[j] : i64c{0, 0};
        }
        if (r > 0) {
#pragma unroll
            for (int f = 0; f < N; ++f) a[f] = i64c{fix_shift_right(a[f].x, r), fix_shift_right(a[f].y, r)};
        }
        FixFft<+1, N, N>::run(a);
        int big = 0;
#pragma unroll
        for (int z = 0; z < N; ++z) big |= fix_mag(a[z]);
        atomicMax(&zbits[q], 64 - __clz(big));
    }
    __syncthreads();                       // Y has been read: the outputs go over it
    if (line) {
        // the exponent of this plane's integers, the scale that brings its largest
        // value to GTOP bits, and the same for the other spin component
        auto raw = [&](int i) { return (smax[i] >> 20) - 1022 - TOP + 2 * fix_levels(N) + max(0, ybits[i] - TOP); };
        const int other = q < XP ? q + XP : q - XP;
        const int s = fix_shared_scale(raw(q) + zbits[q] - GTOP, raw(other) + zbits[other] - GTOP);
        const int sh = max(raw(q) - s, -63);
        int4 *o = Cc + (q * N + y) * RS;
        if (sh >= 0) {
#pragma unroll
            for (int z = 0; z < N; ++z) o[z] = fix_pack(a[z].x << sh, a[z].y << sh);
        } else {
#pragma unroll
            for (int z = 0; z < N; ++z) o[z] = fix_pack(fix_shift_right(a[z].x, -sh), fix_shift_right(a[z].y, -sh));
        }
        if (y == 0) scale[(2 * b + q / XP) * n0 + x0 + xl] = smax[q] >> 20 == 0x7ff ? kFixBad : s;
    }
    __syncthreads();
    for (int al = 0; al < 2; ++al) {
        int4 *u = U + ((2 * b + al) * n0 + x0) * (long)NN;
        const int4 *c = Cc + al * XP * N * RS;
        for (int i = threadIdx.x; i < xp * NN; i += THREADS) u[i] = c[(i / N) * RS + i % N];
    }
}

template <int N>
__global__ void __launch_bounds__(K1Tile<N>::THREADS)
k1_yz_fix(const double2 *__restrict__ S, int n0, int w1, int w2, int s1, int s2, int4 *__restrict__ U,
          int *__restrict__ scale) {
    k1_yz_fix_body<N>(S, n0, w1, w2, s1, s2, U, scale, blockIdx.y);
}

// The same for several k-points, blockIdx.z, from band b0 on.
struct YzBatch {
    int n0, b0;
    struct {
        const double2 *S;
        int4 *U;
        int *scale;
        int w1, w2, s1, s2;
    } job[kK1BatchMax];
};
template <int N>
__global__ void __launch_bounds__(K1Tile<N>::THREADS)
k1_yz_fix_batch(const __grid_constant__ YzBatch jb) {
    const auto &j = jb.job[blockIdx.z];
    k1_yz_fix_body<N>(j.S, jb.n0, j.w1, j.w2, j.s1, j.s2, j.U, j.scale, (long)jb.b0 + blockIdx.y);
}

// FP64 grid -> integer grid in place, one CTA per (x-plane, band).
template <int N>
__global__ void __launch_bounds__(kConvThreads)
k_fix_planes(void *__restrict__ U, int *__restrict__ scale) {
    constexpr int NN = N * N, IT = (2 * NN + kConvThreads - 1) / kConvThreads, TOP = fix_grid_top(N);
    const int x = blockIdx.x, n0 = gridDim.x;
    const long b = blockIdx.y;
    __shared__ int smax[2];
    if (threadIdx.x < 2) smax[threadIdx.x] = 0;
    double2 v[IT];
    int m[2] = {0, 0};
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int t = i * kConvThreads + threadIdx.x;
        v[i] = make_double2(0.0, 0.0);
        if (t < 2 * NN) v[i] = static_cast<double2 *>(U)[((2 * b + t / NN) * n0 + x) * NN + t % NN];
        const int mi = max(__double2hiint(v[i].x) & 0x7fffffff, __double2hiint(v[i].y) & 0x7fffffff);
        m[0] = max(m[0], t < NN ? mi : 0);
        m[1] = max(m[1], t < NN ? 0 : mi);
    }
    __syncthreads();
#pragma unroll
    for (int al = 0; al < 2; ++al) {
        m[al] = __reduce_max_sync(0xffffffffu, m[al]);
        if ((threadIdx.x & 31) == 0) atomicMax(&smax[al], m[al]);
    }
    __syncthreads();
    const int E0 = smax[0] >> 20, E1 = smax[1] >> 20;
    const int e0 = fix_shared_scale(E0, E1), e1 = fix_shared_scale(E1, E0);
    if (threadIdx.x < 2) {
        const int E = threadIdx.x ? E1 : E0, e = threadIdx.x ? e1 : e0;
        scale[(2 * b + threadIdx.x) * n0 + x] = E == 0x7ff ? kFixBad : e - 1022 - TOP;
    }
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int t = i * kConvThreads + threadIdx.x;
        if (t < 2 * NN)
            static_cast<int4 *>(U)[((2 * b + t / NN) * n0 + x) * NN + t % NN] =
                fix_pack(fix_in<TOP>(v[i].x, t < NN ? e0 : e1), fix_in<TOP>(v[i].y, t < NN ? e0 : e1));
    }
}

// Integer grid -> FP64 grid (for the eight-lane kernels on request).
__global__ void __launch_bounds__(kConvThreads)
k_unfix_planes(const int4 *__restrict__ F, const int *__restrict__ scale, int n0, int NN, double2 *__restrict__ U) {
    const int x = blockIdx.x;
    const long b = blockIdx.y;
    const int s0 = scale[2 * b * n0 + x], s1 = scale[(2 * b + 1) * n0 + x];
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    for (int t = threadIdx.x; t < 2 * NN; t += kConvThreads) {
        const long at = ((2 * b + t / NN) * n0 + x) * NN + t % NN;
        const int s = t < NN ? s0 : s1;
        const int4 f = F[at];
        double2 v = make_double2(fix_out(fix_unpack(f.x, f.y), 1086 + s), fix_out(fix_unpack(f.z, f.w), 1086 + s));
        if (s == kFixBad) v = make_double2(nan, nan);
        U[at] = v;
    }
}

// launch(first band, bands) over pieces of at most kMaxGridYZ bands (the band is
// a launch's y index).
template <class F>
cudaError_t by_bands(int nb, F launch) {
    for (int b0 = 0; b0 < nb; b0 += kMaxGridYZ) launch(b0, nb - b0 < kMaxGridYZ ? nb - b0 : kMaxGridYZ);
    return cudaGetLastError();
}

template <int N>
cudaError_t yz_fix(const double2 *S, int nb, const Axes &a, int4 *U, int *scale, cudaStream_t st) {
    using Tile = K1Tile<N>;
    const size_t smem = Tile::smem(a.w[1], a.w[2]);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k1_yz_fix<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return by_bands(nb, [&](int b0, int n) {
        const long planes = 2L * b0 * a.n[0];
        k1_yz_fix<N><<<dim3((a.n[0] + Tile::XP - 1) / Tile::XP, n), Tile::THREADS, smem, st>>>(
            S + planes * a.w[1] * a.w[2], a.n[0], a.w[1], a.w[2], a.s[1], a.s[2], U + planes * N * N, scale + planes);
    });
}
template <int N>
cudaError_t yz_fix_batch(const K1Job *jobs, int n, int nb, cudaStream_t st) {
    using Tile = K1Tile<N>;
    YzBatch jb;
    jb.n0 = jobs[0].a.n[0];
    size_t smem = 0;
    for (int i = 0; i < n; ++i) {
        const Axes &a = jobs[i].a;
        jb.job[i] = {static_cast<const double2 *>(jobs[i].S), static_cast<int4 *>(jobs[i].U), jobs[i].scale,
                     a.w[1], a.w[2], a.s[1], a.s[2]};
        const size_t s = Tile::smem(a.w[1], a.w[2]);
        smem = s > smem ? s : smem;
    }
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k1_yz_fix_batch<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)smem);
        if (e != cudaSuccess) return e;
    }
    return by_bands(nb, [&](int b0, int m) {
        jb.b0 = b0;
        k1_yz_fix_batch<N><<<dim3((jb.n0 + Tile::XP - 1) / Tile::XP, m, n), Tile::THREADS, smem, st>>>(jb);
    });
}
template <int N>
cudaError_t fix_planes(void *U, int nb, const Axes &a, int *scale, cudaStream_t st) {
    return by_bands(nb, [&](int b0, int n) {
        const long planes = 2L * b0 * a.n[0];
        k_fix_planes<N><<<dim3(a.n[0], n), kConvThreads, 0, st>>>(static_cast<int4 *>(U) + planes * N * N, scale + planes);
    });
}

#define BGW_FOR_FIX_LEN(n, CALL)          \
    switch (n) {                          \
        case 16: return CALL(16);         \
        case 18: return CALL(18);         \
        case 20: return CALL(20);         \
        case 24: return CALL(24);         \
        case 27: return CALL(27);         \
        case 30: return CALL(30);         \
        case 32: return CALL(32);         \
        case 36: return CALL(36);         \
        case 40: return CALL(40);         \
        default: return cudaErrorInvalidValue; \
    }

}  // namespace

cudaError_t grid_fix_tables_init() {
    int4 tq[kTwTotal];
    int2 cq[kQcount];
    fix_tables(tq, cq);
    const cudaError_t e = cudaMemcpyToSymbol(c_twq, tq, sizeof tq);
    return e == cudaSuccess ? cudaMemcpyToSymbol(c_consq, cq, sizeof cq) : e;
}

cudaError_t wfn_to_fix(const double *coeff, int ngw, int nb, const int *cube_map, const Axes &a, void *S, void *U,
                       int *scale, cudaStream_t st) {
    const cudaError_t e = wfn_xpass_f64(coeff, ngw, 2 * nb, cube_map, a, S, st);
    if (e != cudaSuccess) return e;
    const double2 *s = static_cast<const double2 *>(S);
    int4 *u = static_cast<int4 *>(U);
#define BGW_CALL(N) yz_fix<N>(s, nb, a, u, scale, st)
    BGW_FOR_FIX_LEN(a.n[1], BGW_CALL)
#undef BGW_CALL
}

cudaError_t wfn_to_fix_batch(const K1Job *jobs, int n, int nb, cudaStream_t st) {
    const cudaError_t e = wfn_xpass_batch_f64(jobs, n, 2 * nb, st);
    if (e != cudaSuccess) return e;
#define BGW_CALL(N) yz_fix_batch<N>(jobs, n, nb, st)
    BGW_FOR_FIX_LEN(jobs[0].a.n[1], BGW_CALL)
#undef BGW_CALL
}

cudaError_t grid_to_fix(void *U, int nb, const Axes &a, int *scale, cudaStream_t st) {
#define BGW_CALL(N) fix_planes<N>(U, nb, a, scale, st)
    BGW_FOR_FIX_LEN(a.n[1], BGW_CALL)
#undef BGW_CALL
}

cudaError_t fix_to_grid(const void *F, const int *scale, int nb, const Axes &a, void *U, cudaStream_t st) {
    const int NN = a.n[1] * a.n[2];
    return by_bands(nb, [&](int b0, int n) {
        const long planes = 2L * b0 * a.n[0];
        k_unfix_planes<<<dim3(a.n[0], n), kConvThreads, 0, st>>>(static_cast<const int4 *>(F) + planes * NN, scale + planes,
                                                                 a.n[0], NN, static_cast<double2 *>(U) + planes * NN);
    });
}

}  // namespace bgw
