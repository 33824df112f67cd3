// FP64-accurate complex products on tcgen05 tensor cores (sm_103a).
//
// The FP64 pipe does 2 operations per clock per SM, the tensor cores 8192
// BF16 multiply-adds: a product of FP64 accuracy costs less as the 36 products
// of BF16 digits below.  A real row gets a power-of-two scale from its largest
// component; N = x 2^s (|N| <= 2^62) is cut into eight signed base-256 digits,
//   x = 2^e sum_t S_t,  S_t = d_t 2^(-8t), d_t in [-128, 128] (exact in BF16),
// and the products S_t S_u with t + u <= 7 are kept.  What is dropped is 2^-62
// of the scales: an FP64 sum rounds at 2^-53 of its terms, so rows whose
// largest entries meet small ones (W near G = 0, orthogonal states there) keep
// nine bits in hand.  (Seven digits and 28 products had the error of FP64 sums
// or up to a third more on such rows.)
// Where one operand's entries rise along k as the other's fall (v(G) in W against
// matrix elements that vanish with G -> 0), scales per row cut off what the other
// makes up for: dz_balance finds each column's largest entry relative to its rows
// and the split moves half the difference of the two operands, a power of two per
// k, from one to the other.
// Products of one order t + u are integers in units of 2^(-8(t+u)); over 160 k
// the sums of orders 0 to 5 (1 to 6 products of at most 2^14) stay below 2^24
// units, so an FP32 accumulator in TMEM holds them exactly; they are moved to
// 64-bit integers every 160 k.  Orders 6 and 7 share a seventh accumulator,
// whose rounding is 2^-58 of the scales.  The sums leave as FP64, rounded once.
//
// Complex products as one real one: row m of A is (re, im) along k' = 2k, 2k+1;
// row n of B is two real rows, (re, -im) and (im, re), whose products with row m
// are the real and the imaginary part.
//
// dz_split  scales and digits, tiles [rows/128][k'/32][128][32] of each digit
// dz_gemm   persistent, one CTA per SM over (matrix, 128 x 64 tile): warp 16
//           TMA (96 KB a 32-k' block: 8 digits of 128 + 64 rows, two stages),
//           warp 17 MMA (72 of M128 N64 K16 a block), warps 0-15 promote and
//           write.  Bound: shared-memory reads of the MMAs (a 128 x 64 x 16 MMA
//           reads 6 KB, 48 clocks, against 32 of the tensor core).
// Every mbarrier wait is bounded, as in bgw_chi0_f64tc.cu; a block whose wait gave
// up writes NaN for the rest of its tiles, so that what is built on them shows it.
#include "bgw_dz.h"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <cstring>

#include "bgw_fft_i64.cuh"
#include "bgw_tc_common.cuh"

namespace bgw {
namespace {

using namespace tc;

constexpr int kM = 128, kN = 64, kKB = 32, kSl = 8, kStg = 2;
constexpr int kTileA = kM * kKB * 2, kTileB = kN * kKB * 2;
constexpr int kStage = kSl * (kTileA + kTileB);
constexpr int kSub = 5;                       // k' blocks per promotion
constexpr int kAcc = 7;
constexpr int kCols = 512;                    // seven accumulators of 64 columns, allocated as a power of two
constexpr int kEpi = 16;                      // epilogue warps
constexpr int kThreads = (kEpi + 2) * 32;
constexpr int kTopD = 62;                     // |N| <= 2^kTopD
constexpr int kErrFull = 1, kErrEmpty = 2, kErrAccum = 3, kErrDrain = 4;

// ---------------------------------------------------------------- digits --
constexpr int kSpRows = 32, kSpThreads = 256;
constexpr int kMaxOps = 4;

struct SplitOp {
    DzOperand op;
    __nv_bfloat16 *x;
    int *scale;
    int rows, rows_pad, b;
    int batch0;        // first matrix of the planes written
    long tiles;        // 128-row tiles of the planes
    unsigned first;    // first block of this operand
};
struct SplitArgs {
    SplitOp o[kMaxOps];
    int n, K, kblocks;
};

// Element (row, k) of an operand, weight and conjugation applied.
__device__ __forceinline__ double2 dz_load(const DzOperand &op, const double2 *base, long row, int k) {
    double2 v = __ldg(base + row * op.sr + k * op.sk);
    if (op.w) {
        const double w = op.w[k];
        v.x *= w;
        v.y *= w;
    }
    if (op.conj) v.y = -v.y;
    return v;
}

// Four k' values (two complex) of one real row: a 8-byte store per digit.
__device__ __forceinline__ void dz_store(__nv_bfloat16 *x, long plane, const long long (&n)[4]) {
    unsigned long long u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = (unsigned long long)n[i] + 0x0080808080808080ull;   // bytes 0-6 offset by 128
    float s = 1.0f;
#pragma unroll
    for (int t = 0; t < kSl; ++t) {
        __nv_bfloat162 lo, hi;
        float d[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            d[i] = (t == 0 ? (float)((int)(u[i] >> 32) >> 24) : (float)((int)((u[i] >> (56 - 8 * t)) & 0xff) - 128)) * s;
        lo = __floats2bfloat162_rn(d[0], d[1]);
        hi = __floats2bfloat162_rn(d[2], d[3]);
        *reinterpret_cast<uint2 *>(x + t * plane) =
            make_uint2(*reinterpret_cast<unsigned *>(&lo), *reinterpret_cast<unsigned *>(&hi));
        s *= 0x1p-8f;
    }
}

// Exponent of a value's larger component for the comparisons below.
constexpr int kExpZero = -4096, kExpBad = 1 << 20;      // zero or subnormal; not finite
__device__ __forceinline__ int dz_exponent(double2 v) {
    const int e = max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff) >> 20;
    return e == 0 ? kExpZero : e == 0x7ff ? kExpBad : e;
}
// Power of two that column k of this operand is multiplied by.
__device__ __forceinline__ int dz_shift(const DzOperand &op, int k) {
    if (!op.cols) return 0;
    const int c = op.cols[k], o = op.other[k];
    if (c <= kExpZero || o <= kExpZero) return 0;
    return op.second ? -((c - o) >> 1) : (o - c) >> 1;
}

// Column exponents of both operands of a product, each entry's taken relative to
// its row's largest: a block has kBalRows rows, a warp each, and keeps their
// entries' exponents in shared memory [row][K] for the columns.  Bound: one
// latency of the operands' read and the launch.
constexpr int kBalRows = 8;
struct BalanceArgs {
    DzOperand op[2];
    long rows[2];
    int *col[2];
    int *err;
    int K;
};
__global__ void __launch_bounds__(32 * kBalRows) k_dz_balance(const __grid_constant__ BalanceArgs a) {
    extern __shared__ short ex[];
    __shared__ int er[kBalRows];
    const long groups0 = (a.rows[0] + kBalRows - 1) / kBalRows;
    const int w = blockIdx.x >= groups0, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.err = 0;
    const DzOperand op = a.op[w];
    const long row = (w ? blockIdx.x - groups0 : blockIdx.x) * kBalRows + warp;
    const bool there = row < a.rows[w];
    const double2 *base = op.p + (there ? row : 0) * op.sr;
    int m = kExpZero;
#pragma unroll 4
    for (int k = lane; k < a.K; k += 32) {
        const int e = there ? dz_exponent(dz_load(op, base, 0, k)) : kExpZero;
        m = max(m, e);
        ex[warp * a.K + k] = (short)min(e, 0x7fff);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) er[warp] = m;
    __syncthreads();
    for (int k = threadIdx.x; k < a.K; k += 32 * kBalRows) {
        int c = kExpZero;
#pragma unroll
        for (int i = 0; i < kBalRows; ++i) {
            const int e = ex[i * a.K + k];
            if (er[i] != kExpBad && e != kExpZero) c = max(c, e - er[i]);      // a row that is not finite has no say
        }
        if (c > *(volatile int *)&a.col[w][k]) atomicMax(&a.col[w][k], c);
    }
}

// 32 rows of one operand per block, a part of their k' blocks each along y (every
// block finds its rows' largest entries itself).
__global__ void __launch_bounds__(kSpThreads) k_dz_split(const __grid_constant__ SplitArgs a) {
    __shared__ double2 sm[kSpRows][kKB / 2 + 1];
    __shared__ int smax[kSpRows];
    extern __shared__ int shift[];                    // of every k
    int w = 0;
    while (w + 1 < a.n && blockIdx.x >= a.o[w + 1].first) ++w;
    const SplitOp &o = a.o[w];
    const int blocks = o.rows_pad / (o.b ? 2 * kSpRows : kSpRows);     // blocks per matrix
    const unsigned bl = blockIdx.x - o.first;
    const int b = bl / blocks, r0 = (bl % blocks) * kSpRows;
    const double2 *base = o.op.p + b * o.op.sb;
    const bool along_rows = o.op.sr == 1;             // consecutive lanes take consecutive rows
    const int t = threadIdx.x;
    if (t < kSpRows) smax[t] = kExpZero;
    for (int k = t; k < a.K; k += kSpThreads) shift[k] = dz_shift(o.op, k);
    __syncthreads();
    // the rows' largest components
    if (along_rows) {
        const int row = r0 + t % kSpRows;
        int m = kExpZero;
        if (row < o.rows)
            for (int k = t / kSpRows; k < a.K; k += kSpThreads / kSpRows)
                m = max(m, dz_exponent(dz_load(o.op, base, row, k)) + shift[k]);
        atomicMax(&smax[t % kSpRows], m);
    } else {
        // a warp's rows together, for as many loads in flight
        constexpr int kWarps = kSpThreads / 32, kPer = kSpRows / kWarps;
        int m[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) m[i] = kExpZero;
#pragma unroll 2
        for (int k = t % 32; k < a.K; k += 32)
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int row = min(r0 + t / 32 + kWarps * i, o.rows - 1);
                m[i] = max(m[i], dz_exponent(dz_load(o.op, base, row, k)) + shift[k]);
            }
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            m[i] = __reduce_max_sync(0xffffffffu, m[i]);
            if (t % 32 == 0) smax[t / 32 + kWarps * i] = m[i];
        }
    }
    __syncthreads();
    if (blockIdx.y == 0 && t < kSpRows && r0 + t < o.rows) {
        const int E = smax[t];
        o.scale[(long)(o.batch0 + b) * o.rows + r0 + t] = E >= kExpBad / 2 ? kFixBad : E - 1022 - kTopD + 8 * (kSl - 1);
    }
    const int rr = t / 8, seg = t % 8;                // this thread's row and pair of complex values
    const int E = smax[rr];
    const long plane = o.tiles * kM * (long)a.kblocks * kKB;
    auto fetch = [&](int kb, double2 (&v)[2]) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int kk = kb * (kKB / 2) + 2 * seg + i;
            v[i] = r0 + rr < o.rows && kk < a.K ? dz_load(o.op, base, r0 + rr, kk) : make_double2(0.0, 0.0);
        }
    };
    const int kb0 = a.kblocks * (int)blockIdx.y / (int)gridDim.y, kb1 = a.kblocks * (int)(blockIdx.y + 1) / (int)gridDim.y;
    double2 ahead[2];
    if (!along_rows) fetch(kb0, ahead);
    for (int kb = kb0; kb < kb1; ++kb) {
        double2 v[2];
        if (along_rows) {
            __syncthreads();
            for (int i = t; i < kSpRows * (kKB / 2); i += kSpThreads) {
                const int row = i % kSpRows, k = i / kSpRows;
                const int kk = kb * (kKB / 2) + k;
                sm[row][k] = r0 + row < o.rows && kk < a.K ? dz_load(o.op, base, r0 + row, kk) : make_double2(0.0, 0.0);
            }
            __syncthreads();
            v[0] = sm[rr][2 * seg];
            v[1] = sm[rr][2 * seg + 1];
        } else {
            v[0] = ahead[0];
            v[1] = ahead[1];
            if (kb + 1 < kb1) fetch(kb + 1, ahead);
        }
        long long n[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int kk = kb * (kKB / 2) + 2 * seg + i;
            const int s = kk < a.K ? E - shift[kk] : E;
            n[2 * i] = fix_in<kTopD>(v[i].x, s);
            n[2 * i + 1] = fix_in<kTopD>(v[i].y, s);
        }
        if (o.b) {
            const long row = (long)(o.batch0 + b) * o.rows_pad + 2 * (r0 + rr);
            __nv_bfloat16 *x = o.x + ((row / kM * a.kblocks + kb) * kM + row % kM) * kKB + 4 * seg;
            const long long p[4] = {n[0], -n[1], n[2], -n[3]}, q[4] = {n[1], n[0], n[3], n[2]};
            dz_store(x, plane, p);
            dz_store(x + kKB, plane, q);
        } else {
            const long row = (long)(o.batch0 + b) * o.rows_pad + r0 + rr;
            dz_store(o.x + ((row / kM * a.kblocks + kb) * kM + row % kM) * kKB + 4 * seg, plane, n);
        }
    }
}

// ------------------------------------------------------------------ GEMM --
// As in bgw_chi0_f64tc.cu: K-major, 64-byte swizzle, 8-row atoms 512 B apart.
__device__ __forceinline__ uint64_t desc64(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}
// kind::f16, D = F32, A = B = BF16, both K-major, M = 128, N = 64
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kN >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);

__device__ __forceinline__ void mma_dz(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate)
        : "memory");
}
// 64 rows x 32 k' (4 KB) at {0, row, kb, rt, plane} of the 5-D map
__device__ __forceinline__ void tma_rows(uint32_t dst, const CUtensorMap *map, uint32_t bar, int row, int kb, int rt,
                                         int plane) {
    const int zero = 0;
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(zero), "r"(row), "r"(kb), "r"(rt), "r"(plane)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

enum { kOne, kMinusOne, kReal, kComplex };
struct GemmArgs {
    CUtensorMap ma, mb;
    const int *ea, *eb;      // scales [batch][M], [batch][N]
    DzOut out;
    int M, N, ta, tb;        // rows, columns, tiles per matrix
    int rpa, rpb;            // padded rows per matrix of each operand
    int b0a, b0b;            // first matrix of each operand's planes
    int nkb, items;
    int alpha;               // kOne ...: no FP64 compare per output
    int drop;                // test hook: block 0 never issues its first stage
};

__global__ void __launch_bounds__(kThreads, 1) k_dz_gemm(const __grid_constant__ GemmArgs g, int *__restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kStg], empty_bar[kStg], set_full, set_free;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStg; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        mbar_init(smem_u32(&set_full), 1);
        mbar_init(smem_u32(&set_free), kEpi * 32);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kEpi) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const int per = g.ta * g.tb;

    if (warp == kEpi) {
        if (lane == 0) {
            long pit = 0, dropped = -1;
            bool stop = false;
            for (int item = blockIdx.x; item < g.items && !stop; item += gridDim.x) {
                const int b = item / per, ti = item % per / g.tb, tj = item % per % g.tb;
                const int ra = (g.b0a + b) * g.rpa + ti * kM, rb = (g.b0b + b) * g.rpb + tj * kN;
                for (int kb = 0; kb < g.nkb; ++kb, ++pit) {
                    const int s = (int)(pit % kStg);
                    if (!mbar_wait(smem_u32(&empty_bar[s]), (uint32_t)(((pit / kStg) & 1) ^ 1))) {
                        atomicExch(err, kErrEmpty);
                        atomicExch(&abort_flag, 1);
                        stop = true;
                        break;
                    }
                    if (*(volatile int *)&abort_flag) {
                        stop = true;
                        break;
                    }
                    if (g.drop && blockIdx.x == 0 && pit == 0) {
                        dropped = pit;
                        continue;
                    }
                    const uint32_t st0 = ring + s * kStage, fb = smem_u32(&full_bar[s]);
                    mbar_expect_tx(fb, kStage);
                    for (int t = 0; t < kSl; ++t) {
                        tma_rows(st0 + t * kTileA, &g.ma, fb, 0, kb, ra / kM, t);
                        tma_rows(st0 + t * kTileA + kTileA / 2, &g.ma, fb, 64, kb, ra / kM, t);
                        tma_rows(st0 + kSl * kTileA + t * kTileB, &g.mb, fb, rb % kM, kb, rb / kM, t);
                    }
                }
            }
            // every issued load must land before the CTA can exit
            for (long q = pit > kStg ? pit - kStg : 0; q < pit; ++q)
                if (q != dropped && !mbar_wait(smem_u32(&full_bar[q % kStg]), (uint32_t)((q / kStg) & 1))) {
                    atomicExch(err, kErrDrain);
                    break;
                }
        }
        __syncwarp();
    } else if (warp == kEpi + 1) {
        if (lane == 0) {
            long pit = 0, gsub = 0;
            bool stop = false;
            for (int item = blockIdx.x; item < g.items && !stop; item += gridDim.x) {
                for (int kb = 0; kb < g.nkb; ++kb, ++pit) {
                    const bool first = kb % kSub == 0;
                    if (first && !mbar_wait(smem_u32(&set_free), (uint32_t)((gsub & 1) ^ 1))) {
                        atomicExch(err, kErrAccum);
                        atomicExch(&abort_flag, 1);
                        stop = true;
                        break;
                    }
                    const int s = (int)(pit % kStg);
                    if (!mbar_wait(smem_u32(&full_bar[s]), (uint32_t)((pit / kStg) & 1))) {
                        atomicExch(err, kErrFull);
                        atomicExch(&abort_flag, 1);
                        stop = true;
                        break;
                    }
                    if (*(volatile int *)&abort_flag) {
                        stop = true;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t st0 = ring + s * kStage;
#pragma unroll
                    for (int k = 0; k < kKB / 16; ++k) {
                        const uint64_t o = (uint64_t)(2 * k);   // 16 BF16 = 32 bytes along k'
#pragma unroll
                        for (int t = 0; t < kSl; ++t) {
                            const uint64_t ad = desc64(st0 + t * kTileA) + o;
#pragma unroll
                            for (int u = 0; u + t < kSl; ++u) {
                                const int lev = t + u < kAcc - 1 ? t + u : kAcc - 1;
                                const uint64_t bd = desc64(st0 + kSl * kTileA + u * kTileB) + o;
                                const bool start = first && k == 0 && t == 0 && u < kAcc;
                                mma_dz(tmem + (uint32_t)(lev * kN), ad, bd, start ? 0u : 1u);
                            }
                        }
                    }
                    mma_commit(smem_u32(&empty_bar[s]));
                    if (kb % kSub == kSub - 1 || kb == g.nkb - 1) {
                        mma_commit(smem_u32(&set_full));
                        ++gsub;
                    }
                }
            }
        }
        __syncwarp();
    } else {
        // warp w: TMEM lanes 32 (w & 3).. (tile rows), columns 16 (w >> 2)..
        const int quarter = warp & 3, group = warp >> 2;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(16 * group);
        long gsub = 0;
        for (int item = blockIdx.x; item < g.items; item += gridDim.x) {
            const int b = item / per, ti = item % per / g.tb, tj = item % per % g.tb;
            long long n[16];       // sum of orders 0-5 in units of 2^-36,
            float f[16];           // what lies below them, and orders 6 and 7
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                n[i] = 0;
                f[i] = 0.f;
            }
            const int nsub = (g.nkb + kSub - 1) / kSub;
            for (int sub = 0; sub < nsub; ++sub, ++gsub) {
                bool got = !*(volatile int *)&abort_flag && mbar_wait(smem_u32(&set_full), (uint32_t)(gsub & 1));
                got = __all_sync(0xffffffffu, got && !*(volatile int *)&abort_flag);
                if (!got) {                     // no further waits: NaN for this tile and the rest
                    if (lane == 0) atomicExch(err, kErrAccum);
                    atomicExch(&abort_flag, 1);
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint32_t v[16];
                int h[16];
                // orders 0 and 1 (below 2^20 and 2^21 units), 2 and 3 (2^23, 2^24) join in 32 bits
#pragma unroll
                for (int o = 0; o < 4; o += 2) {
                    const float s0 = o ? 0x1p16f : 1.0f, s1 = o ? 0x1p24f : 0x1p8f;
                    tmem_ld16(lane_base + (uint32_t)(o * kN), v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) h[i] = __float2int_rn(__uint_as_float(v[i]) * s0) * 256;
                    tmem_ld16(lane_base + (uint32_t)((o + 1) * kN), v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int d = h[i] + __float2int_rn(__uint_as_float(v[i]) * s1);
                        n[i] += (long long)d << (o ? 12 : 28);
                    }
                }
                tmem_ld16(lane_base + (uint32_t)(4 * kN), v);
#pragma unroll
                for (int i = 0; i < 16; ++i) n[i] += (long long)__float2int_rn(__uint_as_float(v[i]) * 0x1p32f) << 4;
                tmem_ld16(lane_base + (uint32_t)(5 * kN), v);
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int d = __float2int_rn(__uint_as_float(v[i]) * 0x1p40f);
                    n[i] += d >> 4;
                    f[i] += (float)(d & 15) * 0x1p-40f;
                }
                tmem_ld16(lane_base + (uint32_t)((kAcc - 1) * kN), v);
#pragma unroll
                for (int i = 0; i < 16; ++i) f[i] += __uint_as_float(v[i]);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                mbar_arrive(smem_u32(&set_free));
            }
            const int m = ti * kM + 32 * quarter + lane;
            const int n0 = (tj * kN + 16 * group) / 2;
            const DzOut &o = g.out;
            if (m < g.M && !(m >= o.skip0 && m < o.skip1)) {
                const int ea = *(volatile int *)&abort_flag ? kFixBad : g.ea[(long)(g.b0a + b) * g.M + m];
                const int *ebp = g.eb + (long)(g.b0b + b) * g.N;
                double2 *c = o.c + b * o.sb + m * o.sm + n0 * o.sn;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int nn = n0 + i;
                    if (nn >= g.N || (nn >= o.skip0 && nn < o.skip1)) continue;
                    const int eb = ebp[nn];
                    double2 *p = c + i * o.sn;
                    double2 old = make_double2(0.0, 0.0);
                    if (o.accumulate) old = *p;
                    double d[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int q = 2 * i + h;
                        long long x = n[q];
                        // the last sum is a fraction of x's unit: bring x up to make room for it
                        const int sh = min(max(__clzll(x < 0 ? ~x : x) - 2, 0), 26);
                        // units of 2^-52: up to 2^34 of them where a long sum's terms agree in sign
                        const long long fr = __float2ll_rn(f[q] * 0x1p52f);
                        x = (x << sh) + (sh >= 16 ? fr << (sh - 16) : fr >> (16 - sh));
                        if (g.alpha == kMinusOne) x = -x;
                        d[h] = fix_out(x, 1086 - 36 - sh + ea + eb);
                    }
                    double2 r = make_double2(d[0], d[1]);
                    if (ea == kFixBad || eb == kFixBad) r.x = r.y = __longlong_as_double(0x7ff8000000000000ll);
                    if (g.alpha == kComplex)
                        r = make_double2(o.ar * r.x - o.ai * r.y, o.ar * r.y + o.ai * r.x);
                    else if (g.alpha == kReal)
                        r = make_double2(o.ar * r.x, o.ar * r.y);
                    if (o.accumulate) r = make_double2(r.x + old.x, r.y + old.y);
                    *p = r;
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == kEpi)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

long round_up(long x, long m) { return (x + m - 1) / m * m; }
size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

int pad_rows(int rows, bool b) { return (int)(b ? round_up(2L * rows, kN) : round_up(rows, kM)); }
long tile_rows(const DzPlanes &p) { return round_up((long)p.batch * p.rows_pad, kM); }
size_t plane_bytes(const DzPlanes &p) { return align256((size_t)kSl * tile_rows(p) * p.kblocks * kKB * 2); }

cudaError_t make_map(const DzPlanes &p, CUtensorMap *m) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = nullptr;
    const cudaError_t e = tc::tensor_map_encoder(&enc);
    if (e != cudaSuccess) return e;
    const cuuint64_t tile = (cuuint64_t)kM * kKB * 2, nt = (cuuint64_t)(tile_rows(p) / kM);
    const cuuint64_t dims[5] = {(cuuint64_t)kKB, (cuuint64_t)kM, (cuuint64_t)p.kblocks, nt, (cuuint64_t)kSl};
    const cuuint64_t strides[4] = {(cuuint64_t)kKB * 2, tile, tile * p.kblocks, tile * p.kblocks * nt};
    const cuuint32_t box[5] = {kKB, 64, 1, 1, 1}, estr[5] = {1, 1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, p.x, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? cudaSuccess
               : cudaErrorInvalidValue;
}

}  // namespace

DzPlanes dz_planes(void *ws, int rows, int K, int batch, bool b) {
    DzPlanes p;
    p.x = ws;
    p.rows = rows;
    p.rows_pad = pad_rows(rows, b);
    p.kblocks = (int)(round_up(2L * K, kKB) / kKB);
    p.batch = p.used = batch;
    p.first = 0;
    p.b = b;
    p.scale = reinterpret_cast<int *>(static_cast<char *>(ws) + plane_bytes(p));
    return p;
}

size_t dz_planes_bytes(int rows, int K, int batch, bool b) {
    const DzPlanes p = dz_planes(nullptr, rows, K, batch, b);
    return plane_bytes(p) + align256(sizeof(int) * (size_t)batch * rows);
}

size_t dz_balance_bytes(int K) { return align256(sizeof(int) * 2 * (size_t)K); }

cudaError_t dz_balance(DzOperand &A, long rowsA, DzOperand &B, long rowsB, int K, void *ws, int *err, cudaStream_t st) {
    BalanceArgs a;
    a.op[0] = A;
    a.op[1] = B;
    a.rows[0] = rowsA;
    a.rows[1] = rowsB;
    a.col[0] = static_cast<int *>(ws);
    a.col[1] = a.col[0] + K;
    a.err = err;
    a.K = K;
    const size_t smem = sizeof(short) * kBalRows * (size_t)K;
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024)
        e = cudaFuncSetAttribute(k_dz_balance, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    // every byte 0x80: far below kExpZero.  (Cleared by the product before it instead,
    // at the start of its k_dz_gemm, the products took 7 us longer each.)
    if (e == cudaSuccess) e = cudaMemsetAsync(ws, 0x80, sizeof(int) * 2 * (size_t)K, st);
    if (e != cudaSuccess) return e;
    const long blocks = (rowsA + kBalRows - 1) / kBalRows + (rowsB + kBalRows - 1) / kBalRows;
    k_dz_balance<<<(unsigned)blocks, 32 * kBalRows, smem, st>>>(a);
    A.cols = B.other = a.col[0];
    B.cols = A.other = a.col[1];
    A.second = false;
    B.second = true;
    return cudaGetLastError();
}

cudaError_t dz_split(const DzOperand *op, const DzPlanes *pl, int n, int K, cudaStream_t st) {
    if (n < 1 || n > kMaxOps) return cudaErrorInvalidValue;
    SplitArgs a;
    a.n = n;
    a.K = K;
    a.kblocks = pl[0].kblocks;
    unsigned blocks = 0;
    for (int i = 0; i < n; ++i) {
        const DzPlanes &p = pl[i];
        a.o[i] = SplitOp{op[i], static_cast<__nv_bfloat16 *>(p.x), p.scale, p.rows, p.rows_pad, p.b ? 1 : 0,
                         p.first, tile_rows(p) / kM, blocks};
        blocks += (unsigned)(p.used * (p.rows_pad / (p.b ? 2 * kSpRows : kSpRows)));
    }
    // few rows: the k' blocks of a row, at least two at a time, go to as many thread
    // blocks as give every SM two (7 x 21 pairs of 350 G: 44 -> 24 us a launch)
    const int parts = (int)(2 * 152 / blocks), most = a.kblocks / 2;
    const int y = parts < 1 || most < 1 ? 1 : parts < most ? parts : most;
    k_dz_split<<<dim3(blocks, y), kSpThreads, sizeof(int) * (size_t)K, st>>>(a);
    return cudaGetLastError();
}

cudaError_t dz_gemm(const DzPlanes &A, const DzPlanes &B, const DzOut &out, int sm_count, cudaStream_t st, int *err,
                    bool drop) {
    GemmArgs g;
    memset(&g, 0, sizeof g);
    cudaError_t e = make_map(A, &g.ma);
    if (e == cudaSuccess) e = make_map(B, &g.mb);
    if (e != cudaSuccess) return e;
    g.ea = A.scale;
    g.eb = B.scale;
    g.out = out;
    g.M = A.rows;
    g.N = B.rows;
    g.rpa = A.rows_pad;
    g.rpb = B.rows_pad;
    g.ta = A.rows_pad / kM;
    g.tb = B.rows_pad / kN;
    g.nkb = A.kblocks;
    g.b0a = A.first;
    g.b0b = B.first;
    g.items = A.used * g.ta * g.tb;
    g.alpha = out.ai != 0.0 ? kComplex : out.ar == 1.0 ? kOne : out.ar == -1.0 ? kMinusOne : kReal;
    g.drop = drop;
    const int smem = kStg * kStage + 1024;
    e = cudaFuncSetAttribute(k_dz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_dz_gemm<<<g.items < sm_count ? g.items : sm_count, kThreads, smem, st>>>(g, err);
    return cudaGetLastError();
}

}  // namespace bgw
