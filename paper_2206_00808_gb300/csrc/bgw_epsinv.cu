// Dielectric matrix inverse and screened interaction on the GPU (FP64).
//
// arXiv:2206.00808, Sec. II, the two equations before the P formula:
//     eps_GG'(q, w) = delta_GG' - v(q+G) P_GG'(q, w),    W_GG' = eps^-1_GG' v(q+G').
// With s_G = sqrt(v(q+G)) the symmetrised matrix
//     eps~ = S^-1 eps S = I - S P S        (S = diag(s))
// is Hermitian, and positive definite because P = chi0 is negative
// semidefinite on the imaginary axis (every pair weight 2D/(D^2+w^2) < 0).
// Then eps^-1 = S eps~^-1 S^-1 and W = eps^-1 S^2 = S eps~^-1 S.
//
// eps~ is inverted in place by blocked Gauss-Jordan elimination without
// pivoting (valid for Hermitian positive definite matrices: every pivot block
// is a Schur complement of one and is itself positive definite).  For the
// block K of kb <= 32 indices and the rest R, one step is
//     P = A_KK^-1,  A_RR -= A_RK P A_KR,  A_KR <- P A_KR,  A_RK <- -A_RK P,  A_KK <- P
// (the block form of the scalar in-place Gauss-Jordan step); after every block
// has been taken the array holds the inverse.  Each step is four launches:
// k6_diag (one CTA per matrix inverts the kb x kb block in shared memory),
// k6_panels (P A_KR and A_RK P into a workspace), k6_update (the rank-kb
// update of all (r, c) outside K, tiled 32 x 32 in shared memory: this is
// where the 8 n^3 flops per matrix go, on the FP64 pipe), k6_writeback.
// All matrices of a call (one per frequency) go through each launch together.
//
// From kDzMinN rows on, the two panels and the update are products on tensor
// cores from BF16 digits (bgw_dz.cu, more exact than FP64 sums): the digits of
// A_RK, of A_KR and of P both ways, one product for both panels (as 2 nf
// matrices), the digits of P A_KR, and one product for the update.  The FP64
// pipe ran the update at 0.94 of its rate, 64 ms for 16 x 800^2; now 9.1 ms, of
// which the update takes 4.6 (bound by its epilogue's integer work), k6_diag 2.0
// (one SM a matrix) and the digits 0.8.
//
// Elimination does not notice a scaling of rows and columns by powers of two, but
// digits, cut on a scale per row, do: where eps~ = D B D, a large d_k of one factor
// meets 1/d_k of the other (s_0 2^20 times the others', a metal's head at small q:
// 7e-14 of the largest entry instead of 1e-15).  So k6_balance takes D out: it
// finds the power of two nearest 1/sqrt(eps~_GG) for every G, which k6_build
// applies with S and k6_scale undoes.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>

#include "../../include/bgw_chi.h"
#include "bgw_dz.h"

namespace {

constexpr int kB = 32;           // Gauss-Jordan block
constexpr int kTile = 32;        // update tile (rows and columns): many CTAs per panel step
constexpr int kErrPivot = 1;
// Rows from which the products run on tensor cores.  One matrix of 96 rows: 566 us
// a call in FP64, 454 from digits; 160 917 / 725, 16 matrices of 224 rows 2637 /
// 1139 (with a k6_diag 8 us a block faster).  (Digits are also faster below, 64
// rows 396 / 323 us and 48 rows 314 / 275, where a call is launches and k6_diag;
// small matrices keep their workspace.)
constexpr int kDzMinN = 96;

struct Z {
    double x, y;
};
__device__ __forceinline__ Z zmul(Z a, Z b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ Z zfma(Z a, Z b, Z c) {   // a * b + c
    return {fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y))};
}

// Power-of-two scales of eps~ (see above), per matrix: x = 2^e with e nearest
// -log2(eps~_GG) / 2, and s x and s / x.
__global__ void k6_balance(const double2 *__restrict__ chi, const double *__restrict__ s, int n,
                           double *__restrict__ sx, double *__restrict__ sox, int *__restrict__ ex) {
    const long j = blockIdx.y;
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    const double sg = s[g], d = 1.0 - sg * sg * chi[(j * n + g) * (long)n + g].x;
    int e = 0;
    if (d > 0.0 && isfinite(d)) e = -((ilogb(d) + 1) >> 1);       // else: a pivot will not be positive
    ex[j * n + g] = e;
    sx[j * n + g] = scalbn(sg, e);
    sox[j * n + g] = scalbn(sg, -e);
}

// A = X (I - S chi S) X in place; chi: [nf][n][n] complex128.  sx: S X, one
// vector (stride 0, X = I, ex null) or one per matrix (stride n).
__global__ void k6_build(double2 *__restrict__ A, const double *__restrict__ sx, int stride,
                         const int *__restrict__ ex, int n) {
    const long j = blockIdx.z;
    const int r = blockIdx.y;
    double2 *row = A + (j * n + r) * (long)n;
    sx += j * stride;
    const double sr = sx[r];
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        double2 v = row[c];
        const double f = -sr * sx[c];
        v.x *= f;
        v.y *= f;
        if (c == r) v.x += ex ? scalbn(1.0, 2 * ex[j * n + r]) : 1.0;
        row[c] = v;
    }
}

// Invert the kb x kb block at (k0, k0) of every matrix in place (unblocked
// Gauss-Jordan, no pivoting).  One CTA per matrix, a 2 x 2 group of entries
// per thread.  Bound: the FP64 pipe of one SM, 4 kb^2 operations a pivot; the
// reciprocal of the next pivot is formed by the one thread that updates it
// while the others still update (every thread forming its own took 175 us a
// call of 16 blocks).  The products of an update are summed before they meet the
// entry, which is then rounded once: two fused multiply-adds onto it round it
// twice, for half as much error again in the inverse (95 rows 5.1e-16 against
// 3.4e-16).  The scaled row is formed once, by one warp, for half of what that
// costs (16 blocks 72 -> 80 us).
__device__ __forceinline__ Z zinv(Z p, int *bad) {
    const double t = p.y / p.x, den = fma(p.y, t, p.x);  // 1/p = (1 - i t) / (p.x + p.y t), p.y ~ 0 here
    if (!(p.x > 0.0) || !isfinite(p.x * p.x + p.y * p.y)) *bad = 1;       // not positive definite
    const double f = 1.0 / den;
    return {f, -t * f};
}

__global__ void __launch_bounds__(256) k6_diag(double2 *__restrict__ A, int n, int k0, int kb, int *err) {
    __shared__ Z row[2][kB], col[2][kB], pivinv[2], scaled[kB];
    __shared__ int bad[2];       // of the current and the next pivot: never written while it is read
    const long j = blockIdx.x;
    double2 *M = A + j * (long)n * n;
    const int r0 = threadIdx.x / 16, c0 = threadIdx.x % 16;       // entries (r0 + 16 i, c0 + 16 l)
    if (threadIdx.x < 2) bad[threadIdx.x] = 0;
    __syncthreads();
    Z a[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const int r = r0 + 16 * i, c = c0 + 16 * l;
            double2 v = make_double2(r == c ? 1.0 : 0.0, 0.0);     // the identity beyond kb
            if (r < kb && c < kb) v = M[(long)(k0 + r) * n + k0 + c];
            a[i][l] = {v.x, v.y};
            if (r == 0) row[0][c] = a[i][l];
            if (c == 0) col[0][r] = a[i][l];
            if (r == 0 && c == 0) pivinv[0] = zinv(a[i][l], &bad[0]);
        }
    __syncthreads();
    for (int k = 0; k < kb; ++k) {
        const int cur = k & 1, nxt = cur ^ 1;
        const Z p = pivinv[cur];
        if (bad[cur]) {                                     // uniform: set before the last barrier
            if (threadIdx.x == 0) atomicExch(err, kErrPivot);
            return;
        }
        // row k scaled, g = a_k. / p, and the multipliers -a_.k of this thread's rows
        if (threadIdx.x < kB) scaled[threadIdx.x] = threadIdx.x == k ? p : zmul(row[cur][threadIdx.x], p);
        __syncthreads();
        Z g[2], f[2];
#pragma unroll
        for (int l = 0; l < 2; ++l) g[l] = scaled[c0 + 16 * l];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            f[i] = col[cur][r0 + 16 * i];
            f[i] = {-f[i].x, -f[i].y};
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                const int r = r0 + 16 * i, c = c0 + 16 * l;
                Z v = c == k ? Z{0.0, 0.0} : a[i][l];       // column k becomes -a_rk / p
                const Z t = zmul(f[i], g[l]);
                v = r == k ? g[l] : Z{v.x + t.x, v.y + t.y};
                a[i][l] = v;
                if (r == k + 1) row[nxt][c] = v;
                if (c == k + 1) col[nxt][r] = v;
                if (r == k + 1 && c == k + 1) pivinv[nxt] = zinv(v, &bad[nxt]);
            }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const int r = r0 + 16 * i, c = c0 + 16 * l;
            if (r < kb && c < kb) M[(long)(k0 + r) * n + k0 + c] = make_double2(a[i][l].x, a[i][l].y);
        }
}

// T[j][i][c] = sum_k P[i][k] A[k0+k][c]   (row panel, every column c)
// U[j][r][i] = sum_k A[r][k0+k] P[k][i]   (column panel, every row r)
// with P = A_KK already inverted in place.  Each thread computes kPanelI
// consecutive i for one column (or row) x.  grid (ceil(n/128), kB/kPanelI,
// 2 nf): z even for T, odd for U.
constexpr int kPanelI = 8;

__global__ void __launch_bounds__(128) k6_panels(const double2 *__restrict__ A, int n, int k0, int kb,
                                                 double2 *__restrict__ T, double2 *__restrict__ U) {
    __shared__ Z P[kB][kB + 1];
    const long j = blockIdx.z >> 1;
    const bool row_panel = (blockIdx.z & 1) == 0;
    const double2 *M = A + j * (long)n * n;
    for (int i = threadIdx.x; i < kb * kb; i += blockDim.x) {
        const double2 v = M[(long)(k0 + i / kb) * n + k0 + i % kb];
        P[i / kb][i % kb] = {v.x, v.y};
    }
    __syncthreads();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int i0 = blockIdx.y * kPanelI;
    if (x >= n || i0 >= kb) return;
    Z acc[kPanelI];
#pragma unroll
    for (int i = 0; i < kPanelI; ++i) acc[i] = {0.0, 0.0};
    if (row_panel) {                                      // column c = x of P A_K.
        for (int k = 0; k < kb; ++k) {
            const double2 v = M[(long)(k0 + k) * n + x];
            const Z b = {v.x, v.y};
#pragma unroll
            for (int i = 0; i < kPanelI; ++i)
                if (i0 + i < kb) acc[i] = zfma(P[i0 + i][k], b, acc[i]);
        }
        double2 *t = T + j * (long)kB * n + x;
#pragma unroll
        for (int i = 0; i < kPanelI; ++i)
            if (i0 + i < kb) t[(long)(i0 + i) * n] = make_double2(acc[i].x, acc[i].y);
    } else {                                              // row r = x of A_.K P
        const double2 *row = M + (long)x * n + k0;
        for (int k = 0; k < kb; ++k) {
            const double2 v = row[k];
            const Z a = {v.x, v.y};
#pragma unroll
            for (int i = 0; i < kPanelI; ++i)
                if (i0 + i < kb) acc[i] = zfma(a, P[k][i0 + i], acc[i]);
        }
        double2 *u = U + (j * (long)n + x) * kB + i0;
#pragma unroll
        for (int i = 0; i < kPanelI; ++i)
            if (i0 + i < kb) u[i] = make_double2(acc[i].x, acc[i].y);
    }
}

// A[r][c] -= sum_k A[r][k0+k] T[k][c] for r, c outside [k0, k0+kb).
// One CTA per 32 x 32 tile (rows r0.., columns c0..) of one matrix; 256
// threads, each a 2 x 2 block of complex outputs (small tiles keep every SM
// busy at N_G of a few hundred); outputs in the K rows or K columns are
// computed and dropped.
constexpr int kLRow = kB + 1, kRRow = kTile + 1;
constexpr size_t kUpdateSmem = sizeof(Z) * ((size_t)kTile * kLRow + (size_t)kB * kRRow);

__global__ void __launch_bounds__(256) k6_update(double2 *__restrict__ A, int n, int k0, int kb,
                                                 const double2 *__restrict__ T) {
    extern __shared__ Z upd_sm[];
    Z (*L)[kLRow] = reinterpret_cast<Z (*)[kLRow]>(upd_sm);                       // A[r0 + i][k0 + k]
    Z (*R)[kRRow] = reinterpret_cast<Z (*)[kRRow]>(upd_sm + (size_t)kTile * kLRow);   // T[k][c0 + i]
    const long j = blockIdx.z;
    const int r0 = blockIdx.y * kTile, c0 = blockIdx.x * kTile;
    double2 *M = A + j * (long)n * n;
    const double2 *Tj = T + j * (long)kB * n;
    for (int i = threadIdx.x; i < kTile * kB; i += blockDim.x) {
        const int r = i / kB, k = i % kB;
        Z v = {0.0, 0.0};
        if (r0 + r < n && k < kb) {
            const double2 w = M[(long)(r0 + r) * n + k0 + k];
            v = {w.x, w.y};
        }
        L[r][k] = v;
    }
    for (int i = threadIdx.x; i < kB * kTile; i += blockDim.x) {
        const int k = i / kTile, c = i % kTile;
        Z v = {0.0, 0.0};
        if (c0 + c < n && k < kb) {
            const double2 w = Tj[(long)k * n + c0 + c];
            v = {w.x, w.y};
        }
        R[k][c] = v;
    }
    __syncthreads();
    constexpr int RA = kTile / 16;                              // outputs per thread per axis
    const int tr = threadIdx.x / 16, tc = threadIdx.x % 16;   // rows tr + 16a, columns tc + 16b
    Z acc[RA][RA];
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
        for (int b = 0; b < RA; ++b) acc[a][b] = {0.0, 0.0};
    for (int k = 0; k < kb; ++k) {
        Z l[RA], r[RA];
#pragma unroll
        for (int a = 0; a < RA; ++a) l[a] = L[tr + 16 * a][k];
#pragma unroll
        for (int b = 0; b < RA; ++b) r[b] = R[k][tc + 16 * b];
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
            for (int b = 0; b < RA; ++b) acc[a][b] = zfma(l[a], r[b], acc[a][b]);
    }
#pragma unroll
    for (int a = 0; a < RA; ++a) {
        const int r = r0 + tr + 16 * a;
        if (r >= n || (r >= k0 && r < k0 + kb)) continue;
#pragma unroll
        for (int b = 0; b < RA; ++b) {
            const int c = c0 + tc + 16 * b;
            if (c >= n || (c >= k0 && c < k0 + kb)) continue;
            double2 *o = M + (long)r * n + c;
            double2 v = *o;
            v.x -= acc[a][b].x;
            v.y -= acc[a][b].y;
            *o = v;
        }
    }
}

// A_KR <- T (columns outside K), A_RK <- -U (rows outside K).
__global__ void k6_writeback(double2 *__restrict__ A, int n, int k0, int kb, const double2 *__restrict__ T,
                             const double2 *__restrict__ U) {
    const long j = blockIdx.z;
    double2 *M = A + j * (long)n * n;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n || (x >= k0 && x < k0 + kb)) return;
    const double2 *t = T + j * (long)kB * n + x;
    for (int i = 0; i < kb; ++i) M[(long)(k0 + i) * n + x] = t[(long)i * n];
    const double2 *u = U + (j * (long)n + x) * kB;
    for (int i = 0; i < kb; ++i) {
        const double2 v = u[i];
        M[(long)x * n + k0 + i] = make_double2(-v.x, -v.y);
    }
}

// The same from panels stored by column, T[c][i], and by row, U[r][i]: a block
// takes 32 columns (rows) and turns T through shared memory.
__global__ void __launch_bounds__(256) k6_writeback_t(double2 *__restrict__ A, int n, int k0, int kb,
                                                      const double2 *__restrict__ T, const double2 *__restrict__ U) {
    __shared__ double2 t[32][kB + 1];
    const long j = blockIdx.z;
    double2 *M = A + j * (long)n * n;
    const int x0 = blockIdx.x * 32;
    for (int e = threadIdx.x; e < 32 * kB; e += 256) {
        const int x = x0 + e / kB, i = e % kB;
        if (x < n && i < kb) {
            const long at = (j * (long)n + x) * kB + i;
            t[e / kB][i] = T[at];
            if (x < k0 || x >= k0 + kb) {
                const double2 u = U[at];
                M[(long)x * n + k0 + i] = make_double2(-u.x, -u.y);
            }
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 32 * kB; e += 256) {
        const int x = x0 + e % 32, i = e / 32;
        if (x < n && i < kb && (x < k0 || x >= k0 + kb)) M[(long)(k0 + i) * n + x] = t[e % 32][i];
    }
}

// From the inverse A of X eps~ X: W = S X A X S (mode 1) or eps^-1 = S X A X S^-1
// (mode 2), with sx = S X and div = S X^-1 (both S, stride 0, where X = I).
__global__ void k6_scale(double2 *__restrict__ A, const double *__restrict__ sx, const double *__restrict__ div,
                         int stride, int n, int inverse_cols) {
    const long j = blockIdx.z;
    const int r = blockIdx.y;
    double2 *row = A + (j * n + r) * (long)n;
    sx += j * stride;
    div += j * stride;
    const double sr = sx[r];
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        double2 v = row[c];
        const double f = inverse_cols ? sr / div[c] : sr * sx[c];
        v.x *= f;
        v.y *= f;
        row[c] = v;
    }
}

// v 2^e, exactly; through the exponent field where that can hold it.
__device__ __forceinline__ double times_pow2(double v, int e) {
    const int hi = __double2hiint(v), f = (hi >> 20) & 0x7ff;
    if (f == 0 || f == 0x7ff || f + e < 1 || f + e > 0x7fe) return scalbn(v, e);
    return __hiloint2double(hi + e * (1 << 20), __double2loint(v));
}

// eps~^-1 = X A X (mode 0).
__global__ void k6_unbalance(double2 *__restrict__ A, const int *__restrict__ ex, int n) {
    const long j = blockIdx.z;
    const int r = blockIdx.y;
    double2 *row = A + (j * n + r) * (long)n;
    const int er = ex[j * n + r];
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        const int e = er + ex[j * n + c];
        if (e == 0) continue;
        const double2 v = row[c];
        row[c] = make_double2(times_pow2(v.x, e), times_pow2(v.y, e));
    }
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Workspace: the panels U and T, s, the error words and, on tensor cores, the
// digit planes of the panels (2 nf matrices), of P (2 nf) and of P A_KR (nf),
// and the scales s x, s / x and log2 x of every matrix.
struct Work {
    size_t U, T, s, err, panels, p, t, sx, sox, ex, total;
    Work(int n, int nf) {
        const size_t panel = sizeof(double2) * (size_t)nf * kB * n;
        U = 0;
        T = panel;
        s = align256(2 * panel);
        err = s + align256(sizeof(double) * (size_t)n);
        panels = p = t = sx = sox = ex = total = err + 256;
        if (n >= kDzMinN) {
            p = panels + bgw::dz_planes_bytes(n, kB, 2 * nf, false);
            t = p + bgw::dz_planes_bytes(kB, kB, 2 * nf, true);
            sx = t + bgw::dz_planes_bytes(n, kB, nf, true);
            sox = sx + align256(sizeof(double) * (size_t)nf * n);
            ex = sox + align256(sizeof(double) * (size_t)nf * n);
            total = ex + align256(sizeof(int) * (size_t)nf * n);
        }
    }
};

}  // namespace

void bgw_set_global_error(const std::string &msg);

extern "C" size_t bgw_epsinv_workspace_bytes(int ng, int nfreq) {
    if (ng < 1 || nfreq < 1) return 0;
    return Work(ng, nfreq).total;
}

extern "C" bgw_status bgw_coulomb_sqrt(const double *avec, const double *q, int ng, const int *gvec, double *s) {
    if (!avec || !q || !gvec || !s || ng < 1) {
        bgw_set_global_error("coulomb_sqrt: null pointer or ng < 1");
        return BGW_E_ARG;
    }
    const double kPi = 3.14159265358979323846;
    const double kE2 = 27.211386245988;     // e^2 in eV bohr (1 Hartree bohr)
    const double *a0 = avec, *a1 = avec + 3, *a2 = avec + 6;
    // reciprocal rows b_i = 2 pi (a_j x a_k) / det, (i, j, k) cyclic
    const double *pa[3][2] = {{a1, a2}, {a2, a0}, {a0, a1}};
    double b[3][3];
    const double det = a0[0] * (a1[1] * a2[2] - a1[2] * a2[1]) - a0[1] * (a1[0] * a2[2] - a1[2] * a2[0]) +
                       a0[2] * (a1[0] * a2[1] - a1[1] * a2[0]);
    if (!(std::fabs(det) > 0.0) || !std::isfinite(det)) {
        bgw_set_global_error("coulomb_sqrt: singular cell");
        return BGW_E_ARG;
    }
    for (int i = 0; i < 3; ++i) {
        const double *u = pa[i][0], *w = pa[i][1];
        b[i][0] = 2 * kPi * (u[1] * w[2] - u[2] * w[1]) / det;
        b[i][1] = 2 * kPi * (u[2] * w[0] - u[0] * w[2]) / det;
        b[i][2] = 2 * kPi * (u[0] * w[1] - u[1] * w[0]) / det;
    }
    const double omega = std::fabs(det);
    for (int g = 0; g < ng; ++g) {
        double k[3] = {0, 0, 0};
        for (int i = 0; i < 3; ++i)
            for (int x = 0; x < 3; ++x) k[x] += (q[i] + gvec[3 * g + i]) * b[i][x];
        const double k2 = k[0] * k[0] + k[1] * k[1] + k[2] * k[2];
        s[g] = k2 > 1e-24 ? std::sqrt(4 * kPi * kE2 / (omega * k2)) : 0.0;
    }
    return BGW_OK;
}

extern "C" bgw_status bgw_epsinv(int ng, int nfreq, const double *s, void *chi, int mode, void *work,
                                 size_t work_bytes, void *stream) {
    auto fail = [](bgw_status st, const std::string &m) {
        bgw_set_global_error(m);
        return st;
    };
    if (ng < 1 || nfreq < 1 || !s || !chi) return fail(BGW_E_ARG, "epsinv: ng, nfreq >= 1 and s, chi required");
    if (mode < 0 || mode > 2) return fail(BGW_E_ARG, "epsinv: mode must be 0 (eps~^-1), 1 (W) or 2 (eps^-1)");
    if (nfreq > 32767 || ng > 65535) return fail(BGW_E_ARG, "epsinv: ng <= 65535 and nfreq <= 32767 required");
    for (int g = 0; g < ng; ++g) {
        if (!(s[g] >= 0.0) || !std::isfinite(s[g])) return fail(BGW_E_ARG, "epsinv: s must be finite and >= 0");
        if (mode == 2 && s[g] == 0.0) return fail(BGW_E_ARG, "epsinv: mode 2 needs s > 0 (q + G = 0 in the sphere)");
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t need = bgw_epsinv_workspace_bytes(ng, nfreq);
    void *own = nullptr;
    cudaError_t e = cudaSuccess;
    if (!work) {
        e = cudaMalloc(&own, need);
        if (e != cudaSuccess)
            return fail(e == cudaErrorMemoryAllocation ? BGW_E_NOMEM : BGW_E_CUDA,
                        std::string("epsinv: workspace: ") + cudaGetErrorString(e));
        work = own;
    } else if (work_bytes < need) {
        return fail(BGW_E_ARG, "epsinv: workspace of " + std::to_string(work_bytes) + " bytes, " +
                                   std::to_string(need) + " needed");
    }
    char *w = static_cast<char *>(work);
    const Work o(ng, nfreq);
    double2 *U = reinterpret_cast<double2 *>(w + o.U), *T = reinterpret_cast<double2 *>(w + o.T);
    double *sd = reinterpret_cast<double *>(w + o.s);
    int *err = reinterpret_cast<int *>(w + o.err);        // [0] pivots, [1] device-side waits
    double2 *A = static_cast<double2 *>(chi);
    e = cudaMemcpyAsync(sd, s, sizeof(double) * ng, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, 2 * sizeof(int), st);
    const unsigned rowblocks = (unsigned)((ng + 255) / 256);
    const bool tensor = ng >= kDzMinN;
    double *sx = tensor ? reinterpret_cast<double *>(w + o.sx) : sd, *sox = tensor ? reinterpret_cast<double *>(w + o.sox) : sd;
    int *ex = tensor ? reinterpret_cast<int *>(w + o.ex) : nullptr;
    const int stride = tensor ? ng : 0;
    if (e == cudaSuccess) {
        if (tensor) k6_balance<<<dim3(rowblocks, nfreq), 256, 0, st>>>(A, sd, ng, sx, sox, ex);
        k6_build<<<dim3(rowblocks, ng, nfreq), 256, 0, st>>>(A, sx, stride, ex, ng);
        e = cudaGetLastError();
    }
    const unsigned tiles = (unsigned)((ng + kTile - 1) / kTile);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k6_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kUpdateSmem);
    int sms = 148;
    if (tensor && e == cudaSuccess) {
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    const char *fault = std::getenv("BGW_FAULT");      // test hook: the first product loses an operand load
    const bool drop = fault && !std::strcmp(fault, "drop@epsinv");
    for (int k0 = 0; k0 < ng && e == cudaSuccess; k0 += kB) {
        const int kb = ng - k0 < kB ? ng - k0 : kB;
        k6_diag<<<nfreq, 256, 0, st>>>(A, ng, k0, kb, err);
        if (tensor) {
            const long n2 = (long)ng * ng;
            bgw::DzPlanes pa = bgw::dz_planes(w + o.panels, ng, kB, 2 * nfreq, false), pr = pa;
            bgw::DzPlanes bp = bgw::dz_planes(w + o.p, kb, kB, 2 * nfreq, true), br = bp;
            pa.used = pr.used = pr.first = bp.used = br.used = br.first = nfreq;
            const double2 *row = A + (long)k0 * ng, *col = A + k0, *P = row + k0;
            // U[r] = A_rK P with P read by columns, T[c] = P A_Kc with P read by rows
            const bgw::DzPlanes pl[4] = {pa, pr, bp, br};
            const bgw::DzOperand op[4] = {{col, n2, ng, 1, false, nullptr}, {row, n2, 1, ng, false, nullptr},
                                          {P, n2, 1, ng, false, nullptr}, {P, n2, ng, 1, false, nullptr}};
            e = bgw::dz_split(op, pl, 4, kb, st);
            bgw::DzPlanes both = pa, bothp = bp;
            both.used = bothp.used = 2 * nfreq;
            if (e == cudaSuccess)
                e = bgw::dz_gemm(both, bothp, bgw::DzOut{U, (long)ng * kB, kB, 1, 0, 0, 1.0, 0.0, false}, sms, st, err + 1,
                                 drop && k0 == 0);
            const bgw::DzPlanes bt = bgw::dz_planes(w + o.t, ng, kB, nfreq, true);
            const bgw::DzOperand ot = {T, (long)ng * kB, kB, 1, false, nullptr};
            if (e == cudaSuccess) e = bgw::dz_split(&ot, &bt, 1, kb, st);
            if (e == cudaSuccess)
                e = bgw::dz_gemm(pa, bt, bgw::DzOut{A, n2, ng, 1, k0, k0 + kb, -1.0, 0.0, true}, sms, st, err + 1);
            if (e != cudaSuccess) break;
            k6_writeback_t<<<dim3((ng + 31) / 32, 1, nfreq), 256, 0, st>>>(A, ng, k0, kb, T, U);
        } else {
            k6_panels<<<dim3((ng + 127) / 128, kB / kPanelI, 2 * nfreq), 128, 0, st>>>(A, ng, k0, kb, T, U);
            k6_update<<<dim3(tiles, tiles, nfreq), 256, kUpdateSmem, st>>>(A, ng, k0, kb, T);
            k6_writeback<<<dim3((ng + 127) / 128, 1, nfreq), 128, 0, st>>>(A, ng, k0, kb, T, U);
        }
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && mode > 0) {
        k6_scale<<<dim3(rowblocks, ng, nfreq), 256, 0, st>>>(A, sx, sox, stride, ng, mode == 2);
        e = cudaGetLastError();
    } else if (e == cudaSuccess && tensor) {
        k6_unbalance<<<dim3(rowblocks, ng, nfreq), 256, 0, st>>>(A, ex, ng);
        e = cudaGetLastError();
    }
    int flag[2] = {0, 0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(flag, err, sizeof flag, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (own) cudaFree(own);
    if (e != cudaSuccess) return fail(BGW_E_CUDA, std::string("epsinv: ") + cudaGetErrorString(e));
    if (flag[1]) return fail(BGW_E_TIMEOUT, "epsinv: a device-side wait gave up; the output is invalid");
    if (flag[0]) return fail(BGW_E_ARG, "epsinv: a pivot is not positive: I - S chi S is not positive definite "
                                     "(chi0 must be Hermitian negative semidefinite); the output is invalid");
    return BGW_OK;
}
