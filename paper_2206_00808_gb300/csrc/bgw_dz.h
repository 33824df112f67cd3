// FP64-accurate complex products on tcgen05 tensor cores from BF16 digit
// slices (bgw_dz.cu): C(b, m, n) = [C +] alpha sum_k A(b, m, k) w_k B(b, n, k).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace bgw {

// Operand (b, row, k) at p[b * sb + row * sr + k * sk], complex128; w: a real
// weight per k (may be null).
struct DzOperand {
    const double2 *p;
    long sb, sr, sk;
    bool conj;
    const double *w;
};

// Digit planes of one operand for `batch` matrices of `rows` rows: an A
// operand has one real row per row, a B operand two.
struct DzPlanes {
    void *x;          // BF16 digits
    int *scale;       // exponent of each (batch, row)
    int rows, rows_pad, kblocks;
    int batch;        // matrices the planes hold
    int first, used;  // matrices a split writes or a product reads: first .. first + used - 1
    bool b;           // B operand
};

struct DzOut {
    double2 *c;
    long sb, sm, sn;
    int skip0, skip1;        // rows and columns in [skip0, skip1) are left alone
    double ar, ai;           // alpha
    bool accumulate;
};

// Shared k range of a product; the sums stay exact up to this K.
constexpr int kDzMaxK = 5000;

size_t dz_planes_bytes(int rows, int K, int batch, bool b);
// Describe planes of `rows` x K in ws (dz_planes_bytes long).
DzPlanes dz_planes(void *ws, int rows, int K, int batch, bool b);
// Cut n operands into their digits, one launch (all of the same K).
cudaError_t dz_split(const DzOperand *op, const DzPlanes *pl, int n, int K, cudaStream_t st);
// err: device int, set non-zero when a bounded device wait gave up (the outputs
// that the block had still to write are then NaN).  drop: test hook, block 0
// never issues its first loads.
cudaError_t dz_gemm(const DzPlanes &A, const DzPlanes &B, const DzOut &out, int sm_count, cudaStream_t st, int *err,
                    bool drop = false);

}  // namespace bgw
