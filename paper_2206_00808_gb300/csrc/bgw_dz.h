// FP64-accurate complex products on tcgen05 tensor cores from BF16 digit
// slices (bgw_dz.cu): C(b, m, n) = [C +] alpha sum_k A(b, m, k) w_k B(b, n, k).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace bgw {

// Operand (b, row, k) at p[b * sb + row * sr + k * sk], complex128; w: a real
// weight per k (may be null); cols, other: column exponents of this operand and
// of the other of its product, from dz_balance (null: none).
struct DzOperand {
    const double2 *p;
    long sb, sr, sk;
    bool conj;
    const double *w;
    const int *cols = nullptr, *other = nullptr;
    bool second = false;     // the B operand: takes the opposite shift
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
// Column exponents of the operands of one product (batch 1, k contiguous): the
// largest exponent of each column over the rows, each taken relative to its row's
// largest entry.  ws: dz_balance_bytes long.  Sets cols, other and second of both,
// and *err = 0.
size_t dz_balance_bytes(int K);
cudaError_t dz_balance(DzOperand &A, long rowsA, DzOperand &B, long rowsB, int K, void *ws, int *err, cudaStream_t st);
// Cut n operands into their digits, one launch (all of the same K).
cudaError_t dz_split(const DzOperand *op, const DzPlanes *pl, int n, int K, cudaStream_t st);
// err: device int, set non-zero when a bounded device wait gave up (the outputs
// that the block had still to write are then NaN).  drop: test hook, block 0
// never issues its first loads.
cudaError_t dz_gemm(const DzPlanes &A, const DzPlanes &B, const DzOut &out, int sm_count, cudaStream_t st, int *err,
                    bool drop = false);

}  // namespace bgw
