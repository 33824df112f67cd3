// FP64 instantiation of the sphere -> grid kernels (the matrix elements are
// in bgw_mtxel_f64.cu).
#define BGW_REAL double
#define BGW_SUFFIX f64
#define BGW_GRID_PART 1
#include "bgw_grid_impl.cuh"

namespace bgw {
cudaError_t mtxel_tables_init_f64();
cudaError_t bounds_take_mtxel_f64(unsigned *word);

cudaError_t grid_tables_init_f64() {
    cudaError_t e = f64::upload_tables();
    if (e == cudaSuccess) e = mtxel_tables_init_f64();
    if (e == cudaSuccess) e = grid_fix_tables_init();
    return e == cudaSuccess ? zy_fix_tables_init() : e;
}
cudaError_t wfn_xpass_f64(const double *coeff, int ngw, int B, const int *cube_map, const Axes &a, void *S,
                          cudaStream_t st) {
    return f64::wfn_xpass(reinterpret_cast<const double2 *>(coeff), ngw, B, cube_map, a, static_cast<f64::C *>(S), st);
}
cudaError_t wfn_to_grid_f64(const double *coeff, int ngw, int B, const int *cube_map,
                            const Axes &a, void *S, void *R, void *U, cudaStream_t st, int path) {
    return f64::wfn_to_grid(coeff, ngw, B, cube_map, a, S, R, U, st, path);
}
cudaError_t wfn_xpass_batch_f64(const K1Job *jobs, int n, int B, cudaStream_t st) {
    return f64::wfn_xpass_batch(jobs, n, B, st);
}
cudaError_t bounds_take_grid_f64(unsigned *word) {
    unsigned a = 0, b = 0;
    cudaError_t e = bgw_bounds_take(&a);
    if (e == cudaSuccess) e = bounds_take_mtxel_f64(&b);
    *word = a | b;
    return e;
}
}  // namespace bgw
