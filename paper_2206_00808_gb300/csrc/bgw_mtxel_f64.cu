// FP64 instantiation of the matrix-element kernels.
#define BGW_REAL double
#define BGW_SUFFIX f64
#define BGW_GRID_PART 2
#include "bgw_grid_impl.cuh"

namespace bgw {
cudaError_t mtxel_tables_init_f64() {
    const cudaError_t e = f64::upload_tables();
    return e == cudaSuccess ? zy_fix_tables_init() : e;
}
cudaError_t mtxel_f64(const void *Uv, const void *Uc, int nv, int nc, const Axes &a,
                      const int *gmap, int ng, void *A, void *Bs, void *M, long ldm,
                      cudaStream_t st, int tv, int tc, int lanes, int zy, const XPassHook *hook, int *err,
                      int drop) {
    return f64::mtxel(Uv, Uc, nv, nc, a, gmap, ng, A, Bs, M, ldm, st, tv, tc, lanes, zy, hook, err, drop);
}
cudaError_t bounds_take_mtxel_f64(unsigned *word) { return bgw_bounds_take(word); }
}  // namespace bgw
