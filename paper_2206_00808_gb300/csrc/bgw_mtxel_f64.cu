// FP64 instantiation of the matrix-element kernels.
#define BGW_REAL double
#define BGW_SUFFIX f64
#define BGW_GRID_PART 2
#include "bgw_grid_impl.cuh"

namespace bgw {
cudaError_t mtxel_tables_init_f64() { return f64::upload_tables(); }
cudaError_t mtxel_f64(const void *Uv, const void *Uc, int nv, int nc, const Axes &a, const int *gmap, int ng, void *A,
                      void *Bs, void *M, long ldm, cudaStream_t st, int lanes, const XPassHook *hook, const int *sv,
                      const int *sc) {
    return f64::mtxel(Uv, Uc, nv, nc, a, gmap, ng, A, Bs, M, ldm, st, 0, 0, lanes, 0, hook, nullptr, 0, sv, sc);
}
cudaError_t bounds_take_mtxel_f64(unsigned *word) { return bgw_bounds_take(word); }
}  // namespace bgw
