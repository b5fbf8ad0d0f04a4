// bte_sweep_fp64.cu -- sweep kernel instances for FP64 intensity storage.
#include "bte_rows.cuh"

namespace bte {

cudaError_t launch_sweep_fp64(const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s) {
  if (a.ff) return rows::launch<rows::FF>(a, dim, threads, grid, s);  // double-float arithmetic
  if (a.beta_exp != 0.0) {
    if (a.bmode == 1) return rows::launch<rows::F64<1, true>>(a, dim, threads, grid, s);
    if (a.bmode == 2) return rows::launch<rows::F64<2, true>>(a, dim, threads, grid, s);
    return rows::launch<rows::F64<0, true>>(a, dim, threads, grid, s);
  }
  if (a.bmode == 1) return rows::launch<rows::F64<1, false>>(a, dim, threads, grid, s);
  if (a.bmode == 2) return rows::launch<rows::F64<2, false>>(a, dim, threads, grid, s);
  return rows::launch<rows::F64<0, false>>(a, dim, threads, grid, s);
}

}  // namespace bte
