// bte_sweep_fp32.cu -- sweep kernel instances for FP32 intensity storage.
#include "bte_rows.cuh"

namespace bte {

cudaError_t launch_sweep_fp32(const SweepArgs& a, int dim, int threads, int grid, cudaStream_t s) {
  if (a.explicit_scheme) return rows::launch<rows::F32<true>>(a, dim, threads, grid, s);
  return rows::launch<rows::F32<false>>(a, dim, threads, grid, s);
}

}  // namespace bte
