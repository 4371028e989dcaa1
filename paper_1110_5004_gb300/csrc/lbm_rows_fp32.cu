// Row march, FP32 population storage: the time step.
#include "lbm_rows.cuh"

namespace lbm {

cudaError_t launch_step_fp32(const Phys2& P, const Grid& g, cudaStream_t st) {
  return launch_rows_st<MODE_STEP, ST_FP32>(P, g, MomentOut{}, st);
}

}  // namespace lbm
