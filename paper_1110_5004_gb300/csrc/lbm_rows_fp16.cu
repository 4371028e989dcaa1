// Row march, FP16 population storage: the time step.
#include "lbm_rows.cuh"

namespace lbm {

cudaError_t launch_step_fp16(const Phys2& P, const Grid& g, cudaStream_t st) {
  return launch_rows_st<MODE_STEP, ST_FP16>(P, g, MomentOut{}, st);
}

}  // namespace lbm
