// Row march, BF16 population storage: the time step.
#include "lbm_rows.cuh"

namespace lbm {

cudaError_t launch_step_bf16(const Phys2& P, const Grid& g, cudaStream_t st) {
  return launch_rows_st<MODE_STEP, ST_BF16>(P, g, MomentOut{}, st);
}

}  // namespace lbm
