// Row march, BF16 population storage: the time step.
#include "lbm_rows.cuh"

namespace lbm {

cudaError_t launch_step_bf16(const Phys2& P, const Grid& g, cudaStream_t st) {
  return g.march_nt == MARCH_NT ? launch_rows_nt<MODE_STEP, ST_BF16, MARCH_NT>(P, g, MomentOut{}, st) : launch_narrow_bf16(P, g, st);
}

}  // namespace lbm
