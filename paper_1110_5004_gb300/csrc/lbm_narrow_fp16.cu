// Row march, FP16 population storage: the time step in CTAs of 64 and 32 threads (narrow grids).
#include "lbm_rows.cuh"

namespace lbm {

cudaError_t launch_narrow_fp16(const Phys2& P, const Grid& g, cudaStream_t st) {
  return launch_rows_narrow<MODE_STEP, ST_FP16>(P, g, MomentOut{}, st);
}

}  // namespace lbm
