// Row march: the moment pass of every storage in CTAs of 64 and 32 threads (narrow grids).
#include "lbm_rows.cuh"

namespace lbm {

cudaError_t launch_moments_narrow(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st) {
  switch (g.storage) {
    case ST_FP32: return launch_rows_narrow<MODE_MOMENTS, ST_FP32>(P, g, mo, st);
    case ST_FP16: return launch_rows_narrow<MODE_MOMENTS, ST_FP16>(P, g, mo, st);
    case ST_BF16: return launch_rows_narrow<MODE_MOMENTS, ST_BF16>(P, g, mo, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbm
