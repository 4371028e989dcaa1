// Row march: the moment pass of every storage.
#include "lbm_rows.cuh"

namespace lbm {

cudaError_t launch_moments(const Phys2& P, const Grid& g, const MomentOut& mo, cudaStream_t st) {
  if (g.march_nt != MARCH_NT) return launch_moments_narrow(P, g, mo, st);
  switch (g.storage) {
    case ST_FP32: return launch_rows_nt<MODE_MOMENTS, ST_FP32, MARCH_NT>(P, g, mo, st);
    case ST_FP16: return launch_rows_nt<MODE_MOMENTS, ST_FP16, MARCH_NT>(P, g, mo, st);
    case ST_BF16: return launch_rows_nt<MODE_MOMENTS, ST_BF16, MARCH_NT>(P, g, mo, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbm
