// Ragged batches: members of FP32 population storage.
#include "lbm_batch.cuh"

namespace lbm {

cudaError_t launch_batch_fp32(const SimDesc* sims, const int4* work, int n, int grid, int parity, unsigned int* next, bool sd, bool xw,
                              cudaStream_t st) {
  return launch_batch_st<ST_FP32>(sims, work, n, grid, parity, next, sd, xw, st);
}

}  // namespace lbm
