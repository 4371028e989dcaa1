// Ragged batches: members of BF16 population storage.
#include "lbm_batch.cuh"

namespace lbm {

cudaError_t launch_batch_bf16(const SimDesc* sims, const int4* work, int n, int grid, int parity, unsigned int* next, bool sd, bool xw,
                              cudaStream_t st) {
  return launch_batch_st<ST_BF16>(sims, work, n, grid, parity, next, sd, xw, st);
}

}  // namespace lbm
