// Ragged batches: members of BF16 population storage.
#include "lbm_batch.cuh"

namespace lbm {

cudaError_t launch_batch_bf16(const BatchPart& p, cudaStream_t st) { return launch_batch_st<ST_BF16>(p, st); }

}  // namespace lbm
