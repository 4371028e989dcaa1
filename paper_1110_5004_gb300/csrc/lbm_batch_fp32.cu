// Ragged batches: members of FP32 population storage.
#include "lbm_batch.cuh"

namespace lbm {

cudaError_t launch_batch_fp32(const BatchPart& p, cudaStream_t st) { return launch_batch_st<ST_FP32>(p, st); }

}  // namespace lbm
