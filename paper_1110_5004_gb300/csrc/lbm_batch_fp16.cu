// Ragged batches: members of FP16 population storage.
#include "lbm_batch.cuh"

namespace lbm {

cudaError_t launch_batch_fp16(const BatchPart& p, cudaStream_t st) { return launch_batch_st<ST_FP16>(p, st); }

}  // namespace lbm
