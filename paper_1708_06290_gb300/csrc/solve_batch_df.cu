// Double-float instances of the many-systems launch.
#include "batch.cuh"

namespace ssv {

int batch_config_df(BatchPlan* bp) { return batch_config_any<true>(bp); }
void batch_launch_df(const BatchPlan* bp, cudaStream_t st) { batch_launch_any<true>(bp, st); }

}  // namespace ssv
