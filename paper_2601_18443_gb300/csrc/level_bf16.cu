// level_bf16.cu -- the level kernels for BF16 populations.
#include "level.cuh"

namespace lbmdev {

template void launch_level_store<__nv_bfloat16>(cudaStream_t, const LevelView &, const LevelView &, const LevelView &, bool,
                                     const RecView &, const StepConsts &, const LevelStep &, const LevelTune &);
template void launch_level_batch_store<__nv_bfloat16>(cudaStream_t, const BatchArgs &, unsigned, int);

}  // namespace lbmdev
