// level_f32.cu -- the level kernels for FP32 populations.
#include "level.cuh"

namespace lbmdev {

template void launch_level_store<float>(cudaStream_t, const LevelView &, const LevelView &, const LevelView &, bool,
                                     const RecView &, const StepConsts &, const LevelStep &, const LevelTune &);
template void launch_level_batch_store<float>(cudaStream_t, const BatchArgs &, unsigned, int);

}  // namespace lbmdev
