// level_f16.cu -- the level kernels for FP16 populations.
#include "level.cuh"

namespace lbmdev {

template void launch_level_store<__half>(cudaStream_t, const LevelView &, const LevelView &, const LevelView &, bool,
                                     const RecView &, const StepConsts &, const LevelStep &, const LevelTune &);
template void launch_level_batch_store<__half>(cudaStream_t, const BatchArgs &, unsigned, int);

}  // namespace lbmdev
