// teuk_batch_f32.cu -- the batched split-scheme step kernels and their launchers, FP32 state.
#include "teuk_split.cuh"

namespace teuk {

template int split_batch_blocks_per_sm<float>(int, size_t, int);
template cudaError_t launch_split_batch<float>(const StepParams<float> *, const int2 *, int, int, size_t, int,
                                               bool, cudaStream_t);

}  // namespace teuk
