// teuk_pipe_f32.cu -- the pipelined split-scheme kernels and their launchers, FP32 state.
#include "teuk_split.cuh"

namespace teuk {

template size_t pipe_smem_bytes<float>(int, int);
template int pipe_blocks_per_sm<float>(int, int, size_t);
template cudaError_t launch_split_pipe<float>(const StepParams<float> &, int, int, size_t, cudaStream_t);

}  // namespace teuk
