// teuk_pipe_f64.cu -- the pipelined split-scheme kernels and their launchers, FP64 state.
#include "teuk_split.cuh"

namespace teuk {

template size_t pipe_smem_bytes<double>(int, int);
template int pipe_blocks_per_sm<double>(int, int, size_t);
template cudaError_t launch_split_pipe<double>(const StepParams<double> &, int, int, size_t, cudaStream_t);

}  // namespace teuk
