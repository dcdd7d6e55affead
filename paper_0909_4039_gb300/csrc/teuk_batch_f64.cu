// teuk_batch_f64.cu -- the batched split-scheme step kernels and their launchers, FP64 state.
#include "teuk_split.cuh"

namespace teuk {

template int split_batch_blocks_per_sm<double>(int, size_t, int);
template cudaError_t launch_split_batch<double>(const StepParams<double> *, const int2 *, int, int, size_t, int,
                                                bool, cudaStream_t);

}  // namespace teuk
