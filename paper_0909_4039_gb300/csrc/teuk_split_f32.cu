// teuk_split_f32.cu -- the split-scheme step kernels of lone states and their launchers, FP32 state.
// (Batched and pipelined kernels have files of their own: one file of them all
// compiled for three minutes.)
#include "teuk_split.cuh"

namespace teuk {

template cudaError_t launch_apply_step<float>(const StepParams<float> &, int, size_t, cudaStream_t);
template cudaError_t launch_scan_plans<float>(const StepParams<float> &, int *, int *, float2 *, float2 *,
                                               cudaStream_t);
template size_t split2_smem_bytes<float>(int, int);
template int split2_blocks_per_sm<float>(int, int, int, size_t);
template cudaError_t launch_split_step2<float>(const StepParams<float> &, int, size_t, cudaStream_t);
template size_t split3_smem_bytes<float>(int, int);
template int split3_blocks_per_sm<float>(int, int, int, size_t);
template cudaError_t launch_split_step3<float>(const StepParams<float> &, int, size_t, cudaStream_t);
template int split_blocks_per_sm<float>(int, int, int, size_t);
template size_t split_smem_bytes<float>(int, int);
template cudaError_t launch_split_step<float>(const StepParams<float> &, int, size_t, cudaStream_t);


}  // namespace teuk
