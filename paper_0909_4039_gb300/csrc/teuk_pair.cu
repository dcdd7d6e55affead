// teuk_pair.cu -- launchers of the FP32 step kernels on packed pairs.
#include "teuk_pair_tile.cuh"


namespace teuk {

bool pair_eligible(int Nth) { return Nth > 128 && Nth <= 256 && Nth % 4 == 0; }

bool pair_runs(int tile_rows, int Nth, int ks)
{
    // the limit of a block, less the batched kernel's static part (1.7 KB)
    return pair_eligible(Nth) && pair_smem_bytes(tile_rows, Nth, ks) <= 225 * 1024;
}

size_t pair_smem_bytes(int tile_rows, int Nth, int ks) { return pair_smem_plan(tile_rows + 2 * ks, Nth).total; }

static void (*pair_fn(int ks))(const StepParams<float>)
{
    return ks == 1 ? k_pair_step<1> : (ks == 2 ? k_pair_step<2> : k_pair_step<3>);
}
static void (*pair_batch_fn(int ks))(const StepParams<float> *, const int2 *)
{
    return ks == 1 ? k_pair_batch<1> : k_pair_batch<2>;
}

static int blocks_per_sm(const void *fn, size_t smem)
{
    int nb = 0;
    if (smem_limit_max(fn) != cudaSuccess || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, 256, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

int pair_blocks_per_sm(int ks, size_t smem) { return blocks_per_sm((const void *)pair_fn(ks), smem); }
int pair_batch_blocks_per_sm(int ks, size_t smem) { return blocks_per_sm((const void *)pair_batch_fn(ks), smem); }

cudaError_t launch_pair_step(const StepParams<float> &p, int ks, cudaStream_t st)
{
    if (p.first || p.imp_only || p.nfix >= 0 || !pair_runs(p.tile_rows, p.Nth, ks)) return cudaErrorInvalidValue;
    auto fn = p.own && ks == 1 ? k_pair_step<1, true> : pair_fn(ks);
    cudaError_t e = smem_limit_max((const void *)fn);
    if (e != cudaSuccess) return e;
    return launch_dep(fn, dim3((unsigned)((p.Nr + p.tile_rows - 1) / p.tile_rows)), 256,
                      pair_smem_bytes(p.tile_rows, p.Nth, ks), st, p);
}

cudaError_t launch_pair_batch(const StepParams<float> *d_params, const int2 *d_tiles, int ntiles, size_t smem, int ks,
                              cudaStream_t st)
{
    auto fn = pair_batch_fn(ks);
    cudaError_t e = smem_limit_max((const void *)fn);
    if (e != cudaSuccess) return e;
    if (ntiles < 1) return cudaSuccess;
    return launch_dep(fn, dim3((unsigned)ntiles), 256, smem, st, d_params, d_tiles);
}

}  // namespace teuk
