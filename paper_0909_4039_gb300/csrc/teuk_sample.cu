// teuk_sample.cu -- waveform samples: of the extraction rows the step kernels
// leave (k_sample_steps), and of a caller's state (k_sample).  A file of its
// own: the first launch of a kernel loads its module, and together with the
// adjoint kernels' that took a process's first step 30 ms.
#include "teuk_adjoint.cuh"

namespace teuk {
namespace {

// The physical row u = C_{dt/2} s of the extraction row s (planes f, g), in
// shared memory: all threads load, warp 0 solves (the row is warp 0's).
template <typename T, int S>
__device__ __forceinline__ const typename V2<T>::t *physical_row(const StepParams<T> &p, const typename V2<T>::t *f,
                                                                 const typename V2<T>::t *g)
{
    typedef typename V2<T>::t c2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = p.Nth, Nr = p.Nr, i = p.i_ext, tid = threadIdx.x, NT = blockDim.x;
    c2 *xPhi = (c2 *)smem_raw;
    c2 *xPi = xPhi + ((N + 1) & ~1);
    T *xF = (T *)(xPi + ((N + 1) & ~1));
    unsigned long long *xTh2 = (unsigned long long *)(xF + NSF);
    T *xTh = (T *)(xTh2 + pair_th_bytes(N, (int)sizeof(T)) / 8);
    if constexpr (kPaired<T, S>) pair_th_fill(xTh2, p.thtab, N, tid, NT);
    for (int j = tid; j < N; j += NT) {
        xPhi[j] = f[j];
        xPi[j] = g[j];
    }
    if (tid >= NT - 32 && tid - (NT - 32) < NSF) xF[tid - (NT - 32)] = p.stab[(size_t)(2 * i) * NSF + tid - (NT - 32)];
    for (int k = tid; k < NTF * N; k += NT) xTh[k] = p.thtab[k];
    __syncthreads();
    if (tid >= 32) return xPhi;
    const int G = p.group;
    const bool mine = tid < G;
    const bool active = mine && i >= 1 && i <= Nr - 2;
    implicit_row_one<T, S>(p.half, xPhi, xPi, i, xF, xTh, xTh2, N, active, mine, tid % G, G, p.vec != 0, p.half.plan[i]);
    __syncwarp();
    return xPhi;
}

// h = E s (physical) or E C_{dt/2} s of the extraction row of s, as the step
// kernels form it (see seed_dot).
template <typename T, int S>
__global__ void __launch_bounds__(32) k_sample(const StepParams<T> p, const typename V2<T>::t *s, int physical,
                                               double2 *h_out)
{
    const size_t o = (size_t)p.i_ext * p.Nth;
    const typename V2<T>::t *f = s + o, *g = f + (size_t)p.Nr * p.Nth;
    double2 h;
    if (physical) {
        h = sample_warp<T>(p, f);
    } else if constexpr (sizeof(T) == 8) {
        h = seed_dot<T>(p, f, g);
    } else {
        h = sample_warp<T>(p, physical_row<T, S>(p, f, g));
    }
    if (threadIdx.x == 0) *h_out = h;
}

// Threads of a sampling CTA: one warp has the row to solve, and four load its
// tables (7 Ntheta entries one after the other held a lone warp for 10 of the
// 22 us that a launch of 64 x 16 rows of 128 took).
// (One CTA per SM is asked for: without that, the compiler gave the kernels of 32
// elements a lane 32 registers and spilled the row; 1500 x 300 in calls of one
// step, us per call with and without: FP64 410 and 540, four FP32 instances 237
// and 287.)
constexpr int kSampleThreads = 128;

// CTA (b, instance): the b-th step after ctl->sampled, if it has been taken.
// The last CTA of an instance moves ctl->sampled on.
template <typename T, int S>
__device__ __forceinline__ void sample_step(const StepParams<T> &p)
{
    const long long n0 = *((volatile long long *)&p.ctl->sampled), n1 = *((volatile long long *)&p.ctl->step);
    const long long n = n0 + 1 + blockIdx.x;
    // (only the last wave_cap samples stay in the ring: two steps of one slot do not race)
    if (n <= n1 && n > n1 - p.wave_cap) {
        const typename V2<T>::t *r = p.raw + (size_t)(n % kRawSlots) * 2 * p.Nth;
        const typename V2<T>::t *row = physical_row<T, S>(p, r, r + p.Nth);
        if (threadIdx.x < 32) extract_warp<T>(p, row, n);
    }
    __syncthreads();   // (all threads have read the counters)
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&p.ctl->sticket, 1u) == gridDim.x - 1u) {
            p.ctl->sticket = 0u;
            p.ctl->sampled = n1;
        }
    }
}

template <typename T, int S>
__global__ void __launch_bounds__(kSampleThreads, 1) k_sample_steps(const StepParams<T> p)
{
    launch_turn();
    sample_step<T, S>(p);
}

template <typename T, int S>
__global__ void __launch_bounds__(kSampleThreads, 1) k_sample_steps_batch(const StepParams<T> *params)
{
    launch_turn();
    __shared__ __align__(16) StepParams<T> sp;
    for (int k = threadIdx.x; k < (int)(sizeof(StepParams<T>) / 4); k += kSampleThreads)
        reinterpret_cast<int *>(&sp)[k] = reinterpret_cast<const int *>(params + blockIdx.y)[k];
    __syncthreads();
    sample_step<T, S>(sp);
}

}  // namespace

template <typename T>
cudaError_t launch_sample(const StepParams<T> &p, const typename V2<T>::t *s, int physical, double2 *h_out,
                          cudaStream_t st)
{
    const int seg = implicit_seg(p.Nth);
    auto fn = seg == kSegNarrow ? k_sample<T, kSegNarrow> : (seg == kSeg ? k_sample<T, kSeg> : k_sample<T, kSegWide>);
    cudaError_t e = smem_limit_max((const void *)fn);
    if (e != cudaSuccess) return e;
    fn<<<1, 32, sample_smem_bytes<T>(p.Nth), st>>>(p, s, physical, h_out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_sample_steps(const StepParams<T> &p, int pending, cudaStream_t st)
{
    if (pending < 1 || pending > kRawSlots) return cudaErrorInvalidValue;
    const int seg = implicit_seg(p.Nth);
    auto fn = seg == kSegNarrow ? k_sample_steps<T, kSegNarrow>
                                : (seg == kSeg ? k_sample_steps<T, kSeg> : k_sample_steps<T, kSegWide>);
    cudaError_t e = smem_limit_max((const void *)fn);
    if (e != cudaSuccess) return e;
    return launch_dep(fn, dim3((unsigned)pending), kSampleThreads, sample_smem_bytes<T>(p.Nth), st, p);
}

template <typename T>
cudaError_t launch_sample_steps_batch(const StepParams<T> *d_params, int count, int Nmax, int pending, cudaStream_t st)
{
    if (pending < 1 || pending > kRawSlots) return cudaErrorInvalidValue;
    const int seg = implicit_seg(Nmax);
    auto fn = seg == kSegNarrow ? k_sample_steps_batch<T, kSegNarrow>
                                : (seg == kSeg ? k_sample_steps_batch<T, kSeg> : k_sample_steps_batch<T, kSegWide>);
    cudaError_t e = smem_limit_max((const void *)fn);
    if (e != cudaSuccess) return e;
    return launch_dep(fn, dim3((unsigned)pending, (unsigned)count), kSampleThreads, sample_smem_bytes<T>(Nmax), st, d_params);
}

template cudaError_t launch_sample<float>(const StepParams<float> &, const float2 *, int, double2 *, cudaStream_t);
template cudaError_t launch_sample<double>(const StepParams<double> &, const double2 *, int, double2 *, cudaStream_t);
template cudaError_t launch_sample_steps<float>(const StepParams<float> &, int, cudaStream_t);
template cudaError_t launch_sample_steps<double>(const StepParams<double> &, int, cudaStream_t);
template cudaError_t launch_sample_steps_batch<float>(const StepParams<float> *, int, int, int, cudaStream_t);
template cudaError_t launch_sample_steps_batch<double>(const StepParams<double> *, int, int, int, cudaStream_t);

}  // namespace teuk
