// step_multi.cu -- the step kernel over several independent networks in one
// launch (a batch whose partitions all fit on the GPU at once; batch.cu).
//
// Each network has its own partitions, messages and rasters, and its CTAs wait
// only for one another: there is no barrier over the batch.  A step takes what
// it takes the largest of the networks alone, where the batch kernel's step
// costs a grid barrier and four dependent trips to L2 (5 networks of 13,072
// neurons: 6.59 us per step, here 1.57; 12 of 70,900: 8.6 and 1.80; 16 of
// 187,168, four neurons per thread: 9.9 and 4.8).
#include "step_kernel.cuh"

namespace snn {
namespace {

template <int NPT, bool SMEM_RING, int INL, int T = kStepThreads>
__global__ void __launch_bounds__(T, 1)
k_step_multi(const StepParams* __restrict__ params, const int32_t* __restrict__ first, int n_net,
             const long long* step, int n_steps) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ StepParams s_sp;
    int a = 0, b = n_net;                       // first[a] <= blockIdx.x < first[b]
    while (b - a > 1) {
        const int m = (a + b) >> 1;
        if (__ldg(&first[m]) <= (int)blockIdx.x) a = m;
        else b = m;
    }
    static_assert(sizeof(StepParams) % 4 == 0, "copied by words");
    const uint32_t* src = reinterpret_cast<const uint32_t*>(params + a);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&s_sp);
    for (uint32_t k = threadIdx.x; k < sizeof(StepParams) / 4; k += T) dst[k] = __ldg(&src[k]);
    __syncthreads();
    if (threadIdx.x == 0) {
        s_sp.t0 = *step;
        s_sp.n_steps = n_steps;
    }
    __syncthreads();
    step_body<NPT, SMEM_RING, 0, INL, true, T>(s_sp, (int)blockIdx.x - __ldg(&first[a]), smem);
}

// after the launch, when every CTA has read it
__global__ void k_advance(long long* step, int n_steps) { *step += n_steps; }

const void* multi_fn(int npt, bool smem_ring, bool few, int threads) {
    if (few && npt == 1 && smem_ring) {
        switch (threads) {
            case 192: return reinterpret_cast<const void*>(&k_step_multi<1, true, kInlineFew, 192>);
            case 256: return reinterpret_cast<const void*>(&k_step_multi<1, true, kInlineFew, 256>);
            case 352: return reinterpret_cast<const void*>(&k_step_multi<1, true, kInlineFew, 352>);
            default: return reinterpret_cast<const void*>(&k_step_multi<1, true, kInlineFew>);
        }
    }
    switch (npt) {
        case 1: return smem_ring ? reinterpret_cast<const void*>(&k_step_multi<1, true, kInline>) : nullptr;
        case 2: return smem_ring ? reinterpret_cast<const void*>(&k_step_multi<2, true, kInline>)
                                 : reinterpret_cast<const void*>(&k_step_multi<2, false, kInline>);
        case 4: return smem_ring ? nullptr : reinterpret_cast<const void*>(&k_step_multi<4, false, kInline>);
        case 8: return smem_ring ? nullptr : reinterpret_cast<const void*>(&k_step_multi<8, false, kInline>);
        default: return nullptr;
    }
}

}  // namespace

cudaError_t step_multi_configure(int npt, bool smem_ring, bool few, int threads, size_t smem, int* blocks_per_sm) {
    const void* fn = multi_fn(npt, smem_ring, few, threads);
    if (!fn) return cudaErrorInvalidValue;
    const cudaError_t e = allow_shared(fn);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, threads, smem);
}

cudaError_t launch_step_multi(int npt, bool smem_ring, bool few, int threads, size_t smem, int grid, const StepParams* params,
                              const int32_t* first, int n_net, long long* step, int n_steps, cudaStream_t s) {
    const void* fn = multi_fn(npt, smem_ring, few, threads);
    if (!fn) return cudaErrorInvalidValue;
    void* args[] = {&params, &first, &n_net, &step, &n_steps};
    const cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(threads), args, smem, s);
    if (e != cudaSuccess) return e;
    k_advance<<<1, 1, 0, s>>>(step, n_steps);
    return cudaGetLastError();
}

}  // namespace snn
