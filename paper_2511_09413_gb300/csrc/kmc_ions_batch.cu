// kmc_ions_batch.cu -- persistent launches of the ion-list tile (kmc_ions.cuh) over a
// batch's devices.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "kmc_ions.cuh"

namespace kmc {

namespace {

// The batch's persistent launch of one shape (as sweep_batch_kernel).
template <int P, bool ACC, bool OPEN, class M>
__global__ void __launch_bounds__(256, 4) ion_batch_kernel(const __grid_constant__ BatchArgs b, int kind)
{
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ SweepArgs ia;
    __shared__ int s_item;
    const int64_t t0 = *b.t0;
    const int first = b.cls_off[kind], end = b.cls_off[kind + 1];
    for (;;) {
        if (threadIdx.x == 0) s_item = first + (int)atomicAdd(b.work + kind, 1u);
        __syncthreads();
        const int item = s_item;
        if (item >= end) break;
        const BatchItem it = b.items[item];
        const uint32_t *src = (const uint32_t *)&b.inst[it.inst];
        for (int i = threadIdx.x; i < (int)(sizeof(SweepArgs) / 4); i += blockDim.x)
            ((uint32_t *)&ia)[i] = src[i];
        __syncthreads();
        ion_tile<P, ACC, OPEN, M>(ia, b.rk0, b.rk1, t0, b.n_steps, b.flush, it.tile_rail0, smem);
        __syncthreads();
    }
}

}  // namespace

cudaError_t ion_batch_launch(const BatchArgs &b, int kind, int grid, int warps, size_t smem, bool acc,
                             cudaStream_t s)
{
    return with_ions(kind, acc, [&](auto p, auto ac, auto open, auto m) {
        ion_batch_kernel<decltype(p)::value, decltype(ac)::value, decltype(open)::value, decltype(m)>
            <<<grid, warps * 32, smem, s>>>(b, kind);
        return cudaGetLastError();
    });
}

int ion_batch_ctas_per_sm(int kind, int mode, int warps, size_t smem)
{
    if (mode == 2) return ion_grad_ctas_per_sm(kind, warps, smem);
    int n = 0;
    const cudaError_t e = with_ions(kind, mode == 1, [&](auto p, auto ac, auto open, auto m) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, ion_batch_kernel<decltype(p)::value, decltype(ac)::value, decltype(open)::value, decltype(m)>,
            warps * 32, smem);
    });
    return e == cudaSuccess && n > 0 ? n : 1;
}

cudaError_t ion_batch_set_smem_limits()
{
    cudaError_t e = cudaSuccess;
    for (int k = kWordKinds; k < kShapeKinds; ++k)
        for (int acc = 0; acc < 2; ++acc) {
            const cudaError_t r = with_ions(k, acc != 0, [](auto p, auto ac, auto open, auto m) {
                return cudaFuncSetAttribute(
                    ion_batch_kernel<decltype(p)::value, decltype(ac)::value, decltype(open)::value, decltype(m)>,
                    cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
            });
            if (r != cudaSuccess) e = r;
        }
    return e;
}

}  // namespace kmc
