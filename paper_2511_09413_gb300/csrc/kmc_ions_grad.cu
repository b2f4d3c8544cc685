// kmc_ions_grad.cu -- gradient passes on the ion-list tile (kmc_ions.cuh).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "kmc_ions.cuh"

namespace kmc {

namespace {

// Gradient passes (as sweep_grad_kernel and sweep_batch_grad_kernel), 64 rows of
// bits.  Shared memory, not registers, limits the warps of an SM (on 4 lanes per
// rail, 8 rails' lists, bounds and score factors are about 13 KB a warp), so a CTA
// has up to 20 warps of 96 registers.
template <int P, bool OPEN>
__global__ void __launch_bounds__(32 * kGradWarps, 1) ion_grad_kernel(const __grid_constant__ SweepArgs a)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const int64_t tile_rail0 = (int64_t)blockIdx.x * (blockDim.x >> 5) * (32 / P);
    ion_tile<P, true, OPEN, uint64_t, true>(a, a.rk0, a.rk1, a.t0, a.n_steps, a.n_steps, tile_rail0, smem);
}
template <int P, bool OPEN>
__global__ void __launch_bounds__(32 * kGradWarps, 1) ion_batch_grad_kernel(const __grid_constant__ BatchArgs b, int kind)
{
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ SweepArgs ia;
    __shared__ int s_item;
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
        ion_tile<P, true, OPEN, uint64_t, true>(ia, b.rk0, b.rk1, 0, ia.n_steps, ia.n_steps, it.tile_rail0, smem);
        __syncthreads();
    }
}

// Calls f(lanes per rail, open electrodes) for an ion-list kind of the gradient
// pass (64 rows of bits in every shape).
template <class F>
cudaError_t with_ion_grads(int kind, F &&f)
{
    using std::integral_constant;
    const int k = kind - kWordKinds;
    auto go = [&](auto p) {
        return (k & 1) ? f(p, integral_constant<bool, true>()) : f(p, integral_constant<bool, false>());
    };
    switch (k >> 1) {
    case 0: return go(integral_constant<int, 4>());
    case 1: return go(integral_constant<int, 8>());
    case 2: return go(integral_constant<int, 16>());
    default: return go(integral_constant<int, 32>());
    }
}

}  // namespace

cudaError_t ion_grad_launch(const SweepArgs &a, const SweepLaunch &l, cudaStream_t s)
{
    return with_ion_grads(l.kind, [&](auto p, auto open) {
        ion_grad_kernel<decltype(p)::value, decltype(open)::value><<<l.grid, l.warps * 32, l.smem, s>>>(a);
        return cudaGetLastError();
    });
}

cudaError_t ion_batch_grad_launch(const BatchArgs &b, int kind, int grid, int warps, size_t smem, cudaStream_t s)
{
    return with_ion_grads(kind, [&](auto p, auto open) {
        ion_batch_grad_kernel<decltype(p)::value, decltype(open)::value><<<grid, warps * 32, smem, s>>>(b, kind);
        return cudaGetLastError();
    });
}

int ion_grad_ctas_per_sm(int kind, int warps, size_t smem)
{
    int n = 0;
    const cudaError_t e = with_ion_grads(kind, [&](auto p, auto open) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, ion_batch_grad_kernel<decltype(p)::value, decltype(open)::value>, warps * 32, smem);
    });
    return e == cudaSuccess && n > 0 ? n : 1;
}

cudaError_t ion_grad_set_smem_limits()
{
    cudaError_t e = cudaSuccess;
    for (int k = kWordKinds; k < kWordKinds + 8; ++k) {
        const cudaError_t r = with_ion_grads(k, [](auto p, auto open) {
            constexpr int P = decltype(p)::value;
            constexpr bool O = decltype(open)::value;
            const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
            const cudaError_t q = cudaFuncSetAttribute(ion_grad_kernel<P, O>, attr, kGradSmem);
            return q != cudaSuccess ? q : cudaFuncSetAttribute(ion_batch_grad_kernel<P, O>, attr, kGradSmem);
        });
        if (r != cudaSuccess) e = r;
    }
    return e;
}

}  // namespace kmc
