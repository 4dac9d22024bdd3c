// Device helpers shared by the library's kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace esim {

constexpr int kBlock = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Deterministic block sum (fixed tree).  Result valid in thread 0.  All threads
// of the block must call it; `smem` holds one value per warp.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* smem) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) smem[wid] = v;
    __syncthreads();
    T r = 0;
    if (wid == 0) {
        r = lane < nw ? smem[lane] : T(0);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    __syncthreads();
    return r;
}

// count / R as a double (0 for R = 0), count <= R.  Many nodes have few pairs that all end alike;
// 0 and 1 are exact without the division, which is slow here.
__device__ __forceinline__ double pair_ratio(uint64_t count, uint64_t R) {
    if (count == 0 || R == 0) return 0.0;
    return count == R ? 1.0 : (double)count / (double)R;
}

// Programmatic dependent launch: a kernel that starts with prior_done() may be launched with
// launch_after(), which lets it start while the kernel before it in the stream still runs.
// What it does before prior_done() touches nothing that an earlier kernel of the stream
// writes.  next_may_start() lets the kernel after it start likewise.
// Such a kernel begins before its inputs are written.  Only the graph's tables are const
// __restrict__ or read by __ldg in it: the read-only path is for data that does not change while
// the kernel runs, and the wait does not order its loads.
__device__ __forceinline__ void prior_done() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;"); }

template <class... Params, class... Args>
cudaError_t launch_after(cudaStream_t stream, dim3 blocks, unsigned threads, size_t smem, void (*kernel)(Params...),
                         Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = blocks;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // returned here, not to the next launch's check as well
    return e;
}

}  // namespace esim
