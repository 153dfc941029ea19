// Deterministic block / grid reductions (warp shuffles, then the last-block
// pattern: every block stores one partial, the last block to finish sums the
// partials in a fixed order -- no atomics on data, no spinning).
#pragma once
#include "common.cuh"

namespace jfnk {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// FP64 sums over a warp by integer additions: the significands at the largest
// exponent with 5 bits below its last place (32 of them fit 63 bits), which an
// FP64 addition of two lanes' values is not more accurate than.  Five shuffled
// FP64 additions take the pipe 5 x 64 clocks a warp; this takes it 64.
__device__ __forceinline__ double warp_sum(double v) {
    const int hi = __double2hiint(v), be = (hi >> 20) & 0x7ff;
    const int top = __reduce_max_sync(0xffffffffu, be);
    if (top < 64 || top > 2040) {  // near underflow or overflow, or not finite
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
    long long m = ((__double_as_longlong(v) & 0xfffffffffffffLL) | (be ? 0x10000000000000LL : 0LL)) << 5;
    m >>= min(top - be, 63);
    if (hi < 0) m = -m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
    const double d = __ll2double_rn(m);
    return m ? __hiloint2double(__double2hiint(d) + (top - 1080) * (1 << 20), __double2loint(d)) : 0.0;
}

// Sum over the block of one double per warp-summed value.  All threads must
// call it.  `sm` holds >= 32 doubles.  Result valid in thread 0.
template <typename TA>
__device__ __forceinline__ double block_sum(TA v, double* sm) {
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int nt = blockDim.x * blockDim.y * blockDim.z;
    TA w = warp_sum(v);
    if ((tid & 31) == 0) sm[tid >> 5] = (double)w;
    __syncthreads();
    double t = 0.0;
    if (tid < 32) {
        // (a shuffled FP64 addition costs about 100 clocks: only the steps needed)
        const int nw = (nt + 31) / 32;
        t = (tid < nw) ? sm[tid] : 0.0;
        for (int o = nw > 16 ? 16 : nw > 8 ? 8 : nw > 4 ? 4 : nw > 2 ? 2 : nw > 1 ? 1 : 0; o > 0; o >>= 1)
            t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    __syncthreads();
    return t;
}

// Orders this thread's memory accesses before and after for the GPU (with an
// atomic after or before it: release, acquire).
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Last-block completion over a segment of nb CTAs (bid = this CTA's index in
// it).  Thread 0 of every block passes its block sum; returns true in every
// thread of the last block of the segment, with the total in *total (thread
// 0).  The completion counter is reset by the last block.  `early` runs in one
// thread of the last block while the others sum the partials, and is visible to
// thread 0 on return.  (One warp sums up to 128 partials and 4 warps more: an
// FP64 addition takes an SM quarter 64 clocks a warp.  Blocks have at least one
// whole warp.)
template <typename F>
__device__ __forceinline__ bool grid_sum_last_seg(double blocksum, double* partials, unsigned int* counter,
                                                  double* total, unsigned int bid, unsigned int nb, F early) {
    __shared__ double s_part[4];
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int nt = blockDim.x * blockDim.y * blockDim.z;
    if (nb == 1) {  // the only block: no partials, no completion counter
        if (tid == 0) {
            early();
            *total = blocksum;
        }
        return true;
    }
    __shared__ int s_last;
    if (tid == 0) {
        partials[bid] = blocksum;
        fence_gpu();
        unsigned int prev = atomicAdd(counter, 1u);
        fence_gpu();
        s_last = (prev == nb - 1) ? 1 : 0;
    }
    __syncthreads();
    if (!s_last) return false;
    const int act = nb <= 128 ? 32 : nt >= 128 ? 128 : nt & ~31;
    double s = 0.0;
    if (tid < act) {
        double part[4];
        unsigned int i = tid;
        do {  // four loads in flight
#pragma unroll
            for (int k = 0; k < 4; ++k) part[k] = i + k * act < nb ? __ldcg(&partials[i + k * act]) : 0.0;
            i += 4 * act;
            if (act == 32 && nb <= 32)
                s = part[0];
            else
                s += (part[0] + part[1]) + (part[2] + part[3]);
        } while (i < nb);
        s = warp_sum(s);
        if (act > 32 && (tid & 31) == 0) s_part[tid >> 5] = s;
    }
    if (tid == (act < nt ? act : 0)) early();
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < act / 32; ++w) s += s_part[w];
        *total = s;
        *counter = 0u;
    }
    return true;
}

// The whole grid as one segment.
template <typename F>
__device__ __forceinline__ bool grid_sum_last(double blocksum, double* partials, unsigned int* counter,
                                              double* total, F early) {
    return grid_sum_last_seg(blocksum, partials, counter, total,
                             blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z),
                             gridDim.x * gridDim.y * gridDim.z, early);
}
__device__ __forceinline__ bool grid_sum_last(double blocksum, double* partials, unsigned int* counter,
                                              double* total) {
    return grid_sum_last(blocksum, partials, counter, total, [] {});
}

}  // namespace jfnk
