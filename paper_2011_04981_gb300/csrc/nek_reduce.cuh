// Deterministic block reduction helpers: a fixed grid accumulates per-thread
// grid-stride sums, a block adds its threads' sums in a fixed order and writes one
// partial; a single block then sums the partials in order.
//
// An FP64 addition of a warp occupies the scheduler's FP64 pipe for 64 cycles (2 lanes per SM and clock), so a block
// adds its threads' sums through shared memory with one warp a sum: lane l takes the threads l, l + 32, ..., then a
// shuffle tree, 12 additions for 256 threads where a tree in every warp takes 45.  Two sums go to two warps.  The r update
// of the FP32 solve (4 M points, 1216 blocks) went from 18.3 to 13.2 us, k_beta from 10.3 to 6.9 (launch list, cold cache).
#pragma once

#include <cuda_runtime.h>

namespace nek {

// Sum of warp-owned values v over the 32 lanes, in every lane.
__device__ __forceinline__ double warp_tree(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The block's sums of v[0 .. M-1]; sum m is returned in the threads of warp m (the others get 0).
template <int NT, int M>
__device__ __forceinline__ double block_sums(const double (&v)[M], double* sh /* M * NT doubles */)
{
    static_assert(M <= NT / 32, "a warp for every sum");
#pragma unroll
    for (int m = 0; m < M; m++) sh[m * NT + threadIdx.x] = v[m];
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double t = 0.0;
    if (wid < M) {
#pragma unroll
        for (int k = 0; k < NT / 32; k++) t += sh[wid * NT + lane + 32 * k];
        t = warp_tree(t);
    }
    __syncthreads();
    return t;
}

template <int NT>
__device__ __forceinline__ double block_sum(double v, double* sh /* NT doubles */)
{
    const double a[1] = {v};
    return block_sums<NT, 1>(a, sh);  // valid in thread 0
}

// The block's two sums to parts[block] and parts[blocks + block].
template <int NT>
__device__ __forceinline__ void write_two_partials(double a, double b, double* parts, double* sh /* 2 NT doubles */)
{
    const double v[2] = {a, b};
    const double t = block_sums<NT, 2>(v, sh);
    if ((threadIdx.x & 31) == 0 && threadIdx.x < 64) parts[(threadIdx.x >> 5) * gridDim.x + blockIdx.x] = t;
}

// Sum of nparts partials (in a fixed order) by one block of NT threads.  The
// unrolled loop issues a thread's loads together; the adds stay in order.
template <int NT>
__device__ __forceinline__ double sum_partials(const double* __restrict__ parts, int nparts, double* sh)
{
    double v = 0.0;
#pragma unroll 8
    for (int q = threadIdx.x; q < nparts; q += NT) v += parts[q];
    return block_sum<NT>(v, sh);
}

// The sums of parts[0, nparts) and parts[nparts, 2 nparts), both valid in thread 0.
template <int NT>
__device__ __forceinline__ void sum_two_partials(const double* __restrict__ parts, int nparts, double* sh /* 2 NT */,
                                                 double& a, double& b)
{
    double v[2] = {0.0, 0.0};
#pragma unroll 8
    for (int q = threadIdx.x; q < nparts; q += NT) {
        v[0] += parts[q];
        v[1] += parts[nparts + q];
    }
    const double t = block_sums<NT, 2>(v, sh);
    if (threadIdx.x == 32) sh[0] = t;
    __syncthreads();
    a = t;
    b = sh[0];
}

// out[e] = sum of the values v of element e's threads (thread t belongs to
// element t / TPE).  Each element's TPE values are summed in a fixed order
// (lane-strided, then a shuffle tree), so the result depends on nx only, not on
// the number of elements per CTA.  sh: blockDim doubles of shared memory that
// no thread reads any more.
template <int TPE, int EPB>
__device__ __forceinline__ void element_sums(double v, double* sh, double* __restrict__ out, int ne)
{
    __syncthreads();
    sh[threadIdx.x] = v;
    __syncthreads();
    if constexpr (TPE >= 32) {
        if (threadIdx.x < EPB * 32) {  // whole warps: the block has EPB * TPE >= EPB * 32 threads
            const int e = threadIdx.x >> 5, lane = threadIdx.x & 31;
            double t = 0.0;
            for (int q = lane; q < TPE; q += 32) t += sh[e * TPE + q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0 && e < ne) out[e] = t;
        }
    } else {
        if (threadIdx.x < EPB) {
            double t = 0.0;
            for (int q = 0; q < TPE; q++) t += sh[threadIdx.x * TPE + q];
            if ((int)threadIdx.x < ne) out[threadIdx.x] = t;
        }
    }
}

}  // namespace nek
