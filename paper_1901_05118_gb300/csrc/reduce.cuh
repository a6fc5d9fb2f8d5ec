// Deterministic CTA and grid reductions shared by the kernels that fuse an
// inner product (the Bi-CG scalars of Alg. 2).  A fixed grid reduces its
// per-CTA partials in CTA order in the last CTA to finish (atomic ticket), so
// equal inputs always give equal bits.
#pragma once

#include <cuda_runtime.h>

namespace excmg {

// a b + c, fused, evaluated only where the program reaches it.  The compiler
// moves a plain FMA out of a branch that is rarely taken and selects the
// result, and a warp's FP64 instruction holds its pipe for 64 cycles: so placed,
// the shadow updates cost the Bi-CG update 5.75 instead of 3 FP64 instructions
// per entry and kept the pipe 85 % busy (189 against 166 us at 256^3).
__device__ __forceinline__ double fma_here(double a, double b, double c) {
    double d;
    asm volatile("fma.rn.f64 %0, %1, %2, %3;" : "=d"(d) : "d"(a), "d"(b), "d"(c));
    return d;
}

// 0 or 1, unknown to the compiler: the trip count of a loop that stands for a
// branch which has to stay one.  (A short block becomes predicated
// instructions, which hold the FP64 pipe as if they were executed: the step
// with directions on 256^3 takes 236 us so, 218 with the loop, the on-chip Bi-CG on
// 64^3 11.3 and 10.3 us per iteration.)
__device__ __forceinline__ int opaque(bool c) {
    int v = c ? 1 : 0;
    asm volatile("" : "+r"(v));
    return v;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sum of v over the CTA (valid in thread 0).  sh: 32 values of shared memory.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* sh) {
    const int nthreads = blockDim.x * blockDim.y * blockDim.z;
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int lane = tid & 31, wid = tid >> 5;
    v = warp_sum(v);
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    T t = T(0);
    if (wid == 0) {
        t = lane < (nthreads >> 5) ? sh[lane] : T(0);
        t = warp_sum(t);
    }
    __syncthreads();
    return t;
}

__device__ __forceinline__ int flat_block() {
    return blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
}
__device__ __forceinline__ int flat_grid() { return gridDim.x * gridDim.y * gridDim.z; }
__device__ __forceinline__ bool thread0() { return threadIdx.x == 0 && threadIdx.y == 0 && threadIdx.z == 0; }

// Publish this CTA's `count` partial sums and report (to every thread)
// whether this CTA is the last one to do so.
__device__ __forceinline__ bool publish_partials(const double* vals, int count, double* partials,
                                                 unsigned int* ticket, bool* am_last) {
    if (thread0()) {
        const int G = flat_grid(), b = flat_block();
        for (int c = 0; c < count; ++c) partials[c * G + b] = vals[c];
        __threadfence();
        const unsigned int t = atomicAdd(ticket, 1u);
        *am_last = (t == (unsigned)G - 1u);
    }
    __syncthreads();
    return *am_last;
}

// In the last CTA: the total of component c over all CTAs, in CTA order.
__device__ __forceinline__ double gather_partials(const double* partials, int c, double* sh) {
    const int G = flat_grid();
    const int nthreads = blockDim.x * blockDim.y * blockDim.z;
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    double v = 0.0;
    for (int b = tid; b < G; b += nthreads) v += __ldcg(&partials[c * G + b]);
    return block_sum(v, sh);
}

}  // namespace excmg
