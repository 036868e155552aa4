// Device-side helpers shared by the kernels of libevp_gb300 (sm_103a).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace evp {

template <typename T> struct CT;
template <> struct CT<float> { using type = float2; };
template <> struct CT<double> { using type = double2; };

template <typename C> __device__ __forceinline__ C cmk(decltype(C::x) a, decltype(C::x) b) { C c; c.x = a; c.y = b; return c; }
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return cmk<C>(a.x + b.x, a.y + b.y); }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return cmk<C>(a.x - b.x, a.y - b.y); }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) { return cmk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
template <typename C> __device__ __forceinline__ C cconj(C a) { return cmk<C>(a.x, -a.y); }

__device__ __forceinline__ int bitrev(int j, int logN) { return (int)(__brev((unsigned)j) >> (32 - logN)); }

// Block-wide sum of one double per thread; result valid in thread 0. blockDim.x <= 1024.
__device__ __forceinline__ double block_sum(double v, double *sh /* >= 32 doubles */) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    v = (threadIdx.x < nw) ? sh[threadIdx.x] : 0.0;
    if (wid == 0)
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Error-free sum of two floats (Knuth): s is the rounded sum and s + e equals a + b exactly, while s is finite.
__device__ __forceinline__ void two_sum_f(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Programmatic dependent launch (sm_90+). The kernels of one fixed-point iteration are queued back to back; each is
// launched with programmatic stream serialization, so its launch overlaps the exit of its predecessor's last CTAs.
// pdl_wait() blocks until the preceding kernel has completed and its memory is visible (a no-op for a kernel
// launched without the attribute), so it comes before any access to data an earlier kernel wrote. No kernel signals its
// successor earlier (griddepcontrol.launch_dependents): CTAs launched while the predecessor still runs settle on
// whichever SMs have room, and the uneven shares cost more than the launch latency they hide. Iteration times with
// the signal at every kernel's start and without it: 29.3 / 28.0 us (32^3 FP32), 65.8 / 49.1 (64^3 FP32), 222 / 203
// (128^3 FP32), 686 / 608 (64^3 FP64, where the FP64 pipe of the fullest SM decides).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                            Args... args) {
    if (!pdl) {
        kernel<<<grid, block, smem, s>>>(args...);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace evp
