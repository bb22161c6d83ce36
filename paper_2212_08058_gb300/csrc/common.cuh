// common.cuh -- device helpers shared by the sfseg kernels (sm_103a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace sfseg {

constexpr int kMaxRT = 4;
constexpr int kMaxRH = 8;
constexpr int kMaxRW = 8;

// Error flag bits written by kernels into the handle's device flag word.
constexpr int kFlagBadFeature = 1;   // a feature value was negative, NaN or Inf
constexpr int kFlagZeroNorm = 2;     // an iterate norm was exactly zero
constexpr int kFlagNonfinite = 4;    // an iterate norm was NaN or Inf
constexpr int kFlagTimeout = 8;      // a bounded wait inside a kernel gave up
constexpr int kFlagTailStop = 16;    // a soft-binarisation step stopped at its maximum (not an error by itself)

// 1D factors of the separable Gaussian (Sec. 4.2), index d + r for offset d in [-r, r].
struct Taps {
    int rt, rh, rw;
    float gt[2 * kMaxRT + 1];
    float gh[2 * kMaxRH + 1];
    float gw[2 * kMaxRW + 1];
};

// Geometry of the handle's volumes.  Internal volumes have a padded row pitch (a multiple of
// 8 elements, so every row starts 16-byte aligned for bf16 and float); the caller's volumes
// use pitch W.
struct Geom {
    int T, H, W;
    int pitch;   // elements per row of internal volumes
};

__device__ __forceinline__ float ldf(const float* p) { return *p; }
__device__ __forceinline__ float ldf(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void stf(float* p, float v) { *p = v; }
__device__ __forceinline__ void stf(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// Unary term u = s^p with 0^p := 0 (p > 0).
__device__ __forceinline__ float unary_pow(float s, float p) {
    return s > 0.f ? exp2f(p * log2f(s)) : 0.f;
}

// Faster variant on the special-function unit: u = 2^(p log2 s) with the approximate log2 and
// exp2 instructions (relative error a few 1e-7 for p <= 1).  s = 0 gives log2 s = -inf and
// u = +0, so no branch is needed (s < 0 never reaches here: features are checked >= 0).  Both
// take and give subnormal numbers; with FTZ a u below 2^-126 becomes 0, three instructions less.
template <bool FTZ = false>
__device__ __forceinline__ float unary_pow_fast(float s, float p) {
    float l, u;
    asm("lg2.approx.f32 %0, %1;" : "=f"(l) : "f"(s));
    if constexpr (FTZ) asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(u) : "f"(p * l));
    else asm("ex2.approx.f32 %0, %1;" : "=f"(u) : "f"(p * l));
    return u;
}
// No positive float32 s is below 2^-149, so u is subnormal only for p > 126 / 149 = 0.845: up to this p the
// shorter form gives the same numbers.
constexpr float kUnaryFtzP = 0.84f;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum of `v` over the block (blockDim a multiple of 32, at most 256).  All threads must call it;
// the result is valid in thread 0.
// FP64 runs at 2 FMA per clock per SM here, 1/64 of FP32: a butterfly in every warp costs 5 FP64
// additions per warp, 45 for 256 threads, 16 clocks each (about 2.5 us for an SM's eight blocks).
// So the partial sums go through shared memory and one warp adds them: 12 for 256 threads.
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double red[256];
    __syncthreads();   // protects red[] against a previous call
    red[threadIdx.x] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = red[threadIdx.x];
        for (int i = threadIdx.x + 32; i < (int)blockDim.x; i += 32) r += red[i];
        r = warp_sum(r);
    }
    return r;
}

// 1/sqrt(acc) of an FP64 sum of squares, with the flag raised (and 0 returned) when the sum is
// zero or not finite, so that later iterations produce zeros instead of NaNs.  For one thread of
// a block (block_inv_norm gives it to all): an FP64 square root and division in every thread of a
// launch cost more than many of the launches' own work (3.3M voxels, 2432 x 256 threads: 25 us of
// a 28.6 us pass).  Within float's range the reciprocal square root is one FP64 Newton step from
// the FP32 one (relative error below 2^-43 before the rounding to float).
__device__ __forceinline__ float inv_norm_from(const double* acc, int* flags) {
    if (acc == nullptr) return 1.f;
    const double a = *acc;
    if (a > 1e-30 && a < 1e30) {
        const double y = (double)rsqrtf((float)a);
        const double e = fma(-a * y, y, 1.0);
        return (float)fma(0.5 * y, e, y);
    }
    if (!(a > 0.0) || !(a < 1e300)) {
        if (flags) atomicOr(flags, a == 0.0 ? kFlagZeroNorm : kFlagNonfinite);
        return 0.f;
    }
    return (float)(1.0 / sqrt(a));
}

// f() of one thread given to the whole block; every thread must call it.  `I` tells the calls of
// one kernel apart (each has its own shared word).
template <int I = 0, typename F>
__device__ __forceinline__ float block_value(F&& f) {
    __shared__ float value;
    if (threadIdx.x == 0) value = f();
    __syncthreads();
    return value;
}

template <int I = 0>
__device__ __forceinline__ float block_inv_norm(const double* acc, int* flags) {
    return block_value<I>([&] { return inv_norm_from(acc, flags); });
}

}  // namespace sfseg
