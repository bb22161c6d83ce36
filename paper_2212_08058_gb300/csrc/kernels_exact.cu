// kernels_exact.cu -- the element-wise parts of the exact (Eq. 1) kernel's operator, the
// diagnostic of the first-order approximation (Sec. 4.3): M_ij = u_i u_j exp(-a (f_i - f_j)^2) G_ij
// written with g = f - c as the series e^{-a g_i^2} e^{-a g_j^2} sum_n c_n g_i^n g_j^n,
// c_n = (2a)^n / n!, whose terms are separable and go through the TMA kernels three at a time
// (iter_stream.cuh, mode 7).  With A = u e^{-a g^2} a step is: w = A x~, S = s sum_n c_n g^n G*(g^n w),
// the next x~ = A S / a.  The norm s = 1/||x~|| is summed by the pass that forms w and applied by the
// filtering (the operator is linear), so no pass waits for it.
//
// c = 0 is the series in f itself, which g reads then.  The middle of f's range halves max |g|, and the terms
// needed follow x = 2 a max(g)^2: 9 instead of 16 for f in [0, 1] at a = 1, three filterings a step instead
// of six, but its alternating terms cancel digits of small outputs, so it is taken up to
// a (range of f)^2 = 1 (kCentredRange, api.cu).  These passes move 12 bytes per voxel, four columns per
// thread (rows start 128-byte aligned).  Five steps at 32x240x427, (2,7,7), f in [0, 1], the call: 597 us
// centred, 1097 with the series in f.
#include "launch.h"
#include "order_key.cuh"
#include "tma.cuh"
#include "voxels.cuh"

namespace sfseg {

namespace {

// f4(j) for the groups of four columns of every internal row, f1(i, j) for the ragged ends (i the
// caller-layout index, j the internal one).
template <typename F4, typename F1>
__device__ __forceinline__ void for_each_quad(const Geom& g, F4&& f4, F1&& f1) {
    const int64_t rows = (int64_t)g.T * g.H;
    const int w4 = g.W / 4;
    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
        const int64_t j0 = row * g.pitch, i0 = row * g.W;
        for (int c = threadIdx.x; c < w4; c += blockDim.x) f4(j0 + 4 * c);
        for (int w = 4 * w4 + threadIdx.x; w < g.W; w += blockDim.x) f1(i0 + w, j0 + w);
    }
}
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

RowLaunch quad_launch(const Geom& g, int per_sm) {
    const int64_t rows = (int64_t)g.T * g.H, cap = (int64_t)per_sm * num_sms();
    const int w4 = (g.W + 3) / 4;
    return {(int)(rows < cap ? rows : cap), w4 >= 128 ? 128 : (w4 + 31) / 32 * 32};
}

// A thread's sum of squares, each addition's rounding carried into the next (Kahan).  A plain float32 sum
// takes 850 terms of a 120x1080x1920 volume and put the norm of equal voxels 8e-6 off.
struct SquareSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float y = __fmaf_rn(v, v, -c), t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
};

__device__ __forceinline__ void add_sum(const SquareSum& part, double* acc) {
    const double b = block_sum((double)part.s - (double)part.c);
    if (threadIdx.x == 0 && acc) atomicAdd(acc, b);
}

}  // namespace

// One pair of atomics per block: one per warp took 6 us of them for 480 rows.
__global__ void exact_range_kernel(const float* f, Geom g, unsigned* keys) {
    __shared__ unsigned best[2];
    if (threadIdx.x < 2) best[threadIdx.x] = 0u;
    __syncthreads();
    unsigned hi = 0u, lo = 0u;
    for_each_voxel(g, [&](int64_t, int64_t j) {
        hi = max(hi, order_key(f[j]));
        lo = max(lo, order_key(-f[j]));
    });
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_max_sync(0xffffffffu, lo);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(best, hi);
        atomicMax(best + 1, lo);
    }
    __syncthreads();
    if (threadIdx.x < 2) atomicMax(keys + threadIdx.x, best[threadIdx.x]);
}

__global__ void exact_setup_kernel(const float* f, float center, float alpha, float p, Geom g, float* gf, float* A) {
    for_each_voxel(g, [&](int64_t, int64_t j) {
        const float fv = f[j], gv = fv - center;
        if (gf) gf[j] = gv;
        A[j] = unary_pow_fast(fv, p) * expf(-alpha * gv * gv);
    });
}

__global__ void exact_in_kernel(const float* x_user, const float* A, Geom g, float* w, double* acc) {
    SquareSum part;
    for_each_voxel(g, [&](int64_t i, int64_t j) {
        const float v = x_user ? x_user[i] : 1.f;
        w[j] = A[j] * v;
        part.add(v);
    });
    add_sum(part, acc);
}

__global__ void exact_mid_kernel(const float* S, const float* A, float inv_alpha, Geom g, float* w, double* acc) {
    wait_previous_grid();
    SquareSum part;
    auto one = [&](float s, float a) {
        const float x = a * s * inv_alpha;
        part.add(x);
        return a * x;
    };
    for_each_quad(
        g,
        [&](int64_t j) {
            const float4 s = ld4(S + j), a = ld4(A + j);
            st4(w + j, make_float4(one(s.x, a.x), one(s.y, a.y), one(s.z, a.z), one(s.w, a.w)));
        },
        [&](int64_t, int64_t j) { w[j] = one(S[j], A[j]); });
    add_sum(part, acc);
}

__global__ void exact_next_kernel(const float* gf, Geom g, float* v) {
    wait_previous_grid();
    for_each_quad(
        g,
        [&](int64_t j) {
            const float4 a = ld4(gf + j), x = ld4(v + j);
            st4(v + j, make_float4(a.x * a.x * a.x * x.x, a.y * a.y * a.y * x.y, a.z * a.z * a.z * x.z,
                                   a.w * a.w * a.w * x.w));
        },
        [&](int64_t, int64_t j) { v[j] *= gf[j] * gf[j] * gf[j]; });
}

__global__ void exact_out_kernel(const float* S, const float* A, float inv_alpha, Geom g, float* x_user, double* acc) {
    SquareSum part;
    for_each_voxel(g, [&](int64_t i, int64_t j) {
        const float x = A[j] * S[j] * inv_alpha;
        x_user[i] = x;
        part.add(x);
    });
    add_sum(part, acc);
}

void launch_exact_range(const float* f32, Geom g, unsigned* keys, cudaStream_t s) {
    const RowLaunch rl = row_launch(g, num_sms(), 8);
    exact_range_kernel<<<rl.blocks, rl.threads, 0, s>>>(f32, g, keys);
    count_launches(1);
}

void launch_exact_setup(const float* f32, float center, float alpha, float p, Geom g, float* gf, float* A,
                        cudaStream_t s) {
    const RowLaunch rl = row_launch(g, num_sms());
    exact_setup_kernel<<<rl.blocks, rl.threads, 0, s>>>(f32, center, alpha, p, g, gf, A);
    count_launches(1);
}

void launch_exact_in(const float* x_user, const float* A, Geom g, float* w, double* acc, cudaStream_t s) {
    const RowLaunch rl = row_launch(g, num_sms(), 8);
    exact_in_kernel<<<rl.blocks, rl.threads, 0, s>>>(x_user, A, g, w, acc);
    count_launches(1);
}

void launch_exact_mid(const float* S, const float* A, float inv_alpha, Geom g, float* w, double* acc, cudaStream_t s) {
    const RowLaunch rl = quad_launch(g, 16);
    launch_after_previous(exact_mid_kernel, dim3(rl.blocks), rl.threads, 0, s, S, A, inv_alpha, g, w, acc);
    count_launches(1);
}

void launch_exact_next(const float* gf, Geom g, float* v, cudaStream_t s) {
    const RowLaunch rl = quad_launch(g, 16);
    launch_after_previous(exact_next_kernel, dim3(rl.blocks), rl.threads, 0, s, gf, g, v);
    count_launches(1);
}

void launch_exact_out(const float* S, const float* A, float inv_alpha, Geom g, float* x_user, double* acc,
                      cudaStream_t s) {
    const RowLaunch rl = row_launch(g, num_sms(), 8);
    exact_out_kernel<<<rl.blocks, rl.threads, 0, s>>>(S, A, inv_alpha, g, x_user, acc);
    count_launches(1);
}

}  // namespace sfseg
