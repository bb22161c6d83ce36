// kernels_tail.cu -- the soft-binarisation iterations that end the method (Alg. 1 step 3,
// Sec. 4.1).  After the continuous power iterations, each further step applies the Eq. 7
// operator, y = A x, and then squashes the result towards {0, 1} with a sigmoid; the hard
// segmentation is the final x thresholded at 1/2.  The sigmoid acts on y scaled to maximum 1,
//     x <- 1 / (1 + exp(-gain (y / max(y) - center))),
// so that gain and centre mean the same thing for any volume size (the paper leaves the
// sigmoid's parameterisation open).
//
// A step is the stencil launch (for shared maps and a radius that a TMA kernel covers it also takes
// max(y), mode 8 at iter_stream; else y goes to the caller's layout and one reduction takes it), and
// one elementwise pass that writes, for the next step, the stencil's input state u * x in the
// internal layout (so the next stencil launch needs no separate conversion), or x after the last.
#include "common.cuh"
#include "launch.h"
#include "order_key.cuh"
#include "tma.cuh"
#include "voxels.cuh"

namespace sfseg {

__global__ void max_key_kernel(const float* y, int64_t n, unsigned* key) {
    unsigned m = 0u;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        m = max(m, order_key(y[i]));
    m = __reduce_max_sync(0xffffffffu, m);
    __shared__ unsigned wmax[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) wmax[warp] = m;
    __syncthreads();
    if (warp == 0) {
        m = lane < (int)(blockDim.x >> 5) ? wmax[lane] : 0u;
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) atomicMax(key, m);
    }
}

// x = sigmoid(gain (y / max y - center)) for the N voxels, y in the internal layout or (YI false) the
// caller's.  Optional outputs: v (internal layout, u * x, the next stencil input), x and mask (x > 1/2
// as 0/1 bytes), caller layout.  A step that is not the last needs v alone, and reads y from where
// the stencil's TMA store put it: 12 bytes per voxel in 16-byte accesses.  Writing x at every step and
// one voxel per access took 97.5 us for 50x480x854 (16 bytes per voxel).
template <bool YI>
__global__ void sigmoid_step_kernel(const float* y, const unsigned* key, float gain, float center, const float* sm,
                                    float p, Geom g, float* x, float* v, unsigned char* mask, int* flags) {
    wait_previous_grid();
    const float m = order_value(*key);
    if (!(m > 0.f) || isinf(m)) {
        if (blockIdx.x == 0 && threadIdx.x == 0)
            atomicOr(flags, (m > 0.f ? kFlagNonfinite : kFlagZeroNorm) | kFlagTailStop);
        return;
    }
    const float gm = -gain;
    auto act = [&](float yi) { return 1.f / (1.f + expf(gm * (yi / m - center))); };
    auto one = [&](int64_t i, int64_t j) {
        const float xi = act(y[YI ? j : i]);
        if (x) x[i] = xi;
        if (mask) mask[i] = xi > 0.5f ? 1 : 0;
        if (v) v[j] = unary_pow_fast(sm[j], p) * xi;
    };
    if (!YI || x || mask) {
        for_each_voxel(g, one);
        return;
    }
    const int64_t rows = (int64_t)g.T * g.H;
    const int w4 = g.W / 4;
    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
        const int64_t j0 = row * g.pitch;
        for (int c = threadIdx.x; c < w4; c += blockDim.x) {
            const float4 a = *reinterpret_cast<const float4*>(y + j0 + 4 * c);
            const float4 f = *reinterpret_cast<const float4*>(sm + j0 + 4 * c);
            *reinterpret_cast<float4*>(v + j0 + 4 * c) =
                make_float4(unary_pow_fast(f.x, p) * act(a.x), unary_pow_fast(f.y, p) * act(a.y),
                            unary_pow_fast(f.z, p) * act(a.z), unary_pow_fast(f.w, p) * act(a.w));
        }
        for (int w = 4 * w4 + threadIdx.x; w < g.W; w += blockDim.x) one(row * g.W + w, j0 + w);
    }
}

static int grid_for(int64_t n) {
    const int64_t b = (n + 255) / 256;
    const int cap = 8 * num_sms();
    return (int)(b < cap ? (b > 0 ? b : 1) : cap);
}

void launch_max_key(const float* y, int64_t n, unsigned* key, cudaStream_t s) {
    cudaMemsetAsync(key, 0, sizeof(unsigned), s);
    max_key_kernel<<<grid_for(n), 256, 0, s>>>(y, n, key);
    count_launches(1);
}

void launch_sigmoid_step(const float* y, bool y_internal, const unsigned* key, float gain, float center,
                         const float* f32, float p, Geom g, float* x, float* v, unsigned char* mask, int* flags,
                         cudaStream_t s, const float* s32) {
    const float* sm = s32 ? s32 : f32;
    RowLaunch rl = row_launch(g, num_sms());
    if (y_internal) {
        if (!x && !mask) rl.threads = g.W >= 512 ? 128 : (((g.W + 3) / 4 + 31) / 32) * 32;
        launch_after_previous(sigmoid_step_kernel<true>, dim3(rl.blocks), rl.threads, 0, s, y, key, gain, center, sm, p,
                              g, x, v, mask, flags);
    } else {
        launch_after_previous(sigmoid_step_kernel<false>, dim3(rl.blocks), rl.threads, 0, s, y, key, gain, center, sm, p,
                              g, x, v, mask, flags);
    }
    count_launches(1);
}

}  // namespace sfseg
