// kernels_fast.cu -- which kernel runs an Eq. 7 step: the radii with compiled kernels (one file per
// radius, step_*.cu), the radius a step without one is padded to, and the choice between the
// streaming kernel (iter_stream.cuh) and the small-volume one (iter_tile.cuh).
#include "step.h"

namespace sfseg {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static const EncodeTiledFn fn = [] {   // once, whichever thread comes first
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        const bool ok = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                            cudaSuccess &&
                        q == cudaDriverEntryPointSuccess;
        return ok ? (EncodeTiledFn)p : nullptr;
    }();
    return fn;
}

bool make_step_map(CUtensorMap* map, const void* base, bool bf16, const Geom& g, int box_w, int box_h) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const size_t es = bf16 ? 2 : 4;
    cuuint64_t dims[3] = {(cuuint64_t)g.W, (cuuint64_t)g.H, (cuuint64_t)g.T};
    cuuint64_t strides[2] = {(cuuint64_t)g.pitch * es, (cuuint64_t)g.pitch * es * g.H};
    cuuint32_t box[3] = {(cuuint32_t)box_w, (cuuint32_t)box_h, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                    const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

#define SFSEG_RADII(X)                                                                                    \
    X(1, 3, 3) X(2, 7, 7) X(1, 4, 4) X(1, 2, 2) X(1, 5, 5) X(2, 3, 3) X(2, 5, 5) X(1, 7, 7) X(2, 8, 8)
#define SFSEG_DECLARE(A, B, C)                        \
    bool stream_step_##A##_##B##_##C(const StepArgs&); \
    bool tile_step_##A##_##B##_##C(const StepArgs&);
SFSEG_RADII(SFSEG_DECLARE)
#undef SFSEG_DECLARE

namespace {

struct Radius {
    int rt, rh, rw;
    bool own;   // listed as a radius with its own kernel; (2,8,8) serves others only
    bool (*stream)(const StepArgs&);
    bool (*tile)(const StepArgs&);
};
// The method's (1,3,3) and (2,7,7); (1,4,4) and (1,2,2), the radii of (2,7,7) on 2x- and
// 4x-coarsened volumes (sfseg_coarse_start); the neighbourhoods between them.
const Radius kRadii[] = {
#define SFSEG_ROW(A, B, C) {A, B, C, !(A == 2 && B == 8 && C == 8), stream_step_##A##_##B##_##C, tile_step_##A##_##B##_##C},
    SFSEG_RADII(SFSEG_ROW)
#undef SFSEG_ROW
};

const Radius* own_radius(const Taps& tp) {
    for (const Radius& r : kRadii)
        if (r.own && r.rt == tp.rt && r.rh == tp.rh && r.rw == tp.rw) return &r;
    return nullptr;
}

// The compiled radius with the fewest taps that covers tp; the taps beyond tp's are zero, which adds
// exactly nothing.  Radii with rt <= 2 have one; rt = 3 and 4 (whose t-filter state no thread's
// registers hold beside 8 columns) run on the generic stencil.
const Radius* covering_radius(const Taps& tp) {
    const Radius* best = nullptr;
    for (const Radius& r : kRadii)
        if (r.rt >= tp.rt && r.rh >= tp.rh && r.rw >= tp.rw &&
            (!best || r.rt + r.rh + r.rw < best->rt + best->rh + best->rw))
            best = &r;
    return best;
}

// Which kernel a volume takes.  Where the small-tile kernel has at most one block per SM, that one: 1.2
// times as fast or more on all 156 such volumes timed (2x22x33 at (2,8,8) 6.3 us, streaming 9.9).  Else the
// one whose time, modelled from the frames its busiest SM streams, is shorter.  The streaming kernel takes
// 4.7 us and u per frame step, its steps being the whole tiles' frames (rt more each to flush) and the
// share of the tiles left over (3 rt more for the cuts); the small-tile kernel 0.4 us and 1.8 u per step of
// its three CTAs per SM.  u = 0.55 + 0.0235 us per tap.
// Both kernels timed on 92 volumes at four or six radii, 508 pairs: the choice costs 0.6 % on average, more
// than 12 % for eight pairs, at worst 23 % (70x64x112 at (2,7,7): its frames fill the streaming kernel's
// tiles and three quarters of the small ones).  Measured, tile / streaming kernel, (2,7,7): 16x128x128
// 11.7 / 12.6 us, 60x128x128 18.1 / 22.6, 13x480x854 39.4 / 41.3, 32x240x427 31.3 / 29.6, 25x480x854
// 69.8 / 65.2, 64x480x854 168 / 140; (1,3,3): 32x240x427 18.7 / 19.3, 48x240x427 25.6 / 25.3,
// 64x480x854 111 / 99.5.
bool stream_pays(const Geom& g, const Radius& r) {
    const double G = num_sms(), T = g.T, u = 0.55 + 0.0235 * (2 * (r.rt + r.rh + r.rw) + 3);
    const int64_t big = (int64_t)((g.W + 111) / 112) * ((g.H + 17) / 18);      // 18 x 112 tiles
    const int64_t small = (int64_t)((g.W + 63) / 64) * ((g.H + 14) / 15);      // 15 x 64 tiles
    if (small > 3 * (int64_t)num_sms() * 16) return true;    // many waves: the streaming kernel's steps are cheaper
    const int chunk = tile_chunk(g.T, (int)small, 3 * num_sms(), r.rt);
    const double blocks = (double)small * ((g.T + chunk - 1) / chunk), waves = blocks / (3 * G);
    if (blocks <= G) return false;
    const int64_t whole = big / num_sms(), rest = big - whole * num_sms();
    const double stream = 4.7 + u * (whole * (T + r.rt) + (rest ? rest * T / G + 3 * r.rt : 0.0));
    const double tile = 0.4 + 1.8 * u * (chunk + (chunk < g.T ? 2 : 1) * r.rt) * (waves > 1.0 ? waves : 1.0);
    return stream <= tile;
}

thread_local StepKernel g_ran = {};

bool run(const StepArgs& a) {
    const Radius* r = covering_radius(a.tp);
    if (!r) return false;
    // u = s^p may be subnormal for these p, and the small-volume kernel would flush it (its code with both
    // forms of u is 2 % slower on 8x64x64, for all p)
    const bool deep = a.mode != kExactTerm && a.p > kUnaryFtzP;
    const bool stream = deep || stream_pays(a.g, *r);
    if (!(stream ? r->stream(a) : r->tile(a))) return false;
    g_ran = {stream, r->rt, r->rh, r->rw};
    return true;
}

StepArgs args(int mode, const void* vin, void* out, const void* f, const Geom& g, const Taps& tp, float inv_alpha,
              float p, const double* acc_in, double* acc_out, int* flags, cudaStream_t s) {
    StepArgs a;
    a.mode = mode;
    a.vin = vin;
    a.out = out;
    a.f = f;
    a.g = g;
    a.tp = tp;
    a.inv_alpha = inv_alpha;
    a.p = p;
    a.acc_in = acc_in;
    a.acc_out = acc_out;
    a.flags = flags;
    a.s = s;
    return a;
}

}  // namespace

StepKernel last_step_kernel() { return g_ran; }

bool fast_iterate_supported(const Taps& tp) { return own_radius(tp) != nullptr; }
bool fast_step_supported(const Taps& tp) { return covering_radius(tp) != nullptr; }

bool launch_iterate_fast(const void* vin, int vin_type, void* out, int out_type, bool out_x, const void* f,
                         const Geom& g, const Taps& tp, float inv_alpha, float p, const double* acc_in,
                         double* acc_out, int* flags, cudaStream_t s, const float* s32) {
    StepArgs a = args(kStep, vin, out, f, g, tp, inv_alpha, p, acc_in, acc_out, flags, s);
    a.vin_type = vin_type;
    a.out_type = out_type;
    a.out_x = out_x;
    a.s32 = s32;
    return run(a);
}

bool launch_iterate_fast_max(const float* vin, float* y, const float* f, const Geom& g, const Taps& tp,
                             float inv_alpha, float p, unsigned* maxkey, int* flags, cudaStream_t s) {
    StepArgs a = args(kStepMax, vin, y, f, g, tp, inv_alpha, p, nullptr, nullptr, flags, s);
    a.maxkey = maxkey;
    return run(a);
}

bool launch_iterate_fast_last(const float* vin, float* x, const float* f, const Geom& g, const Taps& tp,
                              float inv_alpha, float p, const double* acc_in, double* acc_out, int* flags,
                              cudaStream_t s) {
    return run(args(kStepMax, vin, x, f, g, tp, inv_alpha, p, acc_in, acc_out, flags, s));
}

bool launch_iterate_fast_ckpt(const float* vin, float* out, const float* f, const Geom& g, const Taps& tp,
                              float inv_alpha, float p, const double* acc_in, double* acc_out, float* ckpt, int* flags,
                              cudaStream_t s) {
    StepArgs a = args(kRecord, vin, out, f, g, tp, inv_alpha, p, acc_in, acc_out, flags, s);
    a.out2 = ckpt;
    return run(a);
}

bool launch_filter_fast(const float* vin, float* out, const float* f, const Geom& g, const Taps& tp, float inv_alpha,
                        float p, const double* acc_in, int* flags, cudaStream_t s) {
    return run(args(kQPass, vin, out, f, g, tp, inv_alpha, p, acc_in, nullptr, flags, s));
}

bool launch_adjoint_gpass_fast(const float* vg, float* G, float* Qg, const float* Vk, const float* f, const Geom& g,
                               const Taps& tp, float inv_alpha, float p, double* dot, int* flags, cudaStream_t s) {
    StepArgs a = args(kGPass, vg, G, f, g, tp, inv_alpha, p, nullptr, dot, flags, s);
    a.s32 = Vk;
    a.out2 = Qg;
    return run(a);
}

bool launch_step_q_fast(const float* vin, float* vout, float* Q, const float* f, const Geom& g, const Taps& tp,
                        float inv_alpha, float p, const double* acc_in, int* flags, cudaStream_t s) {
    StepArgs a = args(kStepQ, vin, vout, f, g, tp, inv_alpha, p, acc_in, nullptr, flags, s);
    a.out2 = Q;
    return run(a);
}

bool launch_exact_term_fast(const float* v, float* y, const float* gf, const Geom& g, const Taps& tp,
                            const ExactTerm& ex, const double* acc_in, int* flags, cudaStream_t s) {
    StepArgs a = args(kExactTerm, v, y, gf, g, tp, 1.f, 1.f, acc_in, nullptr, flags, s);
    a.ex = &ex;
    return run(a);
}

}  // namespace sfseg
