// iter_tile.cuh -- the power-iteration step of Eq. 7 with a compiled radius, written for sm_103a: the
// kernel for small and short volumes (the others: iter_stream.cuh).
//
// One CTA (128 threads, three per SM) owns a 15 x 64 tile of (h, w) and streams along t through
// a chunk of frames.  Per incoming frame:
//   1. TMA brings the raw halo tile of v (= u x~) and f into shared memory (15 + 2rh rows of
//      80 columns; zero fill outside the volume gives the zero padding, also for whole frames
//      before the first and after the last).  The copies of the next frames are in flight
//      while frame t is computed.
//   2. h-pass: a thread takes a column pair and 5 output rows (40 pairs x 3 row groups = 120 of
//      the 128 threads); it walks down the 5 + 2rh input rows once, forms the three signals z1 = v, z2 = f^2 v, z3 = f v of each, and accumulates
//      them into its 5 x 3 outputs with packed FP32 FMAs (FFMA2, one per column pair).
//   3. w-pass: a thread takes 8 output columns of one row; it loads its window of the h-pass
//      result once as aligned float2 pairs (the odd taps run as two scalar FMAs) and feeds the three
//      w-filtered signals straight into the t-filter, kept in registers in transposed direct
//      form (2rt running partial sums per value, no frame ring to index).
//   4. Eq. 7 combination for the frame rt behind, the Eq. 8 norm partial and the store of the
//      next state.
// The h-pass result is double-buffered and the epilogue reads f from global memory, so a frame
// needs a single CTA barrier (after its h-pass): warps still finishing frame t overlap with
// warps already starting frame t+1.
// Bytes moved through shared memory per voxel are about 100 at (2,7,7): the TMA write, one
// read of the raw tile per 8 rows, one write and one windowed read of the h-pass result.  No
// pass re-reads its taps from shared memory and the t-filter reads nothing from it.  The frame
// loop is not unrolled, which keeps the kernel small enough for the instruction cache.
#pragma once

#include "order_key.cuh"
#include "step.h"
#include "tma.cuh"

namespace sfseg {
namespace tile {

constexpr int TH = 15;         // tile rows (at most 16: four rows per warp)
constexpr int TW = 64;         // tile columns
constexpr int PADW = 8;        // columns loaded left and right of the tile (16-byte aligned x)
constexpr int BW = TW + 2 * PADW;   // TMA box width
constexpr int QP = BW + 2;     // row pitch of the h-pass result (2 mod 32 avoids bank conflicts)
constexpr int RHS = 5;         // output rows per h-pass item (divides TH)
constexpr int NTHR = 128;
constexpr int kMinBlocks = 3;  // resident CTAs per SM the register allocation targets

// Four pairs of float32 values to columns wbase .. wbase + 7 of an internal-layout row (pitch a
// multiple of 32, wbase of 8): two 16-byte stores when all eight columns are below W, else one
// value at a time.
__device__ __forceinline__ void st_pairs(float* o, const float2 p[4], int wbase, int W) {
    if (wbase + 8 <= W) {
        reinterpret_cast<float4*>(o)[0] = make_float4(p[0].x, p[0].y, p[1].x, p[1].y);
        reinterpret_cast<float4*>(o)[1] = make_float4(p[2].x, p[2].y, p[3].x, p[3].y);
    } else {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            if (wbase + 2 * m < W) o[2 * m] = p[m].x;
            if (wbase + 2 * m + 1 < W) o[2 * m + 1] = p[m].y;
        }
    }
}

template <int RT, int RH, int RW, typename TS, typename TVO, bool OUT_X>
struct Cfg {
    static constexpr int BH = TH + 2 * RH;                // TMA box height
    static constexpr int NSTAGE = 2;      // frame t, and the next ones in flight
    static constexpr int BOX_BYTES = (BW * BH * (int)sizeof(TS) + 127) / 128 * 128;
    static constexpr int STAGE_BYTES = 2 * BOX_BYTES;     // v then f
    static constexpr int Q_BYTES = 3 * TH * QP * 4;       // one h-pass result; two are kept
    static constexpr int SMEM = NSTAGE * STAGE_BYTES + 2 * Q_BYTES + NSTAGE * 8 + 128;
    static constexpr int CP_LO = (PADW - RW) / 2;         // first column pair the w-pass needs
    static constexpr int CP_HI = (PADW + TW + RW + 1) / 2;
    static constexpr int NCP = CP_HI - CP_LO;
    static constexpr int NHITEMS = NCP * (TH / RHS);
    static constexpr int ODD = RW & 1;
    static constexpr int NVAL = 8 + 2 * RW + ODD;         // w-pass window values (aligned start)
    static constexpr int NPAIR = (NVAL + 1) / 2;
    static_assert(NHITEMS <= NTHR, "h-pass items must fit the CTA");
    static_assert(TH % RHS == 0 && TH <= 16, "tile rows: a multiple of the h-pass item, at most 16");
    static_assert(RW <= PADW, "halo wider than the loaded pad");
};

struct Params {
    Geom g;
    float inv_alpha, p;
    float2 gt[2 * kMaxRT + 1], gh[2 * kMaxRH + 1], gw[2 * kMaxRW + 1];   // taps as (g, g) pairs
    int tchunk;
    const double* acc_in;
    double* acc_out;
    int* flags;
    void* out;        // next state (internal pitch) or x~ (caller layout)
    const void* f;    // f in global memory (internal pitch), read by the epilogue
    const float* s;   // separate unary map S_m (SEP kernels), or the state V_k (MODE 5); float32,
                      // internal pitch
    void* out2;       // second output: the record x~ (MODE 4) or Q (MODEs 5 and 6)
    // MODE 7 only: term group j of the exact kernel's series
    int exj;
    float exc[3];     // c_{3j}, c_{3j+1}, c_{3j+2}
    unsigned* maxkey; // MODE 8: atomicMax of the order key of the largest output
    bool nan_key;     // MODE 8: a NaN among the outputs makes the key a NaN's
};

// SEP and MODE as at iter_stream (iter_stream.cuh).
template <int RT, int RH, int RW, typename TS, typename TVO, bool OUT_X, bool SEP, int MODE>
__global__ void __launch_bounds__(NTHR, kMinBlocks)
iter_tile(const __grid_constant__ CUtensorMap mv, const __grid_constant__ CUtensorMap mf, const __grid_constant__ Params P) {
    using C = Cfg<RT, RH, RW, TS, TVO, OUT_X>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + (-smem_u32(smem_raw) & 127u);   // an offset keeps the address space
    float* Qbuf = reinterpret_cast<float*>(smem + C::NSTAGE * C::STAGE_BYTES);   // [2][3][TH][QP]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::NSTAGE * C::STAGE_BYTES + 2 * C::Q_BYTES);

    const int tid = threadIdx.x;
    const Geom g = P.g;
    const int w0 = blockIdx.x * TW, h0 = blockIdx.y * TH;
    const int t0 = blockIdx.z * P.tchunk;
    const int t1 = min(t0 + P.tchunk, g.T);
    // Frames before t = 0 are zero (zero padding): they would add exactly nothing to the
    // t-filter state, so the first chunk starts at frame 0.  Frames after the last are still
    // streamed, to flush the last rt output frames.
    const int tstart = max(t0 - RT, 0), tend = t1 + RT;

    auto stage_v = [&](int frame) -> const TS* {
        return reinterpret_cast<const TS*>(smem + ((frame - tstart) % C::NSTAGE) * C::STAGE_BYTES);
    };
    auto stage_f = [&](int frame) -> const TS* {
        return reinterpret_cast<const TS*>(smem + ((frame - tstart) % C::NSTAGE) * C::STAGE_BYTES + C::BOX_BYTES);
    };
    int next_issue = tstart;         // thread 0: frames [tstart, next_issue) have been requested
    auto issue = [&](int frame) {   // thread 0 only
        next_issue = frame + 1;
        const int st = (frame - tstart) % C::NSTAGE;
        unsigned char* dst = smem + st * C::STAGE_BYTES;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive_expect_tx(&bars[st], 2u * (uint32_t)(BW * C::BH * sizeof(TS)));
        tma_load_3d(dst, &mv, &bars[st], w0 - PADW, h0 - RH, frame);
        tma_load_3d(dst + C::BOX_BYTES, &mf, &bars[st], w0 - PADW, h0 - RH, frame);
    };

    // 1/||x~_k|| comes from one thread of the last warp (an FP64 chain of over a microsecond) while
    // thread 0 requests the first frames: 1.7 us less for a launch of a few frames
    __shared__ float snorm;
    wait_previous_grid();
    if (tid == NTHR - 32) snorm = inv_norm_from(P.acc_in, P.flags);
    if (tid == 0) {
        for (int i = 0; i < C::NSTAGE; ++i) mbar_init(&bars[i], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int i = 0; i < C::NSTAGE - 1 && tstart + i < tend; ++i) issue(tstart + i);
    }
    __syncthreads();
    const float2 s2 = f2(snorm);

    // thread roles
    const int lane = tid & 31, warp = tid >> 5;
    const int wr = warp * 4 + ((lane & 15) >> 2);          // w-pass / epilogue row in the tile
    const int wcs = ((lane >> 4) << 2) | (lane & 3);        // its 8-column segment
    const bool hitem = tid < C::NHITEMS;
    const int hcp = C::CP_LO + tid % C::NCP;                // h-pass column pair
    const int hseg = tid / C::NCP;                          // h-pass row segment

    // the filter taps, copied once from the kernel parameters (measured ~1-2 % faster than reading
    // the parameter bank at every use)
    float2 ghr[2 * RH + 1], gwr[2 * RW + 1], gtr[2 * RT + 1];
#pragma unroll
    for (int d = 0; d <= 2 * RH; ++d) ghr[d] = P.gh[d];
#pragma unroll
    for (int d = 0; d <= 2 * RW; ++d) gwr[d] = P.gw[d];
#pragma unroll
    for (int d = 0; d <= 2 * RT; ++d) gtr[d] = P.gt[d];
    // t-filter in transposed direct form: for each of the 3 signals and 4 column pairs the
    // 2rt running partial sums of the 2rt+1-tap filter; with x[n] the w-filtered frame n and
    // g_j = gt[2rt - j], the output y[n] = sum_j g_j x[n - j] is the t-filtered frame n - rt.
    float2 st[2 * RT][3][4];
#pragma unroll
    for (int a = 0; a < 2 * RT; ++a)
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int m = 0; m < 4; ++m) st[a][k][m] = make_float2(0.f, 0.f);
    float2 part = make_float2(0.f, 0.f);
    float tmax = 0.f;   // MODE 8: the largest output so far (outputs are >= 0)
    bool ok = true;

#pragma unroll 1
    for (int tt = tstart; tt < tend; ++tt) {
        // The stage of frame tt+NSTAGE-1 last held frame tt-1, whose h-pass every thread
        // finished before the previous step's barrier.
        if (tid == 0 && tt + C::NSTAGE - 1 < tend) issue(tt + C::NSTAGE - 1);
        float* Q = Qbuf + ((tt - tstart) & 1) * (3 * TH * QP);
        const int to = tt - RT;          // output frame of this step
        const int h = h0 + wr;
        const int wbase = w0 + wcs * 8;
        // f of the output frame for the epilogue, requested now so that its latency hides
        // behind the two spatial passes.  Outside the volume f is taken as 0, so those
        // positions give x~ = 0 and add nothing to the norm (row padding is not relied on).
        float2 fo[4];
        float2 so[(SEP || MODE == 5) ? 4 : 1];
#pragma unroll
        for (int m = 0; m < 4; ++m) fo[m] = make_float2(0.f, 0.f);
#pragma unroll
        for (int m = 0; m < ((SEP || MODE == 5) ? 4 : 1); ++m) so[m] = make_float2(0.f, 0.f);
        if (to >= t0 && h < g.H && wr < TH) {
            const TS* fg = reinterpret_cast<const TS*>(P.f) + ((int64_t)to * g.H + h) * g.pitch + wbase;
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                if (wbase + 2 * m + 1 < g.W) fo[m] = ld_pair(fg + 2 * m);
                else if (wbase + 2 * m < g.W) fo[m].x = ldf(fg + 2 * m);
            }
            if constexpr (SEP || MODE == 5) {
                const float* sg = P.s + ((int64_t)to * g.H + h) * g.pitch + wbase;
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if (wbase + 2 * m + 1 < g.W) so[m] = ld_pair(sg + 2 * m);
                    else if (wbase + 2 * m < g.W) so[m].x = sg[2 * m];
                }
            }
        }
        const uint32_t parity = (uint32_t)(((tt - tstart) / C::NSTAGE) & 1);
        const bool arrived = mbar_wait_bounded(&bars[(tt - tstart) % C::NSTAGE], parity);
        // ---------------- h-pass: raw stage -> Q[3][TH][QP]
        if (hitem && arrived) {
            const TS* sv = stage_v(tt) + (hseg * RHS) * BW + 2 * hcp;
            const TS* sf = stage_f(tt) + (hseg * RHS) * BW + 2 * hcp;
            float2 acc[RHS][3];
#pragma unroll
            for (int o = 0; o < RHS; ++o)
#pragma unroll
                for (int k = 0; k < 3; ++k) acc[o][k] = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < RHS + 2 * RH; ++j) {
                const float2 v = ld_pair(sv + j * BW);
                const float2 f = ld_pair(sf + j * BW);
                const float2 z3 = mul2(f, v);
                const float2 z2 = mul2(f, z3);
#pragma unroll
                for (int o = 0; o < RHS; ++o) {
                    const int d = j - o;
                    if (d >= 0 && d <= 2 * RH) {
                        const float2 gd = ghr[d];
                        acc[o][0] = fma2(v, gd, acc[o][0]);
                        acc[o][1] = fma2(z2, gd, acc[o][1]);
                        acc[o][2] = fma2(z3, gd, acc[o][2]);
                    }
                }
            }
#pragma unroll
            for (int o = 0; o < RHS; ++o)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    *reinterpret_cast<float2*>(Q + (k * TH + hseg * RHS + o) * QP + 2 * hcp) = acc[o][k];
        }
        // The only barrier of the step: Q of this frame is complete, and every thread is done
        // with the h-pass of the previous frame (whose stage the next copy overwrites).
        if (__syncthreads_or(!arrived)) {
            ok = false;
            break;
        }
        // ---------------- w-pass: Q -> x[n], then the t-filter update
        float2 y[3][4];
        if (wr < TH) {
            const int a0 = PADW + wcs * 8 - RW - C::ODD;   // even
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float* qr = Q + (k * TH + wr) * QP + a0;
                float2 pa[C::NPAIR];
#pragma unroll
                for (int j = 0; j < C::NPAIR; ++j) pa[j] = ld_pair(qr + 2 * j);
                float2 acc[4];   // four independent chains (one per column pair)
#pragma unroll
                for (int m = 0; m < 4; ++m) acc[m] = make_float2(0.f, 0.f);
#pragma unroll
                for (int d = 0; d <= 2 * RW; ++d) {
                    const float2 gd = gwr[d];
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const int q = 2 * m + d + C::ODD;
                        if (q & 1) {   // odd-aligned pair: two scalar FMAs
                            acc[m].x = fmaf(pa[q >> 1].y, gd.x, acc[m].x);
                            acc[m].y = fmaf(pa[(q >> 1) + 1].x, gd.x, acc[m].y);
                        } else {
                            acc[m] = fma2(pa[q >> 1], gd, acc[m]);
                        }
                    }
                }
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float2 x = acc[m];
                    y[k][m] = fma2(x, gtr[2 * RT], st[0][k][m]);
#pragma unroll
                    for (int j = 0; j < 2 * RT - 1; ++j) st[j][k][m] = fma2(x, gtr[2 * RT - 1 - j], st[j + 1][k][m]);
                    st[2 * RT - 1][k][m] = mul2(x, gtr[0]);
                }
            }
        }
        // ---------------- Eq. 7 combination for frame to = tt - RT
        if (to >= t0 && wr < TH) {
            float2 outv[4];
            float2 outq[(MODE >= 4 && MODE <= 6) ? 4 : 1];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const float2 fv = fo[m];
                const float2 sv = SEP ? so[SEP ? m : 0] : fv;
                const float2 u = make_float2(unary_pow_fast<true>(sv.x, P.p), unary_pow_fast<true>(sv.y, P.p));
                const float2 e = fma2(make_float2(-fv.x, -fv.y), fv, f2(P.inv_alpha));   // 1/alpha - f^2
                if constexpr (MODE == 7) {
                    float2 F = make_float2(1.f, 1.f);
                    const float2 f3 = mul2(fv, mul2(fv, fv));
                    for (int i = 0; i < P.exj; ++i) F = mul2(F, f3);
                    const float2 inner = fma2(mul2(fv, f2(P.exc[2])), y[1][m], mul2(f2(P.exc[1]), y[2][m]));
                    outv[m] = mul2(mul2(s2, F), fma2(fv, inner, mul2(f2(P.exc[0]), y[0][m])));
                } else if constexpr (MODE == 0 || MODE == 4 || MODE == 6 || MODE == 8) {
                    float2 B = fma2(e, y[0][m], make_float2(-y[1][m].x, -y[1][m].y));
                    B = fma2(mul2(f2(2.f), fv), y[2][m], B);
                    const float2 xt = mul2(mul2(s2, u), B);
                    part = fma2(xt, xt, part);
                    if constexpr (MODE == 8) tmax = fmaxf(tmax, fmaxf(xt.x, xt.y));
                    outv[m] = (OUT_X || MODE == 8) ? xt : mul2(u, xt);
                    if constexpr (MODE == 4) outq[m] = xt;
                    if constexpr (MODE == 6) {
                        const float2 a1 = fma2(f2(P.p), e, mul2(f2(-2.f), mul2(fv, fv)));
                        const float2 a3 = mul2(f2(2.f * (P.p + 1.f)), fv);
                        const float2 Q = fma2(a1, y[0][m], mul2(f2(-P.p), y[1][m]));
                        outq[MODE == 6 ? m : 0] = mul2(s2, fma2(a3, y[2][m], Q));
                    }
                } else {
                    const float2 a1 = fma2(f2(P.p), e, mul2(f2(-2.f), mul2(fv, fv)));
                    const float2 a3 = mul2(f2(2.f * (P.p + 1.f)), fv);
                    float2 Q = fma2(a1, y[0][m], mul2(f2(-P.p), y[1][m]));
                    Q = mul2(s2, fma2(a3, y[2][m], Q));
                    if constexpr (MODE == 1) {
                        outv[m] = Q;
                    } else {
                        float2 B = fma2(e, y[0][m], make_float2(-y[1][m].x, -y[1][m].y));
                        B = fma2(mul2(f2(2.f), fv), y[2][m], B);
                        outv[m] = mul2(mul2(u, u), B);
                        part = fma2(so[MODE == 5 ? m : 0], B, part);
                        outq[MODE == 5 ? m : 0] = Q;
                    }
                }
            }
            if constexpr (MODE == 4 || MODE == 6) {
                if (h < g.H) {
                    float* o2 = reinterpret_cast<float*>(P.out2) + ((int64_t)to * g.H + h) * g.pitch + wbase;
                    st_pairs(o2, outq, wbase, g.W);
                }
            }
            if constexpr (MODE == 7) {
                if (h < g.H) {
                    float* o = reinterpret_cast<float*>(P.out) + ((int64_t)to * g.H + h) * g.pitch + wbase;
                    if (P.exj > 0) {   // the terms so far
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            if (wbase + 2 * m + 1 < g.W) outv[m] = __fadd2_rn(outv[m], ld_pair(o + 2 * m));
                            else if (wbase + 2 * m < g.W) outv[m].x += o[2 * m];
                        }
                    }
                    st_pairs(o, outv, wbase, g.W);
                }
            } else if constexpr (MODE == 1 || MODE == 5) {
                if (h < g.H) {
                    float* o = reinterpret_cast<float*>(P.out) + ((int64_t)to * g.H + h) * g.pitch + wbase;
                    st_pairs(o, outv, wbase, g.W);
                    if constexpr (MODE == 5) {
                        float* o2 = reinterpret_cast<float*>(P.out2) + ((int64_t)to * g.H + h) * g.pitch + wbase;
                        st_pairs(o2, outq, wbase, g.W);
                    }
                }
            } else
            if (h < g.H) {
                if (OUT_X) {
                    // caller layout: rows of W values, 8-byte aligned when W is even (and the
                    // caller's base is), then one 8-byte store per pair
                    float* o = reinterpret_cast<float*>(P.out) + ((int64_t)to * g.H + h) * g.W + wbase;
                    if (wbase + 8 <= g.W && (reinterpret_cast<uintptr_t>(o) & 7) == 0) {
#pragma unroll
                        for (int m = 0; m < 4; ++m) reinterpret_cast<float2*>(o)[m] = outv[m];
                    } else {
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            if (wbase + 2 * m < g.W) o[2 * m] = outv[m].x;
                            if (wbase + 2 * m + 1 < g.W) o[2 * m + 1] = outv[m].y;
                        }
                    }
                } else {
                    TVO* o = reinterpret_cast<TVO*>(P.out) + ((int64_t)to * g.H + h) * g.pitch + wbase;
                    if (wbase + 8 <= g.W) {
                        if constexpr (sizeof(TVO) == 4) {
                            reinterpret_cast<float4*>(o)[0] = make_float4(outv[0].x, outv[0].y, outv[1].x, outv[1].y);
                            reinterpret_cast<float4*>(o)[1] = make_float4(outv[2].x, outv[2].y, outv[3].x, outv[3].y);
                        } else {
                            __nv_bfloat162 b[4];
#pragma unroll
                            for (int m = 0; m < 4; ++m) b[m] = __float22bfloat162_rn(outv[m]);
                            *reinterpret_cast<uint4*>(o) = *reinterpret_cast<const uint4*>(b);
                        }
                    } else {
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            if (wbase + 2 * m < g.W) stf(o + 2 * m, outv[m].x);
                            if (wbase + 2 * m + 1 < g.W) stf(o + 2 * m + 1, outv[m].y);
                        }
                    }
                }
            }
        }
    }
    // Only now: blocks of the next launch placed while this one's still hold their SMs pile up on the
    // emptier ones (13x152x58 at (2,7,7): 8.9 -> 10.8 us per step when allowed at the start).
    allow_next_grid();
    if (!ok) {
        if (tid == 0) {
            atomicOr(P.flags, kFlagTimeout);
            // let copies still in flight land before the CTA's shared memory goes away: for each
            // stage, wait (bounded) for the phase of the last frame requested into it
            for (int i = 0; i < C::NSTAGE && tstart + i < next_issue; ++i) {
                const int last = i + ((next_issue - 1 - tstart - i) / C::NSTAGE) * C::NSTAGE;   // relative frame
                mbar_wait_bounded(&bars[i], (uint32_t)((last / C::NSTAGE) & 1));
            }
        }
        return;
    }
    const double tot = block_sum((double)part.x + (double)part.y);
    if (tid == 0 && P.acc_out) atomicAdd(P.acc_out, tot);
    if constexpr (MODE == 8) {
        __shared__ unsigned wmax[NTHR / 32];
        const unsigned key = P.nan_key && isnan(part.x + part.y) ? kNanKey : order_key(tmax);
        const unsigned kmax = __reduce_max_sync(0xffffffffu, key);
        if (lane == 0) wmax[warp] = kmax;
        __syncthreads();
        if (tid == 0) {
            unsigned m = wmax[0];
            for (int i = 1; i < NTHR / 32; ++i) m = max(m, wmax[i]);
            if (P.maxkey) atomicMax(P.maxkey, m);
        }
    }
}

template <int RT, int RH, int RW, typename TS, typename TVO, bool OUT_X, bool SEP, int MODE>
static bool launch_t(const StepArgs& a) {
    using C = Cfg<RT, RH, RW, TS, TVO, OUT_X>;
    constexpr bool bf = sizeof(TS) == 2;
    const Geom& g = a.g;
    CUtensorMap mv, mf;
    if (!make_step_map(&mv, a.vin, bf, g, BW, C::BH) || !make_step_map(&mf, a.f, bf, g, BW, C::BH)) return false;
    auto kern = iter_tile<RT, RH, RW, TS, TVO, OUT_X, SEP, MODE>;
    static std::atomic<int> slots_per_sm{1};
    static std::atomic<unsigned long long> attr_set{0};   // devices on which the attribute is set
    if (!(attr_set & device_bit())) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) != cudaSuccess) return false;
        int nb = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, NTHR, C::SMEM);
        slots_per_sm = nb > 0 ? nb : 1;
        attr_set |= device_bit();
    }
    Params P;
    P.g = g;
    P.inv_alpha = a.inv_alpha;
    P.p = a.p;
    // the taps, and zeros where the kernel's radius is wider
    auto fill = [](float2* d, int R, const float* g1, int r) {
        for (int i = -R; i <= R; ++i) {
            const float t = i >= -r && i <= r ? g1[r + i] : 0.f;
            d[R + i] = make_float2(t, t);
        }
    };
    fill(P.gt, RT, a.tp.gt, a.tp.rt);
    fill(P.gh, RH, a.tp.gh, a.tp.rh);
    fill(P.gw, RW, a.tp.gw, a.tp.rw);
    P.f = a.f;
    P.s = a.s32;
    P.out2 = a.out2;
    P.exj = a.ex ? a.ex->j : 0;
    for (int i = 0; i < 3; ++i) P.exc[i] = a.ex ? a.ex->c[i] : 0.f;
    P.maxkey = a.maxkey;
    P.nan_key = a.tp.rt != RT || a.tp.rh != RH || a.tp.rw != RW;
    const int tx = (g.W + TW - 1) / TW, ty = (g.H + TH - 1) / TH;
    P.tchunk = tile_chunk(g.T, tx * ty, slots_per_sm * num_sms(), RT);
    P.acc_in = a.acc_in;
    P.acc_out = a.acc_out;
    P.flags = a.flags;
    P.out = a.out;
    dim3 grid(tx, ty, (g.T + P.tchunk - 1) / P.tchunk);
    launch_after_previous(kern, grid, NTHR, C::SMEM, a.s, mv, mf, P);
    count_launches(1);
    return true;
}

template <int RT, int RH, int RW>
struct Kernel {
    template <typename TS, typename TVO, bool OUT_X, bool SEP, int MODE>
    static bool launch(const StepArgs& a) {
        return launch_t<RT, RH, RW, TS, TVO, OUT_X, SEP, MODE>(a);
    }
};

}  // namespace tile
}  // namespace sfseg
