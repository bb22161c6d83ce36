// iter_stream.cuh -- the power-iteration step of Eq. 7 with a compiled radius, written for sm_103a:
// the kernel for all but small volumes (those: iter_tile.cuh).
//
// One persistent CTA per SM (16 warps: 4 h-pass, 8 w-pass, 4 for copies and the norm) streams frames of
// 18 x 112 tiles of (h, w) along t.  Its warps have roles that run at the same time, connected by rings in
// shared memory:
//   - Copies.  One thread keeps TMA copies of the raw halo boxes of v (= u x~) and f (18 + 2rh rows
//     of 128 columns) in flight, three frames deep; zero fill outside the volume is the zero padding,
//     also for whole frames after the last.
//   - h-pass, warps 0..3: a thread takes a column pair and 9 output rows (64 pairs x 2 row groups);
//     it walks down the 9 + 2rh input rows once, each loaded a row ahead, forms the three signals z1 = v,
//     z2 = f^2 v, z3 = f v of each, and accumulates them into its 9 x 3 outputs with packed FP32 FMAs
//     (FFMA2, one per column pair).  The result goes to a ring of two frames of [3][18][132] floats.
//   - w-pass, warps 4..11: a thread takes 8 output columns of one row (14 x 18 = 252 of 256 threads); it
//     loads its window of the h-pass result as 16-byte pieces (the odd taps run as two scalar FMAs:
//     rebuilding their pairs for packed ones costs more moves) and feeds the three w-filtered signals
//     straight into the t-filter, kept in registers in transposed direct form (2rt running partial sums
//     per value, no frame ring to index).
//   - Epilogue, same threads: Eq. 7 combination for the frame rt behind, with f of that frame from a
//     TMA-fed tile, the Eq. 8 norm partial, and the next state into a tile that a TMA store writes
//     out (which clips at the volume's edges, so no lane tests its column).
// Every hand-over is an mbarrier of the ring slot concerned: no barrier stops all warps.
//
// Why this shape.  The step is bound by the FP32 pipe (105 FMA per voxel at (2,7,7) against 12 bytes), so
// what counts is the work that is not algorithmic and the time the pipe idles.  Against the small-volume
// kernel's three CTAs of 4 warps per SM, each on a 15 x 64 tile with all warps doing the h-pass and then
// the w-pass between CTA barriers: 128 columns are h-filtered for 112 (there 80 for 64), 23 input rows read
// and multiplied per 9 output rows (there 19 per 5), and an SM's work ends at one time (there the oldest
// of its CTAs is favoured and the last runs alone: 121, 145 and 175 us in one wave).
// Two facts of the instruction set decide the rest.  A packed FMA takes 3 clocks when its three register
// pairs are all new and 2 when one is a constant or was read by the instruction before it (measured): taps
// stay in the parameter constants.  And a shared-memory pointer rounded up through an integer loses its
// address space, so that every access is a generic one: the alignment is an offset (152 us per step; 184
// through an integer).
// Measured per step, small-volume kernel / this one: (2,7,7) 64x480x854 168 / 138 us (the algorithmic
// multiply-adds alone 68 us), 120x1080x1920 1170 here; (1,3,3) 64x480x854 111 / 94.
#pragma once

#include "order_key.cuh"
#include "step.h"
#include "tma.cuh"

namespace sfseg {
namespace stream {

constexpr int TW = 112;        // tile columns: 14 segments of 8
constexpr int TH = 18;         // tile rows: 14 x 18 = 252 of the 256 w-pass threads
constexpr int RHS = 9;         // output rows of an h-pass thread
constexpr int PADW = 8;        // columns loaded left and right of the tile (16-byte aligned x)
constexpr int BW = TW + 2 * PADW;   // halo box width: 64 column pairs
constexpr int QP = BW + 4;     // row pitch of the h-pass result: the 16-byte window loads of 4
                               // segments x 2 rows touch all 32 banks once
constexpr int NH = 128, NW = 256;   // threads of the h-pass and of the w-pass
constexpr int NTHR = NH + NW + 128; // and a warpgroup whose first two warps hold a copy thread each
// Registers per thread of the three roles; the sum over the four warpgroups is the 4 x 128 that the
// block is launched with.  The w-pass keeps 96 of t-filter state at rt = 2.
constexpr int kRegsW = 184, kRegsH = 112, kRegsIO = 32;
static_assert(2 * kRegsW + kRegsH + kRegsIO <= 4 * 128, "register split");
static_assert(kRegsW >= 128 && kRegsH <= 128 && kRegsIO <= 128 && kRegsW % 8 == 0 && kRegsH % 8 == 0 &&
                  kRegsIO % 8 == 0,
              "setmaxnreg.inc only raises and .dec only lowers a warp's registers, by multiples of 8");
constexpr int NSTAGE = 3;      // halo boxes in flight
constexpr int NQ = 2;          // h-pass results in the ring (three: the same time)
constexpr int NSEG = TW / 8;
constexpr int kFold = 32;      // frames whose squares are summed in float32

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int x, int y, int z) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(map), "r"(x),
                 "r"(y), "r"(z), "r"(smem_u32(src))
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
template <int N>
__device__ __forceinline__ void regs_up() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void regs_down() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

// The eight columns of a w-pass thread, as four pairs, from and to a tile in shared memory.
__device__ __forceinline__ void ld_cols(const float* t, float2 (&o)[4]) {
    const float4 a = reinterpret_cast<const float4*>(t)[0], b = reinterpret_cast<const float4*>(t)[1];
    o[0] = make_float2(a.x, a.y);
    o[1] = make_float2(a.z, a.w);
    o[2] = make_float2(b.x, b.y);
    o[3] = make_float2(b.z, b.w);
}
__device__ __forceinline__ void ld_cols(const __nv_bfloat16* t, float2 (&o)[4]) {
    const uint4 r = *reinterpret_cast<const uint4*>(t);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&r);
#pragma unroll
    for (int m = 0; m < 4; ++m) o[m] = __bfloat1622float2(h[m]);
}
__device__ __forceinline__ void st_cols(float* t, const float2 (&v)[4]) {
    reinterpret_cast<float4*>(t)[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    reinterpret_cast<float4*>(t)[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
}
__device__ __forceinline__ void st_cols(__nv_bfloat16* t, const float2 (&v)[4]) {
    __nv_bfloat162 b[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) b[m] = __float22bfloat162_rn(v[m]);
    *reinterpret_cast<uint4*>(t) = *reinterpret_cast<const uint4*>(b);
}

// The modes' extra tiles: a second input of the output frame (the separate unary map, V_k, or the
// exact series' sum so far) and a second output.
template <bool SEP, int MODE>
struct Extra {
    static constexpr bool IN2 = SEP || MODE == 5 || MODE == 7;
    static constexpr bool OUT2 = MODE >= 4 && MODE <= 6;
};

template <int RT, int RH, int RW, typename TS, typename TVO, bool OUT_X, bool SEP, int MODE>
struct Cfg {
    using E = Extra<SEP, MODE>;
    static constexpr int BH = TH + 2 * RH;                // halo box height
    static constexpr int up(int b) { return (b + 127) / 128 * 128; }
    static constexpr int BOX = up(BW * BH * (int)sizeof(TS));
    static constexpr int STAGE = 2 * BOX;                 // v then f
    static constexpr int Q = up(3 * TH * QP * 4);         // one h-pass result
    static constexpr int FT = up(TH * TW * (int)sizeof(TS));     // f of the output frame
    static constexpr int T32 = up(TH * TW * 4);
    static constexpr int OT = OUT_X ? 0 : up(TH * TW * (int)sizeof(TVO));
    static constexpr int O_Q = NSTAGE * STAGE;
    static constexpr int O_F = O_Q + NQ * Q;
    static constexpr int O_I2 = O_F + 2 * FT;
    static constexpr int O_O = O_I2 + (E::IN2 ? 2 * T32 : 0);
    static constexpr int O_O2 = O_O + 2 * OT;
    static constexpr int O_BAR = O_O2 + (E::OUT2 ? 2 * T32 : 0);
    // full[NSTAGE], empty[NSTAGE], qfull[NQ], qempty[NQ], ffull[2], done[2], oempty[2], nready
    static constexpr int NBAR = 2 * NSTAGE + 2 * NQ + 7;
    static constexpr int SMEM = O_BAR + NBAR * 8 + 128;
    static constexpr int CP_LO = (PADW - RW) / 2;         // first column pair the w-pass needs
    static constexpr int NCP = (PADW + TW + RW + 1) / 2 - CP_LO;
    // The w-pass window starts OFF columns before the thread's first: 16-byte aligned.
    static constexpr int OFF = (RW + 3) / 4 * 4;
    static constexpr int NPAIR = (OFF + 8 + RW + 3) / 4 * 2;
    static_assert(NCP <= NH / 2 && 2 * RHS == TH, "h-pass items");
    static_assert(NSEG * TH <= NW && NSEG == 14 && TH == 18, "w-pass items (the lane map below)");
    static_assert(RW <= PADW && OFF <= PADW, "halo wider than the loaded pad");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

struct Params {
    Geom g;
    float inv_alpha, p;
    float2 gt[kMaxRT + 1], gh[kMaxRH + 1], gw[kMaxRW + 1];   // taps of offsets 0..r as (g, g) pairs
    int tx, tiles, whole;   // tile columns, tiles, tiles that each CTA streams whole
    const double* acc_in;
    double* acc_out;
    int* flags;
    void* out;        // OUT_X: x~ (caller layout)
    // MODE 7 only: term group j of the exact kernel's series (see below)
    int exj;
    float exc[3];     // c_{3j}, c_{3j+1}, c_{3j+2}
    unsigned* maxkey; // MODE 8: atomicMax of the order key of the largest output
    bool nan_key;     // MODE 8: a NaN among the outputs makes the key a NaN's
};

// The tensor maps: halo boxes of v and f; tiles of f, of the second input, and of both outputs.
struct Maps {
    CUtensorMap v, f, fc, in2, out, out2;
};

// The frames a CTA streams, in runs of one tile each: `whole` tiles from first to last frame (all
// CTAs then stand at the same frame, so that neighbouring tiles' halos are still in L2), then its
// share of the output frames of the tiles left over, cut anywhere (each cut costs 2 rt frames).
struct Run {
    int w0, h0, t0, t1;      // tile origin, output frames [t0, t1)
};
__device__ __forceinline__ bool run_of(const Params& P, int s, Run& r) {
    const int T = P.g.T, b = blockIdx.x, G = gridDim.x;
    int tile;
    if (s < P.whole) {
        tile = s * G + b;
        r.t0 = 0, r.t1 = T;
    } else {   // the leftover tiles' output frames, [pos, end) of them this CTA's
        const long long rest = (long long)(P.tiles - P.whole * G) * T;
        const long long end = rest * (b + 1) / G;
        long long pos = rest * b / G;
        if (s > P.whole) pos = (pos / T + (s - P.whole)) * T;
        if (pos >= end) return false;
        const int q = (int)(pos / T);
        tile = P.whole * G + q;
        r.t0 = (int)(pos - (long long)q * T);
        r.t1 = (int)min((long long)T, r.t0 + (end - pos));
    }
    r.h0 = tile / P.tx * TH;
    r.w0 = tile % P.tx * TW;
    return true;
}

// SEP: the unary term u = s^p comes from a separate map S_m (Eq. 9 with its own channels)
// instead of from f.  MODE 0 is the power-iteration step; MODE 4 is the same step that also
// records x~ (internal layout, out2) for the adjoint.  MODEs 1 and 5 serve the adjoint
// (kernels_bwd.cu): with c_0, c_1, c_2 the three filtered signals of the input v (G*v,
// G*(f^2 v), G*(f v)), Q = a1 c_0 - p c_1 + a3 c_2 with a1 = p (1/alpha - f^2) - 2 f^2,
// a3 = 2 (p + 1) f (the f-derivative weights of the step).  MODE 1 stores s Q.  MODE 5 stores
// G = u^2 B (B the Eq. 7 bracket, so G = u A z for v = u z) and Q, and adds sum V_k B over its
// voxels to acc_out, with V_k = u x~_k the second input (so that <x_k, A z> = s_k sum V_k B needs
// no division by u).  MODE 6 is the step (MODE 0, the state to out) that also stores s Q to out2:
// the adjoint's recomputation and Q-pass share the filtering of V_k.  MODE 7 serves the exact
// (Eq. 1) kernel, exp(-a (f_i - f_j)^2) = e^{-a g_i^2} e^{-a g_j^2} sum_n c_n g_i^n g_j^n with
// c_n = (2a)^n / n! and g = f - c for any constant c: with g in f's place and the input v = g^{3j} w,
// its three filtered signals are the series terms n = 3j (G*v), 3j + 1 (G*(g v)) and 3j + 2
// (G*(g^2 v)); it adds t = s g^{3j} (c_{3j} G*v + g (c_{3j+1} G*(g v) + g c_{3j+2} G*(g^2 v))) to out
// (writes it when j = 0).  All in the internal layout.  MODE 8 writes x~ in the
// internal layout and adds the largest of its outputs to P.maxkey (atomicMax of the order key, one per
// warp; nullable): the maximum a soft-binarisation step (Alg. 1 step 3) scales by, without a pass of its
// own.  fmaxf drops a NaN; for a radius without its own kernel, whose zero taps would spread it further
// than its neighbourhood, P.nan_key lets it through, as a maximum over the written outputs would (the sum
// of squares is a NaN exactly when an output was).  The last step of a power iteration is one too, without the key.
template <int RT, int RH, int RW, typename TS, typename TVO, bool OUT_X, bool SEP, int MODE>
__global__ void __launch_bounds__(NTHR, 1)
iter_stream(const __grid_constant__ Maps M, const __grid_constant__ Params P) {
    using C = Cfg<RT, RH, RW, TS, TVO, OUT_X, SEP, MODE>;
    using E = Extra<SEP, MODE>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // 128-byte aligned by an offset: rounding the pointer itself up through an integer would lose its
    // address space, and every access below would be a generic one
    unsigned char* smem = smem_raw + (-smem_u32(smem_raw) & 127u);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::O_BAR);   // [NSTAGE] halo boxes have landed
    uint64_t* empty = full + NSTAGE;    // [NSTAGE] the h-pass has read them
    uint64_t* qfull = empty + NSTAGE;   // [NQ] the h-pass result is complete
    uint64_t* qempty = qfull + NQ;   // [NQ] the w-pass has read it
    uint64_t* ffull = qempty + NQ;       // [2] the output frame's input tiles have landed
    uint64_t* done = ffull + 2;         // [2] the output frame is finished: tiles read, outputs written
    uint64_t* oempty = done + 2;        // [2] the output tile has been stored
    uint64_t* nready = oempty + 2;      // snorm is there
    __shared__ float snorm;
    __shared__ double red[NW];

    const int tid = threadIdx.x, lane = tid & 31;
    bool ok = true;
    if (tid == NH + NW) {
        for (int i = 0; i < NSTAGE; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], NH / 32);
        }
        for (int i = 0; i < NQ; ++i) {
            mbar_init(&qfull[i], NH / 32);
            mbar_init(&qempty[i], NW / 32);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&ffull[i], 1);
            mbar_init(&done[i], NW / 32);
            mbar_init(&oempty[i], 1);
        }
        mbar_init(nready, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_map(&M.v);
        prefetch_map(&M.f);
    } else if (tid == NH + NW + 32) {
        prefetch_map(&M.fc);
        if constexpr (!OUT_X) prefetch_map(&M.out);
    }
    allow_next_grid();
    __syncthreads();
    wait_previous_grid();

    // Frames outside the volume are zero: those before t = 0 would add exactly nothing to the t-filter
    // state, so a run starts at frame max(t0 - rt, 0); those after the last flush the last rt output
    // frames and go through the passes like the others.  (Branches around the passes for them cost
    // more than the passes: 480p at (2,7,7) 147.6 -> 154 us with one around the w-pass loads of a
    // signal, 156 us with one around the h-pass, 390 us with a flush step of its own, which spills.)
    if (tid >= NH + NW) {
        // ------------------------------------------------ copies
        regs_down<kRegsIO>();
        if (tid == NH + NW) {   // the halo boxes of v and f
            int st = 0, sp = 1, n = 0;   // the first NSTAGE slots are free
            Run r;
            for (int s = 0; ok && run_of(P, s, r); ++s) {
                for (int tt = max(r.t0 - RT, 0); tt < r.t1 + RT; ++tt) {
                    ok = mbar_wait_bounded(&empty[st], sp);
                    if (!ok) break;
                    unsigned char* dst = smem + st * C::STAGE;
                    fence_async();
                    mbar_arrive_expect_tx(&full[st], 2u * (uint32_t)(BW * C::BH * sizeof(TS)));
                    tma_load_3d(dst, &M.v, &full[st], r.w0 - PADW, r.h0 - RH, tt);
                    tma_load_3d(dst + C::BOX, &M.f, &full[st], r.w0 - PADW, r.h0 - RH, tt);
                    ++n;
                    if (++st == NSTAGE) st = 0, sp ^= 1;
                }
            }
            if (!ok)   // let the boxes still in flight land before the shared memory goes away
                for (int k = max(n - NSTAGE, 0); k < n; ++k)
                    mbar_wait_bounded(&full[k % NSTAGE], (uint32_t)(k / NSTAGE) & 1);
        } else if (tid == NH + NW + 32) {   // the output frames' input tiles and their stores
            const bool two = E::IN2 && (MODE != 7 || P.exj > 0);
            int n = 0;                       // output frames so far
            Run r, pr = {}, ppr = {};        // this frame's run, the last two frames' (t0: the frame)
            auto store = [&](const Run& o, int b) {
                if constexpr (!OUT_X) tma_store_3d(&M.out, smem + C::O_O + b * C::OT, o.w0, o.h0, o.t0);
                if constexpr (E::OUT2) tma_store_3d(&M.out2, smem + C::O_O2 + b * C::T32, o.w0, o.h0, o.t0);
                bulk_commit();
            };
            for (int s = 0; ok && run_of(P, s, r); ++s) {
                for (; r.t0 < r.t1; ++r.t0) {
                    const int b = n & 1;
                    if (n >= 2) {            // frame n - 2 is finished by every warp: its buffers
                        ok = mbar_wait_bounded(&done[b], (uint32_t)((n - 2) >> 1) & 1);
                        if (!ok) break;
                        store(ppr, b);
                    }
                    fence_async();
                    mbar_arrive_expect_tx(&ffull[b], (uint32_t)(TH * TW * sizeof(TS)) + (two ? TH * TW * 4u : 0u));
                    tma_load_3d(smem + C::O_F + b * C::FT, &M.fc, &ffull[b], r.w0, r.h0, r.t0);
                    if (two) tma_load_3d(smem + C::O_I2 + b * C::T32, &M.in2, &ffull[b], r.w0, r.h0, r.t0);
                    if (n >= 2) {
                        bulk_wait_read();
                        mbar_arrive(&oempty[b]);
                    }
                    ppr = pr, pr = r;
                    ++n;
                }
            }
            for (int k = max(n - 2, 0); ok && k < n; ++k) {
                ok = mbar_wait_bounded(&done[k & 1], (uint32_t)(k >> 1) & 1);
                if (ok) store(k == n - 1 ? pr : ppr, k & 1);
            }
            if (!ok)
                for (int k = max(n - 2, 0); k < n; ++k) mbar_wait_bounded(&ffull[k & 1], (uint32_t)(k >> 1) & 1);
            bulk_wait_read();
        } else if (tid == NH + NW + 64) {
            // 1/||x~_k||, an FP64 chain of over a microsecond, while the first frames are on their way
            snorm = inv_norm_from(P.acc_in, P.flags);
            mbar_arrive(nready);
        }
    } else if (tid < NH) {
        regs_down<kRegsH>();
        // ------------------------------------------------ h-pass: halo boxes -> Q[3][TH][QP]
        const int cp = C::CP_LO + tid % (NH / 2), seg = tid / (NH / 2);
        const bool item = tid % (NH / 2) < C::NCP;
        float2 ghr[RH + 1];
#pragma unroll
        for (int d = 0; d <= RH; ++d) ghr[d] = P.gh[d];
        int st = 0, sp = 0, q = 0, qp = 1;   // ring slots and phases (the first two Q slots are free)
        Run r;
        for (int s = 0; ok && run_of(P, s, r); ++s) {
#pragma unroll 1
            for (int n = r.t1 + RT - max(r.t0 - RT, 0); n > 0; --n) {
                ok = mbar_wait_bounded(&full[st], sp) && mbar_wait_bounded(&qempty[q], qp);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                if (item) {
                    const TS* sv = reinterpret_cast<const TS*>(smem + st * C::STAGE) + seg * RHS * BW + 2 * cp;
                    const TS* sf = reinterpret_cast<const TS*>(smem + st * C::STAGE + C::BOX) + seg * RHS * BW + 2 * cp;
                    float* Q = reinterpret_cast<float*>(smem + C::O_Q + q * C::Q) + seg * RHS * QP + 2 * cp;
                    float2 acc[RHS][3];
#pragma unroll
                    for (int o = 0; o < RHS; ++o)
#pragma unroll
                        for (int k = 0; k < 3; ++k) acc[o][k] = make_float2(0.f, 0.f);
                    float2 vn = ld_pair(sv), fn = ld_pair(sf);
#pragma unroll
                    for (int j = 0; j < RHS + 2 * RH; ++j) {
                        const float2 v = vn, f = fn;
                        if (j + 1 < RHS + 2 * RH) {
                            vn = ld_pair(sv + (j + 1) * BW);
                            fn = ld_pair(sf + (j + 1) * BW);
                        }
                        const float2 z3 = mul2(f, v);
                        const float2 z2 = mul2(f, z3);
#pragma unroll
                        for (int o = 0; o < RHS; ++o) {
                            const int d = j - o - RH;
                            if (d >= -RH && d <= RH) {
                                const float2 gd = ghr[d < 0 ? -d : d];
                                acc[o][0] = fma2(v, gd, acc[o][0]);
                                acc[o][1] = fma2(z2, gd, acc[o][1]);
                                acc[o][2] = fma2(z3, gd, acc[o][2]);
                            }
                        }
                        // an output row is complete once the input row rh below it is in
                        if (j >= 2 * RH) {
#pragma unroll
                            for (int k = 0; k < 3; ++k)
                                *reinterpret_cast<float2*>(Q + (k * TH + j - 2 * RH) * QP) = acc[j - 2 * RH][k];
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&empty[st]);
                    mbar_arrive(&qfull[q]);
                }
                if (++st == NSTAGE) st = 0, sp ^= 1;
                if (++q == NQ) q = 0, qp ^= 1;
            }
        }
    } else {
        // ------------------------------------------------ w-pass, t-filter, epilogue
        regs_up<kRegsW>();
        const int i = tid - NH;
        // lane map: blocks of 8 lanes cover 4 segments x 2 rows, the last two segments 2 x 4 rows
        // whose distances (0, 1, 4, 5) keep the block's 16-byte loads on distinct banks
        int row, seg;
        if (i < 216) {
            row = i / 24 * 2 + (i % 8) / 4;
            seg = i / 8 % 3 * 4 + i % 4;
        } else if (i < 248) {
            const int j = i - 216, c = j / 8, l = j % 8;
            row = c / 2 * 8 + c % 2 * 2 + (l / 2 % 2) + l / 4 * 4;
            seg = 12 + l % 2;
        } else {
            row = 16 + (i - 248) / 2 % 2;
            seg = 12 + i % 2;
        }
        const bool item = i < NSEG * TH;
        ok = mbar_wait_bounded(nready, 0);
        const float2 s2 = f2(snorm);
        float2 gwr[RW + 1], gtr[RT + 1];
#pragma unroll
        for (int d = 0; d <= RW; ++d) gwr[d] = P.gw[d];
#pragma unroll
        for (int d = 0; d <= RT; ++d) gtr[d] = P.gt[d];
        auto off = [](int d, int r) { return d < r ? r - d : d - r; };
        // t-filter in transposed direct form: for each of the 3 signals and 4 column pairs the
        // 2rt running partial sums of the 2rt+1-tap filter; with x[n] the w-filtered frame n and
        // g_j = gt[2rt - j], the output y[n] = sum_j g_j x[n - j] is the t-filtered frame n - rt.
        float2 st[2 * RT > 0 ? 2 * RT : 1][3][4];
        // The norm (or dot product): kFold frames in float32, those sums in FP64 in shared memory.  One
        // float32 sum over a long run loses digits: 500 equal frames put the norm 1.2e-5 off, where 128
        // squares per sum are at most 3.8e-6 away.  Where the fold stands decides the compiler's schedule of
        // the passes: for rw >= 7 with the output frame's inputs, else around the frame loop.  480p, us per
        // step, inside / around: (1,3,3) 97.5 / 94.0, (2,3,3) 107.0 / 105.0, (1,7,7) 130.2 / 134.3, (2,8,8)
        // 150.3 / 156.2, (2,7,7) 138.1 / 138.7 (in bf16 147 / 151); at the frame's end or after its passes
        // it is never better than both.
        float2 part = make_float2(0.f, 0.f);
        red[i] = 0.0;
        auto fold = [&] {
            red[i] += (double)part.x + (double)part.y;
            part = make_float2(0.f, 0.f);
        };
        constexpr bool kFoldInside = RW >= 7;
        float tmax = 0.f;   // MODE 8: the largest output so far (outputs are >= 0)
        const int tile_off = row * TW + seg * 8;

        int q = 0, qp = 0, e = 0;           // Q ring slot and phase; output frames finished so far
        Run r;
        for (int s = 0; ok && run_of(P, s, r); ++s) {
#pragma unroll
            for (int a = 0; a < 2 * RT; ++a)
#pragma unroll
                for (int k = 0; k < 3; ++k)
#pragma unroll
                    for (int m = 0; m < 4; ++m) st[a][k][m] = make_float2(0.f, 0.f);
            int to = max(r.t0 - RT, 0) - RT;   // output frame of each step
            auto frames = [&](int end) {
#pragma unroll 1
                for (; to < end; ++to) {
                    // ---------------- the output frame's inputs, while the h-pass is still at work
                    const bool emit = to >= r.t0;
                    const int b = e & 1;
                    float2 fo[4], so[4], uo[4];
                    if (emit) {
                        if constexpr (kFoldInside)
                            if (e % kFold == 0) fold();
                        const uint32_t ph = (uint32_t)(e >> 1) & 1;
                        ok = mbar_wait_bounded(&ffull[b], ph) && (e < 2 || mbar_wait_bounded(&oempty[b], ph ^ 1));
                        ld_cols(reinterpret_cast<const TS*>(smem + C::O_F + b * C::FT) + tile_off, fo);
                        if constexpr (E::IN2)
                            ld_cols(reinterpret_cast<const float*>(smem + C::O_I2 + b * C::T32) + tile_off, so);
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            const float2 sv = SEP ? so[m] : fo[m];
                            uo[m] = make_float2(unary_pow_fast<true>(sv.x, P.p), unary_pow_fast<true>(sv.y, P.p));
                        }
                        // again for the rest, in a branch never taken for the usual p: the longer form
                        // throughout costs 1.4 % (solve 480p 7391 -> 7495 us)
                        if (P.p > kUnaryFtzP) {
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                const float2 sv = SEP ? so[m] : fo[m];
                                uo[m] = make_float2(unary_pow_fast(sv.x, P.p), unary_pow_fast(sv.y, P.p));
                            }
                        }
                    }
                    ok = ok && mbar_wait_bounded(&qfull[q], qp);
                    if (!__all_sync(0xffffffffu, ok)) {
                        ok = false;
                        break;
                    }
                    // ---------------- w-pass: Q -> x[n], then the t-filter update
                    float2 y[3][4];
                    if (item) {
                        const float* Q = reinterpret_cast<const float*>(smem + C::O_Q + q * C::Q) + row * QP + PADW +
                                         seg * 8 - C::OFF;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            float2 acc[4];   // four independent chains (one per column pair)
#pragma unroll
                            for (int m = 0; m < 4; ++m) acc[m] = make_float2(0.f, 0.f);
                            float2 pa[C::NPAIR];
#pragma unroll
                            for (int j = 0; j < C::NPAIR / 2; ++j) {
                                const float4 a = reinterpret_cast<const float4*>(Q + k * TH * QP)[j];
                                pa[2 * j] = make_float2(a.x, a.y);
                                pa[2 * j + 1] = make_float2(a.z, a.w);
                            }
#pragma unroll
                            for (int d = 0; d <= 2 * RW; ++d) {
                                const float2 gd = gwr[off(d, RW)];
#pragma unroll
                                for (int m = 0; m < 4; ++m) {
                                    const int c = 2 * m + d + C::OFF - RW;
                                    if (c & 1) {   // odd-aligned pair: two scalar FMAs
                                        acc[m].x = fmaf(pa[c >> 1].y, gd.x, acc[m].x);
                                        acc[m].y = fmaf(pa[(c >> 1) + 1].x, gd.x, acc[m].y);
                                    } else {
                                        acc[m] = fma2(pa[c >> 1], gd, acc[m]);
                                    }
                                }
                            }
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                const float2 x = acc[m];
                                if constexpr (RT == 0) {
                                    y[k][m] = mul2(x, gtr[0]);
                                } else {
                                    y[k][m] = fma2(x, gtr[RT], st[0][k][m]);
#pragma unroll
                                    for (int j = 0; j < 2 * RT - 1; ++j)
                                        st[j][k][m] = fma2(x, gtr[off(2 * RT - 1 - j, RT)], st[j + 1][k][m]);
                                    st[2 * RT - 1][k][m] = mul2(x, gtr[RT]);
                                }
                            }
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&qempty[q]);
                    if (++q == NQ) q = 0, qp ^= 1;
                    if (!emit) continue;
                    // ---------------- Eq. 7 combination for frame to
                    if (item) {
                        float2 outv[4], outq[4];
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            const float2 fv = fo[m];
                            const float2 u = uo[m];
                            const float2 ee = fma2(make_float2(-fv.x, -fv.y), fv, f2(P.inv_alpha));   // 1/alpha - f^2
                            if constexpr (MODE == 7) {
                                float2 F = make_float2(1.f, 1.f);
                                const float2 f3 = mul2(fv, mul2(fv, fv));
                                for (int i3 = 0; i3 < P.exj; ++i3) F = mul2(F, f3);
                                const float2 inner = fma2(mul2(fv, f2(P.exc[2])), y[1][m], mul2(f2(P.exc[1]), y[2][m]));
                                outv[m] = mul2(mul2(s2, F), fma2(fv, inner, mul2(f2(P.exc[0]), y[0][m])));
                                if (P.exj > 0) outv[m] = __fadd2_rn(outv[m], so[m]);   // the terms so far
                            } else if constexpr (MODE == 0 || MODE == 4 || MODE == 6 || MODE == 8) {
                                float2 B = fma2(ee, y[0][m], make_float2(-y[1][m].x, -y[1][m].y));
                                B = fma2(mul2(f2(2.f), fv), y[2][m], B);
                                const float2 xt = mul2(mul2(s2, u), B);
                                part = fma2(xt, xt, part);
                                if constexpr (MODE == 8) tmax = fmaxf(tmax, fmaxf(xt.x, xt.y));
                                outv[m] = (OUT_X || MODE == 8) ? xt : mul2(u, xt);
                                if constexpr (MODE == 4) outq[m] = xt;
                                if constexpr (MODE == 6) {
                                    const float2 a1 = fma2(f2(P.p), ee, mul2(f2(-2.f), mul2(fv, fv)));
                                    const float2 a3 = mul2(f2(2.f * (P.p + 1.f)), fv);
                                    const float2 Qd = fma2(a1, y[0][m], mul2(f2(-P.p), y[1][m]));
                                    outq[m] = mul2(s2, fma2(a3, y[2][m], Qd));
                                }
                            } else {
                                const float2 a1 = fma2(f2(P.p), ee, mul2(f2(-2.f), mul2(fv, fv)));
                                const float2 a3 = mul2(f2(2.f * (P.p + 1.f)), fv);
                                float2 Qd = fma2(a1, y[0][m], mul2(f2(-P.p), y[1][m]));
                                Qd = mul2(s2, fma2(a3, y[2][m], Qd));
                                if constexpr (MODE == 1) {
                                    outv[m] = Qd;
                                } else {
                                    float2 B = fma2(ee, y[0][m], make_float2(-y[1][m].x, -y[1][m].y));
                                    B = fma2(mul2(f2(2.f), fv), y[2][m], B);
                                    outv[m] = mul2(mul2(u, u), B);
                                    part = fma2(so[m], B, part);
                                    outq[m] = Qd;
                                }
                            }
                        }
                        if constexpr (OUT_X) {
                            // caller layout: rows of W values, 8-byte aligned when W is even (and the
                            // caller's base is), then one 8-byte store per pair
                            const Geom& g = P.g;
                            const int h = r.h0 + row, wb = r.w0 + seg * 8;
                            float* o = reinterpret_cast<float*>(P.out) + ((int64_t)to * g.H + h) * g.W + wb;
                            if (h < g.H) {
                                if (wb + 8 <= g.W && (reinterpret_cast<uintptr_t>(o) & 7) == 0) {
#pragma unroll
                                    for (int m = 0; m < 4; ++m) reinterpret_cast<float2*>(o)[m] = outv[m];
                                } else {
#pragma unroll
                                    for (int m = 0; m < 4; ++m) {
                                        if (wb + 2 * m < g.W) o[2 * m] = outv[m].x;
                                        if (wb + 2 * m + 1 < g.W) o[2 * m + 1] = outv[m].y;
                                    }
                                }
                            }
                        } else {
                            st_cols(reinterpret_cast<TVO*>(smem + C::O_O + b * C::OT) + tile_off, outv);
                        }
                        if constexpr (E::OUT2) st_cols(reinterpret_cast<float*>(smem + C::O_O2 + b * C::T32) + tile_off, outq);
                    }
                    fence_async();       // the tiles written here are read by TMA stores
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&done[b]);
                    ++e;
                }
            };
            if constexpr (kFoldInside) {
                frames(r.t1);
            } else {
#pragma unroll 1
                while (ok && to < r.t1) {
                    fold();
                    frames(min(r.t1, to + kFold));
                }
            }
        }
        red[i] += (double)part.x + (double)part.y;
        if constexpr (MODE == 8) {
            const unsigned key = P.nan_key && isnan(red[i]) ? kNanKey : order_key(tmax);
            const unsigned kmax = __reduce_max_sync(0xffffffffu, key);
            if (lane == 0 && P.maxkey) atomicMax(P.maxkey, kmax);
        }
    }
    if (!ok) atomicOr(P.flags, kFlagTimeout);
    if (__syncthreads_or(!ok)) return;
    if (tid < 32 && P.acc_out) {
        double r = red[tid];
        for (int k = tid + 32; k < NW; k += 32) r += red[k];
        r = warp_sum(r);
        if (tid == 0) atomicAdd(P.acc_out, r);
    }
}

template <int RT, int RH, int RW, typename TS, typename TVO, bool OUT_X, bool SEP, int MODE>
static bool launch_t(const StepArgs& a) {
    using C = Cfg<RT, RH, RW, TS, TVO, OUT_X, SEP, MODE>;
    using E = Extra<SEP, MODE>;
    constexpr bool bf = sizeof(TS) == 2;
    const Geom& g = a.g;
    Maps M = {};
    if (!make_step_map(&M.v, a.vin, bf, g, BW, C::BH) || !make_step_map(&M.f, a.f, bf, g, BW, C::BH) ||
        !make_step_map(&M.fc, a.f, bf, g, TW, TH))
        return false;
    if (E::IN2 && !make_step_map(&M.in2, MODE == 7 ? a.out : (const void*)a.s32, false, g, TW, TH)) return false;
    if (!OUT_X && !make_step_map(&M.out, a.out, sizeof(TVO) == 2, g, TW, TH)) return false;
    if (E::OUT2 && !make_step_map(&M.out2, a.out2, false, g, TW, TH)) return false;
    auto kern = iter_stream<RT, RH, RW, TS, TVO, OUT_X, SEP, MODE>;
    static std::atomic<unsigned long long> attr_set{0};   // devices on which the attribute is set
    if (!(attr_set & device_bit())) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) != cudaSuccess) return false;
        attr_set |= device_bit();
    }
    Params P;
    P.g = g;
    P.inv_alpha = a.inv_alpha;
    P.p = a.p;
    // the Gaussian is even: the taps of offsets 0..r, and zeros up to the kernel's radius
    auto fill = [](float2* d, int R, const float* g1, int r) {
        for (int i = 0; i <= R; ++i) {
            const float t = i <= r ? g1[r + i] : 0.f;
            d[i] = make_float2(t, t);
        }
    };
    fill(P.gt, RT, a.tp.gt, a.tp.rt);
    fill(P.gh, RH, a.tp.gh, a.tp.rh);
    fill(P.gw, RW, a.tp.gw, a.tp.rw);
    P.exj = a.ex ? a.ex->j : 0;
    for (int i = 0; i < 3; ++i) P.exc[i] = a.ex ? a.ex->c[i] : 0.f;
    P.maxkey = a.maxkey;
    P.nan_key = a.tp.rt != RT || a.tp.rh != RH || a.tp.rw != RW;
    P.tx = (g.W + TW - 1) / TW;
    P.tiles = P.tx * ((g.H + TH - 1) / TH);
    const int64_t frames = (int64_t)P.tiles * g.T;   // output frames of all tiles
    const int grid = (int)(frames < num_sms() ? frames : num_sms());
    P.whole = P.tiles / grid;
    P.acc_in = a.acc_in;
    P.acc_out = a.acc_out;
    P.flags = a.flags;
    P.out = a.out;
    launch_after_previous(kern, dim3(grid), NTHR, C::SMEM, a.s, M, P);
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

}  // namespace stream
}  // namespace sfseg
