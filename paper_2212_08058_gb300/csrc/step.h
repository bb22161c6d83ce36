// step.h -- the Eq. 7 step's arguments, shared by the two kernels that run it (iter_stream.cuh,
// iter_tile.cuh) and by the dispatch over radii (kernels_fast.cu).
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "launch.h"

namespace sfseg {

// What a step does besides v_{k+1} = u x~_{k+1} from v_k (kernel template parameter MODE; the
// derivation of each is at iter_stream): the plain step; the adjoint's Q-pass; the recording step;
// the adjoint's g-pass; the recomputing step with its Q-pass; a term of the exact kernel's series;
// the step that also takes its largest output.
enum StepMode { kStep = 0, kQPass = 1, kRecord = 4, kGPass = 5, kStepQ = 6, kExactTerm = 7, kStepMax = 8 };

struct StepArgs {
    int mode = kStep;
    const void* vin = nullptr;      // v (internal layout)
    int vin_type = kF32;
    void* out = nullptr;            // the next state (internal layout), or x~ (caller layout) when out_x
    int out_type = kF32;
    bool out_x = false;
    const void* f = nullptr;        // f in vin's type (internal layout)
    Geom g{};
    Taps tp{};
    float inv_alpha = 1.f, p = 1.f;
    const double* acc_in = nullptr;
    double* acc_out = nullptr;
    int* flags = nullptr;
    const float* s32 = nullptr;     // separate unary map (kStep), V_k (kGPass)
    void* out2 = nullptr;           // the record (kRecord), Q (kGPass, kStepQ)
    const ExactTerm* ex = nullptr;  // kExactTerm
    unsigned* maxkey = nullptr;     // kStepMax
    cudaStream_t s = nullptr;
};

// A map over an internal volume with boxes of box_w x box_h x 1 (kernels_fast.cu).
bool make_step_map(CUtensorMap* map, const void* base, bool bf16, const Geom& g, int box_w, int box_h);

// Frame-chunk length of the small-volume kernel minimising (waves x frames per chunk) for `slots`
// resident CTAs.
inline int tile_chunk(int T, int tiles, int slots, int rt) {
    long best_cost = -1;
    int best = T;
    for (int nt = 1;;) {   // the distinct chunk lengths
        const int chunk = (T + nt - 1) / nt;
        const int nct = (T + chunk - 1) / chunk;
        const long waves = ((long)tiles * nct + slots - 1) / slots;
        const long cost = waves * (chunk + 2 * rt);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = chunk;
        }
        if (chunk == 1) break;
        nt = (T + chunk - 2) / (chunk - 1);
    }
    return best;
}

// Calls K::launch<TS, TVO, OUT_X, SEP, MODE>(a) for the step that `a` describes; false where no such
// kernel is compiled.
template <class K>
bool step_dispatch(const StepArgs& a) {
    using bf = __nv_bfloat16;
    switch (a.mode) {
        case kStep:
            if (a.s32) {   // separate unary map: float32 storage only (the generic stencil serves bf16)
                if (a.vin_type != kF32) return false;
                return a.out_x ? K::template launch<float, float, true, true, kStep>(a)
                               : K::template launch<float, float, false, true, kStep>(a);
            }
            if (a.vin_type == kF32)
                return a.out_x ? K::template launch<float, float, true, false, kStep>(a)
                               : K::template launch<float, float, false, false, kStep>(a);
            if (a.out_x) return K::template launch<bf, float, true, false, kStep>(a);
            return a.out_type == kBF16 ? K::template launch<bf, bf, false, false, kStep>(a)
                                       : K::template launch<bf, float, false, false, kStep>(a);
        case kRecord: return K::template launch<float, float, false, false, kRecord>(a);
        case kQPass: return K::template launch<float, float, false, false, kQPass>(a);
        case kGPass: return K::template launch<float, float, false, false, kGPass>(a);
        case kStepQ: return K::template launch<float, float, false, false, kStepQ>(a);
        case kExactTerm: return K::template launch<float, float, false, false, kExactTerm>(a);
        case kStepMax: return K::template launch<float, float, false, false, kStepMax>(a);
    }
    return false;
}

}  // namespace sfseg
