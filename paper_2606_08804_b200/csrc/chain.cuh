// What the state chains of the tcgen05 path share: the per-token scales of a chunk.
#pragma once
#include "internal.h"

namespace qd {

// Log-decays (and, with QD_NORM_QK, 1/|k|) of a chunk, fetched by a load warp a chunk ahead of the loads that they go with.
struct TokenScales {
    const float *g, *rk;                 // of the call's first chunk of the sequence; rk: null if keys come normalised
    int lane;
    float g0, g1, gc, r0, r1;
    __device__ __forceinline__ TokenScales(const float* g_, const float* rk_, size_t row, int lane_)
        : g(g_ + row), rk(rk_ ? rk_ + row : nullptr), lane(lane_), r0(1.f), r1(1.f) {}
    __device__ __forceinline__ void fetch(int n) {
        const float* gn = g + (size_t)n * kChunk;
        g0 = gn[lane]; g1 = gn[32 + lane]; gc = gn[kChunk - 1];
        if (rk) { r0 = rk[(size_t)n * kChunk + lane]; r1 = rk[(size_t)n * kChunk + 32 + lane]; }
    }
    // gamma_C / gamma_t for the 64 tokens, then gamma_C
    __device__ __forceinline__ void put(float* s) const {
        s[lane] = __expf(gc - g0) * r0;
        s[32 + lane] = __expf(gc - g1) * r1;
        if (lane == 0) s[64] = __expf(gc);
    }
};

}  // namespace qd
