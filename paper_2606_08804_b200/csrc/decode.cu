// Recurrent step (Section 3.3.1, final update rule and read-out) of one or several tokens, in place:
//   x = k + lambda q ;  p = alpha h^T x ;  delta = beta (v - p) ;  h <- alpha h + k delta^T ;
//   o = h_new^T q = alpha h^T q + (k.q) delta .
// A CTA owns DVS columns of one state (columns evolve independently); every thread keeps its part of the slice in
// registers between the only read and the only write of the state, all loads are issued before the first use.
// One token is bound by HBM traffic: 80.4 us for 4096 states of 128 x 128 in fp32, 1.02 of the measured copy bandwidth (48
// of 41 us at that bandwidth with a bf16 state, whose rows are read 16 bytes per thread like those of an fp32 one).
#include "internal.h"
#include "sm100.cuh"

namespace qd {
namespace {

// Several tokens per call (multi-token / speculative decoding): S consecutive tokens of every sequence go through the
// same recurrence, one after the other, while the state slice stays in registers -- one read and one write of the state
// for S tokens instead of S of each.  Token tensors are token-major [B, S, H, d] like those of the chunkwise calls.  A
// token's arithmetic does not depend on S, so with an fp32 state S tokens give the bits of S single-token calls.
// Past two tokens the step is bound by the fp32 arithmetic and by what delays it, not by HBM.  So q, k and x of up to
// kBlock tokens are staged (and normalised, and k.q summed) before the first one is applied, by one warp per token and
// under the loads of the state; a token then costs its two row products, one reduction over row groups and the update,
// with two barriers.  Fetching each token when its turn came, with four barriers (seven with QD_NORM_QK), took 20 us per
// token of 256 x 16 states, 35 with normalisation; this takes 12 and 14 (of 5 at the rate of the FMA pipe).
// Four CTAs per SM are asked for: left to itself the compiler schedules the row products for fewer registers in flight
// (190 instead of 166 us for eight tokens).  At d_k = 128 that is 128 registers, of which an fp32 state leaves 8 - 16 bytes to
// spill; five CTAs would spill 64 - 204.
// SB16 (QD_STATE_BF16): the state is STORED in bf16 (half the bytes of the step); it is widened to fp32 when read, all S
// tokens of the call are applied in fp32, and it is rounded to bf16 once, when written back.
constexpr int kBlock = 8;
template <typename IO, int DK, int DVS, int NT, bool LOGITS, bool NORM, bool SB16>      // flags, compile-time
__global__ void __launch_bounds__(NT, 4) k_decode(int S, int H, int dv, const IO* __restrict__ q, const IO* __restrict__ k,
                                                     const IO* __restrict__ v, const IO* __restrict__ beta,
                                                     const IO* __restrict__ alpha, const IO* __restrict__ lam,
                                                     void* __restrict__ state_, IO* __restrict__ o) {
    constexpr int NC = SB16 ? 8 : 4;                             // columns per thread: 16 bytes of a state row
    constexpr int CT = DVS / NC, RP = NT / CT, NP = DK / RP;
    static_assert(NT % CT == 0 && DK % RP == 0, "bad decode tiling");
    constexpr int TOKEN = 3 * DK + DVS;
    extern __shared__ __align__(16) float stok[];                // per token: x [DK], q [DK], k [DK], v [DVS]
    __shared__ __align__(16) float redx[2][RP][DVS], redq[2][RP][DVS];
    __shared__ __align__(16) float sdelta[2][DVS];
    __shared__ float scoef[kBlock][4];                           // beta, alpha, k.q
    const int nsl = dv / DVS, bh = blockIdx.x / nsl, j0 = (blockIdx.x % nsl) * DVS, tid = threadIdx.x;
    const int b = bh / H, hh = bh % H;
    const int ct = tid % CT, rg = tid / CT, lane = tid & 31;

    uint4* base = reinterpret_cast<uint4*>(static_cast<unsigned char*>(state_) + (((size_t)bh * DK + rg) * dv + j0) * (SB16 ? 2 : 4)) + ct;
    const size_t rstride = (size_t)RP * dv / NC;
    // launched while the kernel before it drains (2 us less per step): nothing is read before that kernel has completed
    sm100::grid_dep_wait();
    sm100::grid_dep_launch();
    float h[NP][NC];
    uint4 raw[NP];
#pragma unroll
    for (int pz = 0; pz < NP; ++pz) raw[pz] = __ldcs(base + pz * rstride);
    auto stage = [&](int s0) {
        const int nb = min(kBlock, S - s0);
        for (int s = tid >> 5; s < nb; s += NT / 32) {
            const size_t row = ((size_t)b * S + s0 + s) * H + hh;        // token row of this head in the [B, S, H] view
            float *tx = stok + s * TOKEN, *tq = tx + DK, *tk = tq + DK, *tv = tk + DK;
            float qv[DK / 32], kv[DK / 32], kq = 0.f;
#pragma unroll
            for (int i = 0; i < DK / 32; ++i) { qv[i] = ld(q, row * DK + i * 32 + lane); kv[i] = ld(k, row * DK + i * 32 + lane); }
            float vv[DVS / 32];
#pragma unroll
            for (int i = 0; i < DVS / 32; ++i) vv[i] = ld(v, row * dv + j0 + i * 32 + lane);
            const float zb = ld(beta, row), za = alpha ? ld(alpha, row) : 0.f, zl = lam ? ld(lam, row) : 0.f;
            const float la = lam ? gate(zl, LOGITS) : 0.f;
            float part[DK / 32];
#pragma unroll
            for (int i = 0; i < DK / 32; ++i) part[i] = fmaf(kv[i], qv[i], 0.f);
            if (NORM) {
                // q^ = q / sqrt(|q|^2 + eps), k^ likewise
                float ssq = 0.f, ssk = 0.f, kq1 = 0.f;
#pragma unroll
                for (int i = 0; i < DK / 32; ++i) { ssq = fmaf(qv[i], qv[i], ssq); ssk = fmaf(kv[i], kv[i], ssk); kq1 += part[i]; }
#pragma unroll
                for (int w = 16; w > 0; w >>= 1) {
                    ssq += __shfl_xor_sync(0xffffffffu, ssq, w);
                    ssk += __shfl_xor_sync(0xffffffffu, ssk, w);
                    kq1 += __shfl_xor_sync(0xffffffffu, kq1, w);
                }
                const float rq = 1.f / sqrtf(ssq + kNormEps), rk = 1.f / sqrtf(ssk + kNormEps);
#pragma unroll
                for (int i = 0; i < DK / 32; ++i) { qv[i] *= rq; kv[i] *= rk; }
                kq = kq1 * rq * rk;
            } else {
                // 32 elements by butterfly, then the groups of 32 in order
#pragma unroll
                for (int w = 16; w > 0; w >>= 1)
#pragma unroll
                    for (int i = 0; i < DK / 32; ++i) part[i] += __shfl_xor_sync(0xffffffffu, part[i], w);
#pragma unroll
                for (int i = 0; i < DK / 32; ++i) kq += part[i];
            }
#pragma unroll
            for (int i = 0; i < DK / 32; ++i) {
                tx[i * 32 + lane] = fmaf(la, qv[i], kv[i]);
                tq[i * 32 + lane] = qv[i];
                tk[i * 32 + lane] = kv[i];
            }
#pragma unroll
            for (int i = 0; i < DVS / 32; ++i) tv[i * 32 + lane] = vv[i];
            if (lane == 0) {
                scoef[s][0] = gate(zb, LOGITS);
                scoef[s][1] = alpha ? gate(za, LOGITS) : 1.f;
                scoef[s][2] = kq;
            }
        }
        __syncthreads();
    };
    stage(0);
#pragma unroll
    for (int pz = 0; pz < NP; ++pz) {
        const uint32_t w[4] = {raw[pz].x, raw[pz].y, raw[pz].z, raw[pz].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (SB16) {
                h[pz][(2 * e) % NC] = __uint_as_float(w[e] << 16);
                h[pz][(2 * e + 1) % NC] = __uint_as_float(w[e] & 0xffff0000u);
            } else {
                h[pz][e] = __uint_as_float(w[e]);
            }
        }
    }
    for (int s0 = 0;;) {
        const int nb = min(kBlock, S - s0);
#pragma unroll 1
        for (int s = 0; s < nb; ++s) {
            const float *tx = stok + s * TOKEN, *tq = tx + DK, *tk = tq + DK;
            const int bf = s & 1;
            const size_t row = ((size_t)b * S + s0 + s) * H + hh;
            float ax[NC], aq[NC];
#pragma unroll
            for (int e = 0; e < NC; ++e) { ax[e] = 0.f; aq[e] = 0.f; }
#pragma unroll
            for (int pz = 0; pz < NP; ++pz) {
                const float xi = tx[pz * RP + rg], qi = tq[pz * RP + rg];
#pragma unroll
                for (int e = 0; e < NC; ++e) { ax[e] = fmaf(h[pz][e], xi, ax[e]); aq[e] = fmaf(h[pz][e], qi, aq[e]); }
            }
#pragma unroll
            for (int e = 0; e < NC; e += 4) {
                *reinterpret_cast<float4*>(&redx[bf][rg][ct * NC + e]) = make_float4(ax[e], ax[e + 1], ax[e + 2], ax[e + 3]);
                *reinterpret_cast<float4*>(&redq[bf][rg][ct * NC + e]) = make_float4(aq[e], aq[e + 1], aq[e + 2], aq[e + 3]);
            }
            __syncthreads();
            const float al = scoef[s][1];
            if (tid < DVS) {
                float rx = 0.f, rq = 0.f;
#pragma unroll
                for (int r = 0; r < RP; ++r) { rx += redx[bf][r][tid]; rq += redq[bf][r][tid]; }
                const float dl = scoef[s][0] * (tk[DK + tid] - al * rx);
                sdelta[bf][tid] = dl;
                st(o, row * dv + j0 + tid, fmaf(al, rq, scoef[s][2] * dl));
            }
            __syncthreads();
            float dl[NC];
#pragma unroll
            for (int e = 0; e < NC; e += 4) {
                const float4 t = *reinterpret_cast<const float4*>(&sdelta[bf][ct * NC + e]);
                dl[e] = t.x; dl[e + 1] = t.y; dl[e + 2] = t.z; dl[e + 3] = t.w;
            }
#pragma unroll
            for (int pz = 0; pz < NP; ++pz) {
                const float ki = tk[pz * RP + rg];
#pragma unroll
                for (int e = 0; e < NC; ++e) h[pz][e] = fmaf(al, h[pz][e], ki * dl[e]);
            }
        }
        s0 += kBlock;
        if (s0 >= S) break;
        __syncthreads();                                                 // the staged tokens are rewritten
        stage(s0);
    }
#pragma unroll
    for (int pz = 0; pz < NP; ++pz) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (SB16) {
                const __nv_bfloat162 t = __floats2bfloat162_rn(h[pz][(2 * e) % NC], h[pz][(2 * e + 1) % NC]);
                w[e] = *reinterpret_cast<const uint32_t*>(&t);
            } else {
                w[e] = __float_as_uint(h[pz][e]);
            }
        }
        __stcs(base + pz * rstride, make_uint4(w[0], w[1], w[2], w[3]));
    }
}

template <typename IO, int DK>
cudaError_t launch(int B, int S, int H, int dv, const void* q, const void* k, const void* v, const void* beta,
                         const void* alpha, const void* lam, void* state, void* o, bool logits, bool norm, bool sb16,
                         cudaStream_t stream) {
    constexpr int DVS = 64, NT = 128;
    dim3 grid((unsigned)(dv / DVS) * (unsigned)(B * H));
    auto kern = logits ? (norm ? k_decode<IO, DK, DVS, NT, true, true, false> : k_decode<IO, DK, DVS, NT, true, false, false>)
                       : (norm ? k_decode<IO, DK, DVS, NT, false, true, false> : k_decode<IO, DK, DVS, NT, false, false, false>);
    if (sb16)
        kern = logits ? (norm ? k_decode<IO, DK, DVS, NT, true, true, true> : k_decode<IO, DK, DVS, NT, true, false, true>)
                      : (norm ? k_decode<IO, DK, DVS, NT, false, true, true> : k_decode<IO, DK, DVS, NT, false, false, true>);
    return launch_overlapped(kern, grid, dim3(NT), (S < kBlock ? S : kBlock) * (3 * DK + DVS) * sizeof(float), stream, S, H, dv,
                             (const IO*)q, (const IO*)k, (const IO*)v, (const IO*)beta, (const IO*)alpha, (const IO*)lam, state, (IO*)o);
}

}  // namespace

cudaError_t decode_steps(int B, int S, int H, int dk, int dv, int dtype, const void* q, const void* k, const void* v,
                         const void* beta, const void* alpha, const void* lam, void* state, void* o,
                         bool logits, bool norm, bool sb16, cudaStream_t stream) {
    if (dtype == QD_BF16) {
        if (dk == 128) return launch<__nv_bfloat16, 128>(B, S, H, dv, q, k, v, beta, alpha, lam, state, o, logits, norm, sb16, stream);
        return launch<__nv_bfloat16, 64>(B, S, H, dv, q, k, v, beta, alpha, lam, state, o, logits, norm, sb16, stream);
    }
    if (dk == 128) return launch<float, 128>(B, S, H, dv, q, k, v, beta, alpha, lam, state, o, logits, norm, sb16, stream);
    return launch<float, 64>(B, S, H, dv, q, k, v, beta, alpha, lam, state, o, logits, norm, sb16, stream);
}

}  // namespace qd
