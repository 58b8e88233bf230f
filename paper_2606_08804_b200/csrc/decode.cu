// Recurrent step (Section 3.3.1, final update rule and read-out) of one or several tokens, in place:
//   x = k + lambda q ;  p = alpha h^T x ;  delta = beta (v - p) ;  h <- alpha h + k delta^T ;
//   o = h_new^T q = alpha h^T q + (k.q) delta .
// A CTA owns DVS columns of one state (columns evolve independently); every thread keeps its part of the slice in
// registers between the only read and the only write of the state, all loads are issued before the first use.
// One token is bound by HBM traffic: 80.5 us for 4096 states of 128 x 128 in fp32, 1.04 of the measured copy bandwidth (44 on the same
// tokens again and again, 46.7 on new ones, of 42 us at that bandwidth with a bf16 state, whose rows are read 16 bytes per thread
// like those of an fp32 one).
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
// ONE (bf16 state, a single token), KEEP false: the state is needed once more only to be updated, so it stays as it was read, is
// widened each time and written back as it is updated: 32 registers instead of 64, and five CTAs to an SM instead of four, which with
// 16 KB each are too little on its way to keep HBM busy (256 x 16 states 47.7 -> 44.0 us, 100 x 8 12.2 -> 11.1; six CTAs, which spill
// 70 bytes, 49.5).  With an fp32 state it would gain nothing (30 x 16 states 11.8 -> 12.4).  It is one_token_kept's choice at d_k = 128:
// for one CTA it takes longer.  At d_k = 64 it gains at any number of CTAs (4 of them 1.72 -> 1.60 us).
// VEC: a thread has groups of four rows that are neighbours, so that its parts of x, q and k are read four at a time while what a CTA
// loads at a time stays close together.  One token of 149 x 8 states 18.45 us with rows a whole group apart, 18.9 with all rows
// of a thread next to each other, 18.3 so; 8 tokens of 256 x 16 153 / 148 / 146.5, of a bf16 state 155 / 152 / 150.6.  Rows a
// whole group apart where the tokens of an fp32 state are normalised, which leaves fewer registers, and for several fp32 tokens on
// a bf16 state with d_k = 128 (3 tokens of 256 x 16 states 80.5 in groups of four, 75.7 so; 4 tokens 100.2 and 92.4).  The order of the
// sums follows the rows, so the rule looks neither at the number of states nor, with an fp32 state, at S.
constexpr int kBlock = 8;
template <typename IO, int DK, int DVS, int NT, bool LOGITS, bool NORM, bool SB16, bool ONE, bool KEEP>      // flags, compile-time
__global__ void __launch_bounds__(NT, KEEP ? 4 : 5) k_decode(int S, int H, int dv, const IO* __restrict__ q, const IO* __restrict__ k,
                                                     const IO* __restrict__ v, const IO* __restrict__ beta,
                                                     const IO* __restrict__ alpha, const IO* __restrict__ lam,
                                                     void* __restrict__ state_, IO* __restrict__ o) {
    constexpr int NC = SB16 ? 8 : 4;                             // columns per thread: 16 bytes of a state row
    constexpr int CT = DVS / NC, RP = NT / CT, NP = DK / RP;
    static_assert(NT % CT == 0 && DK % RP == 0 && NP % 4 == 0, "bad decode tiling");
    static_assert(KEEP || ONE, "several tokens need the state in fp32 from token to token");
    constexpr int TOKEN = 3 * DK + DVS;
    constexpr bool VEC = SB16 ? ONE || NORM || DK == 64 || sizeof(IO) == 2 : !NORM;
    extern __shared__ __align__(16) float stok[];                // per token: x [DK], q [DK], k [DK], v [DVS]
    __shared__ __align__(16) float redx[2][RP][DVS], redq[2][RP][DVS];
    __shared__ __align__(16) float sdelta[2][DVS];
    __shared__ float scoef[kBlock][4];                           // beta, alpha, k.q
    const int nsl = dv / DVS, bh = blockIdx.x / nsl, j0 = (blockIdx.x % nsl) * DVS, tid = threadIdx.x;
    const int b = bh / H, hh = bh % H;
    const int ct = tid % CT, rg = tid / CT, lane = tid & 31;

    uint4* base = reinterpret_cast<uint4*>(static_cast<unsigned char*>(state_) + (((size_t)bh * DK + (VEC ? rg * 4 : rg)) * dv + j0) * (SB16 ? 2 : 4)) + ct;
    const size_t rowq = (size_t)dv / NC;
    const size_t rstride = (size_t)RP * dv / NC;
    auto at = [&](int pz) { return VEC ? base + ((pz >> 2) * 4 * RP + (pz & 3)) * rowq : base + pz * rstride; };
    // launched while the kernel before it drains (2 us less per step): nothing is read before that kernel has completed
    sm100::grid_dep_wait();
    sm100::grid_dep_launch();
    float h[KEEP ? NP : 1][NC];                                  // the state in fp32
    uint4 raw[NP];
#pragma unroll
    for (int pz = 0; pz < NP; ++pz) raw[pz] = __ldcs(at(pz));
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
    // What a staged vector has for G rows of this thread, from the p-th on.  Rows a whole group apart are read one at a time, where
    // d_k = 128 leaves an fp32 state registers four (8 normalised tokens of 256 x 16 states 170.9 -> 169.2 us; at d_k = 64 57.6 -> 58.2).
    constexpr int G = VEC || (DK == 128 && !SB16) ? 4 : 1;
    auto rows = [&](const float* t, int p, float (&r)[G]) {
        if constexpr (VEC) {
            const float4 f = *reinterpret_cast<const float4*>(t + rg * 4 + p * RP);
            r[0] = f.x; r[1] = f.y; r[2] = f.z; r[3] = f.w;
        } else {
#pragma unroll
            for (int z = 0; z < G; ++z) r[z] = t[(p + z) * RP + rg];
        }
    };
    auto widen = [&](const uint4& r, float (&d)[NC]) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (SB16) {
                d[(2 * e) % NC] = __uint_as_float(w[e] << 16);
                d[(2 * e + 1) % NC] = __uint_as_float(w[e] & 0xffff0000u);
            } else {
                d[e] = __uint_as_float(w[e]);
            }
        }
    };
    auto write = [&](int pz, const float (&d)[NC]) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (SB16) {
                const __nv_bfloat162 t = __floats2bfloat162_rn(d[(2 * e) % NC], d[(2 * e + 1) % NC]);
                w[e] = *reinterpret_cast<const uint32_t*>(&t);
            } else {
                w[e] = __float_as_uint(d[e]);
            }
        }
        __stcs(at(pz), make_uint4(w[0], w[1], w[2], w[3]));
    };
    if (KEEP)
#pragma unroll
        for (int pz = 0; pz < NP; ++pz) widen(raw[pz], h[pz % (KEEP ? NP : 1)]);
    for (int s0 = 0;;) {
        const int nb = ONE ? 1 : min(kBlock, S - s0);
#pragma unroll 1
        for (int s = 0; s < nb; ++s) {
            const float *tx = stok + s * TOKEN, *tq = tx + DK, *tk = tq + DK;
            const int bf = s & 1;
            const size_t row = ((size_t)b * S + s0 + s) * H + hh;
            float ax[NC], aq[NC];
#pragma unroll
            for (int e = 0; e < NC; ++e) { ax[e] = 0.f; aq[e] = 0.f; }
#pragma unroll
            for (int p = 0; p < NP; p += G) {
                if (!KEEP) asm volatile("" ::: "memory");                // G rows at a time
                float xi[G], qi[G];
                rows(tx, p, xi);
                rows(tq, p, qi);
#pragma unroll
                for (int z = 0; z < G; ++z) {
                    float one[NC];
                    if (!KEEP) widen(raw[p + z], one);
                    const float (&hr)[NC] = KEEP ? h[(p + z) % (KEEP ? NP : 1)] : one;
#pragma unroll
                    for (int e = 0; e < NC; ++e) { ax[e] = fmaf(hr[e], xi[z], ax[e]); aq[e] = fmaf(hr[e], qi[z], aq[e]); }
                }
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
            if (!KEEP)                                                   // widened anew, instead of being kept widened
#pragma unroll
                for (int pz = 0; pz < NP; ++pz) asm volatile("" : "+r"(raw[pz].x), "+r"(raw[pz].y), "+r"(raw[pz].z), "+r"(raw[pz].w));
            float dl[NC];
#pragma unroll
            for (int e = 0; e < NC; e += 4) {
                const float4 t = *reinterpret_cast<const float4*>(&sdelta[bf][ct * NC + e]);
                dl[e] = t.x; dl[e + 1] = t.y; dl[e + 2] = t.z; dl[e + 3] = t.w;
            }
#pragma unroll
            for (int p = 0; p < NP; p += G) {
                if (!KEEP) asm volatile("" ::: "memory");                // G rows at a time
                float ki[G];
                rows(tk, p, ki);
#pragma unroll
                for (int z = 0; z < G; ++z) {
                    float one[NC];
                    if (!KEEP) widen(raw[p + z], one);
                    float (&hr)[NC] = KEEP ? h[(p + z) % (KEEP ? NP : 1)] : one;
#pragma unroll
                    for (int e = 0; e < NC; ++e) hr[e] = fmaf(al, hr[e], ki[z] * dl[e]);
                    if (!KEEP) write(p + z, hr);
                }
            }
        }
        s0 += kBlock;
        if (ONE || s0 >= S) break;
        __syncthreads();                                                 // the staged tokens are rewritten
        stage(s0);
    }
    if (KEEP)
#pragma unroll
        for (int pz = 0; pz < NP; ++pz) write(pz, h[pz % (KEEP ? NP : 1)]);
}

// One token on a bf16 state with d_k = 128: whether the widened state is kept, which lets four CTAs share an SM, or widened twice,
// which lets five.  Kept where five would bring nothing: they do when more than four to an SM are wanted, and when two launches,
// the second of which begins while the first drains, fit on the GPU five to an SM but not four.  Widened twice / kept, us per call
// of many: 8 CTAs 2.23 / 1.95, 290 2.86 / 2.59, but 300 3.22 / 3.45, 350 3.32 / 3.51; then 400 4.20 / 3.59, 592 4.41 / 3.69, but 608 4.33 /
// 5.00.  Normalised tokens 290 3.20 / 3.10, 350 3.67 / 4.12, 592 4.85 / 4.20; fp32 tokens 592 4.70 / 3.69.
bool one_token_kept(unsigned ctas) {
    const bool two_want_five = 2 * ctas > 4 * kSMs && 2 * ctas <= 5 * kSMs;
    return ctas <= 4 * kSMs && !two_want_five;
}

template <typename IO, int DK>
cudaError_t launch(int B, int S, int H, int dv, const void* q, const void* k, const void* v, const void* beta,
                         const void* alpha, const void* lam, void* state, void* o, bool logits, bool norm, bool sb16,
                         cudaStream_t stream) {
    constexpr int DVS = 64, NT = 128;
    dim3 grid((unsigned)(dv / DVS) * (unsigned)(B * H));
    using Kern = decltype(&k_decode<IO, DK, DVS, NT, false, false, false, false, true>);
#define QD_GATES(...)                                                                                                        \
    {k_decode<IO, DK, DVS, NT, false, false, __VA_ARGS__>, k_decode<IO, DK, DVS, NT, false, true, __VA_ARGS__>,              \
     k_decode<IO, DK, DVS, NT, true, false, __VA_ARGS__>, k_decode<IO, DK, DVS, NT, true, true, __VA_ARGS__>}
    static const Kern table[4][4] = {QD_GATES(false, false, true), QD_GATES(true, false, true), QD_GATES(true, true, false),
                                     QD_GATES(true, true, DK == 128)};
#undef QD_GATES
    const int form = !sb16 ? 0 : S > 1 ? 1 : DK == 128 && one_token_kept(grid.x) ? 3 : 2;
    const Kern kern = table[form][(logits ? 2 : 0) + (norm ? 1 : 0)];
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
