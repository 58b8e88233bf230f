// Tensor-core (tcgen05 / TMEM / TMA) chunkwise forward for bf16, d_k = d_v = 128, chunk 64.
//
// Two kernels, following Section 3.3.2:
//   k_tc_prep       one CTA per chunk, four to an SM: g, X = K + diag(lambda) Q, the Gram
//                   blocks X K^T and Q K^T, the UT-transform inverse, and the WY factors.  It leaves,
//                   per chunk, in bf16:  Qg = diag(gamma) Q  [token][dk],
//                   P = Gamma o (Q K^T) causal incl. diagonal [token][64],
//                   Wt = (T diag(gamma) X)^T  [dk][64 tokens],   Ut = (T V)^T  [dv][64 tokens].
//   k_tc_chain_fwd  one CTA per (batch, head), or two that share its d_v rows (chain_rows; k_tc_chain_fwd_half): walks the
//                   chunks in order with the fp32 state in registers, everything transposed so that d_v is the MMA M dimension:
//                     Delta^T = Ut - h^T Wt            O^T = h^T Qg^T + Delta^T P^T
//                     h^T <- gamma_C h^T + (Delta diag(gamma_C/gamma))^T K
// With few long sequences the two run beside each other, part by part (tc_fwd_parts).
// All waits are bounded; on expiry the CTA records QD_ERR_TIMEOUT in the workspace status word, lets what it has in flight
// come to an end (mbar_drain), releases its tensor memory and returns.
#include "chain.cuh"
#include "internal.h"
#include "sm100.cuh"
#include "tf32.cuh"

namespace qd {
namespace {
using namespace sm100;
typedef __nv_bfloat16 bf16;

constexpr int C = kChunk;      // 64
constexpr int D = 128;         // d_k = d_v

// =================================================================================================
struct PrepParams {
    float* rqk;                // non-null: L2-normalise q and k here; [0, BH*Tp) <- 1/|q_t|, [BH*Tp, 2 BH*Tp) <- 1/|k_t|
    int T, Tp, H, N, Ns, BH;   // T tokens per sequence, of which the N chunks from n0 on; the workspace holds Tp = 64 Ns rows per sequence
    int n0;
    int beside;                // 1: runs beside the forward chain launched before it (see tc_fwd_parts), so it waits for that at its end
    const bf16 *beta, *alpha, *lam;
    float* g;
    bf16* Qg;
    bf16* Mt;                  // optional: ((I+A)^-1)^T per chunk, [column i][row r]; kept for the backward
    unsigned* status;
};

// 48 KB: K (then A in fp32, then the T tiles, then P) | Q (then V, then W~^T) | X (then U~^T).  Four CTAs fit on one SM.
constexpr int kPrepSmem = 3 * 16384 + 1024;
constexpr int kPrepCompute = 128, kPrepThreads = kPrepCompute + 32;       // + a warp that issues every copy and every product

// The 64 x 64 matrices of the inverse are kept transposed, [column i][row r], so that a column is contiguous; groups of
// four rows are permuted by column so that the fragment loads of a 16 x 8 or 8 x 8 piece, the epilogue's stores (fragments: eight
// rows, every second column) and 16-byte accesses along a column all spread over the banks.
__device__ __forceinline__ int at_swizzle(int i) { return (((i ^ (i >> 2)) & 1) << 3) | ((i & 2) << 3) | (i & 4); }
__device__ __forceinline__ int at_off(int i, int r) { return i * C + (r ^ at_swizzle(i)); }

// acc (16 x 16) += X Y over k = 0..15: X(m, k) = a[at_off(am + m, ak + k)], Y(k, n) = b[at_off(bk + k, bn + n)] with am, ak, bk
// multiples of 8, bn of 16, fp32-accurate (three tf32 products).
__device__ __forceinline__ void mm16(float (&acc)[2][4], const float* a, int am, int ak, const float* b, int bk, int bn) {
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
    const float *a0 = a + (am + g) * C + t + (g & 4), *a1 = a + (am + g) * C + t + (4 - (g & 4));    // columns t, t + 4 of a step
    const int am8 = at_swizzle(g) & 24;
    const float *b0 = b + (bk + t) * C + (bn ^ (t << 3)) + g, *b1 = b + (bk + t + 4) * C + (bn ^ (t << 3) ^ 8) + (g ^ 4);
    const int b8 = (t & 1) ? -8 : 8;                                                                   // column + 8 of Y
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int ac = (ak + 8 * s) ^ am8;
        uint32_t ah[4], al[4], bh[2][2], bl[2][2];
        tf32_split(a0[ac], ah[0], al[0]); tf32_split(a0[ac + 8 * C], ah[1], al[1]);
        tf32_split(a1[ac], ah[2], al[2]); tf32_split(a1[ac + 8 * C], ah[3], al[3]);
        tf32_split(b0[8 * s * C], bh[0][0], bl[0][0]); tf32_split(b1[8 * s * C], bh[0][1], bl[0][1]);
        tf32_split(b0[8 * s * C + b8], bh[1][0], bl[1][0]); tf32_split(b1[8 * s * C - b8], bh[1][1], bl[1][1]);
#pragma unroll
        for (int j = 0; j < 2; ++j) mma_tf32(acc[j], al, bh[j]);
#pragma unroll
        for (int j = 0; j < 2; ++j) mma_tf32(acc[j], ah, bl[j]);
#pragma unroll
        for (int j = 0; j < 2; ++j) mma_tf32(acc[j], ah, bh[j]);
    }
}
__device__ __forceinline__ void put16(const float (&acc)[2][4], float sign, float* d, int dm, int dn) {
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            *reinterpret_cast<float2*>(d + at_off(dm + g + 8 * h, dn + 8 * j + 2 * t)) = make_float2(sign * acc[j][2 * h], sign * acc[j][2 * h + 1]);
}
// the four warps that do the arithmetic of a chunk among themselves
__device__ __forceinline__ void psync() { asm volatile("bar.sync 1, %0;" ::"n"(kPrepCompute) : "memory"); }
// M = (I + A)^-1, in place, both transposed (at_off): A^T comes strictly upper triangular in this view, M^T leaves with its zeros
// and ones.  Block-wise: the 16 x 16 diagonal blocks by right-looking substitution, a column in the registers of a lane, a block
// to a warp; then blocks joined twice, M21^T = -M11^T (A21^T M22^T), on the warp-level tensor instruction, zero blocks left out.
// A column walked over all 64 rows in registers takes 63 dependent steps whose broadcast loads of A are bound by
// shared-memory wavefronts: 7300 cycles against 3100 for this (5300 with the SM's other CTAs at work).
__device__ __forceinline__ void invert(float* Ac) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < 16) {
        const int j = lane, o = warp * 16;
        float m[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) m[r] = r == j ? 1.f : 0.f;
#pragma unroll
        for (int i = 0; i < 15; ++i) {
#pragma unroll
            for (int r4 = (i + 1) / 4; r4 < 4; ++r4) {
                const float4 a = *reinterpret_cast<const float4*>(Ac + at_off(o + i, o + 4 * r4));     // zero at and above row i
                m[4 * r4] = fmaf(-a.x, m[i], m[4 * r4]); m[4 * r4 + 1] = fmaf(-a.y, m[i], m[4 * r4 + 1]);
                m[4 * r4 + 2] = fmaf(-a.z, m[i], m[4 * r4 + 2]); m[4 * r4 + 3] = fmaf(-a.w, m[i], m[4 * r4 + 3]);
            }
        }
        __syncwarp(0xffffu);
#pragma unroll
        for (int r4 = 0; r4 < 4; ++r4)
            *reinterpret_cast<float4*>(Ac + at_off(o + j, o + 4 * r4)) = make_float4(m[4 * r4], m[4 * r4 + 1], m[4 * r4 + 2], m[4 * r4 + 3]);
    }
    psync();
    if (!(warp & 1)) {                                           // 16 -> 32: one warp per pair of blocks
        const int o = warp * 16;
        float s[2][4] = {}, m[2][4] = {};
        mm16(s, Ac, o, o + 16, Ac, o + 16, o + 16);
        __syncwarp();
        put16(s, 1.f, Ac, o, o + 16);
        __syncwarp();
        mm16(m, Ac, o, o, Ac, o, o + 16);
        __syncwarp();
        put16(m, -1.f, Ac, o, o + 16);
    }
    psync();
    {   // 32 -> 64: 16 x 16 to a warp
        const int tm = (warp & 2) * 8, tn = (warp & 1) * 16;
        float s[2][4] = {}, m[2][4] = {};
        mm16(s, Ac, tm, 32, Ac, 32, 32 + tn);
        if (tn) mm16(s, Ac, tm, 48, Ac, 48, 48);                 // M22^T is upper triangular: k <= n
        psync();
        put16(s, 1.f, Ac, tm, 32 + tn);
        psync();
        mm16(m, Ac, tm, 16, Ac, 16, 32 + tn);
        if (!tm) mm16(m, Ac, 0, 0, Ac, 0, 32 + tn);              // M11^T likewise: k >= m
        psync();
        put16(m, -1.f, Ac, tm, 32 + tn);
    }
    psync();
}

// One CTA prepares a chunk of one head.  What bounds it is the chain of short phases -- copy, Gram products, A, inverse, T, WY
// products, copies out -- of 7 us at least; so a CTA is as small as it can be, 4 warps that do the arithmetic and one that issues
// every copy and every product, 48 KB, 128 columns of tensor memory, and four of them share an SM.  (Pairs of chunks,
// two CTAs of twice the size to an SM: 113 against 108 us on 128 sequences of 32 chunks, 406 against 384 on 32 of 512, 18.7 against
// 17 on 16 of 14.  592 persistent CTAs: 121 and 447 -- four of them on an SM then go through their phases in step.)
//   scan / coefficients   thread t < 64 owns token t
//   row-wise elementwise  16 threads per 256-byte row (coalesced), 8 rows per pass
//   Gram epilogue         64-row products, 16 rows to a warp, in fragment layout (tmem_ld_frag)
//   triangular inverse    by warps, see invert
//   final epilogue        thread d owns row d of U~^T and of W~^T
// Both Gram products start as soon as Q and K are there: X K^T = K K^T + diag(lambda) Q K^T is combined in the epilogue, so
// nothing waits for X, which is formed under the products.  V takes Q's place when they have read it.
// NORM (QD_NORM_QK): q and k come un-normalised; 1/|q_t|, 1/|k_t| are factors wherever a row is used.  LOGITS
// (QD_COEF_LOGITS): the coefficients are logits of sigmoid gates.  Compile-time, because even the untaken sigmoid /
// log-sigmoid code on the path of the scan, which every later phase of the CTA waits for, cost the kernel 8 %.
template <bool NORM, bool LOGITS>
__global__ void __launch_bounds__(kPrepThreads, 4) k_tc_prep(const __grid_constant__ CUtensorMap mapQ,
                                                             const __grid_constant__ CUtensorMap mapK,
                                                             const __grid_constant__ CUtensorMap mapV,
                                                             const __grid_constant__ CUtensorMap mapUt,
                                                             const __grid_constant__ CUtensorMap mapWt,
                                                             const __grid_constant__ CUtensorMap mapP, PrepParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *sK = smem, *sQ = smem + 16384, *sX = smem + 32768;
    float* sA = reinterpret_cast<float*>(sK);                   // A^T, then M^T: [column][row], at_off
    // bar_x, bar_t, bar_o: one arrival per compute warp -- Q read and X written; T tiles written; results staged
    __shared__ uint64_t bar_qk, bar_v, bar_g, bar_w, bar_x, bar_t, bar_o;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    __shared__ __align__(16) float sg[C], srk[C];
    __shared__ float sbeta[C], slam[C], srq[C], swsum;

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    // CTAs are numbered chunk-major, last chunk first: the forward chain, which starts with chunk 0 of every sequence,
    // then finds the tiles written last (and K, read last) still in L2
    const int n = p.n0 + p.N - 1 - (int)blockIdx.x / p.BH, bh = (int)blockIdx.x % p.BH;
    const int b = bh / p.H, hh = bh % p.H;
    const int t0 = n * C;                                            // first token of the chunk
    const size_t wtok0 = (size_t)bh * p.Tp + (size_t)t0;             // first row in the workspace's [BH*Tp] view

    // What a CTA reads is on its way before anything else is set up: with the SM's other CTAs at work a third of its time went by until
    // Q and K had come.  Prompts of 128 sequences of 32 chunks 164.0 -> 161.4 us, of 4 of 16 24.5 -> 23.8.  Nothing is read or written
    // before the kernel before this one has completed, unless this one runs beside it: then it reads inputs, which are older than
    // that chain, and writes rows that the chain does not touch.
    // A token past the end of the sequence is an exact no-op of the recurrence: beta = 0, alpha = 1 (and q = k = v = 0).
    const bf16 zero = __ushort_as_bfloat16(0);
    const bool live = tid < C && t0 + tid < p.T, has_a = live && p.alpha, has_l = live && p.lam;
    bf16 za = zero, zb = zero, zl = zero;
    if (warp == 4) {
        if (lane == 0) {
            mbar_init(&bar_qk, 1); mbar_init(&bar_v, 1); mbar_init(&bar_g, 1); mbar_init(&bar_w, 1);
            mbar_init(&bar_x, 4); mbar_init(&bar_t, 4); mbar_init(&bar_o, 4);
            mbar_init_fence();
            s_abort = 0;
            if (!p.beside) grid_dep_wait();
            // the call's status word starts at zero: the first CTA to start clears it, a second before any wait can expire
            if (blockIdx.x == 0 && !p.beside) *p.status = 0;
            mbar_expect_tx(&bar_qk, 32768);
            for (int blk = 0; blk < 2; ++blk) {          // rows at t >= T arrive as zeros
                tma_load_3d(sQ + blk * 8192, &mapQ, hh * D + blk * 64, t0, b, &bar_qk);
                tma_load_3d(sK + blk * 8192, &mapK, hh * D + blk * 64, t0, b, &bar_qk);
            }
            for (int blk = 0; blk < 2; ++blk) tma_prefetch_3d(&mapV, hh * D + blk * 64, t0, b);       // loaded when Q has been used
        }
        __syncwarp();
        tmem_alloc(&tmem_slot, 128);
        tmem_relinquish();
    } else if (tid < C) {
        if (!p.beside) grid_dep_wait();
        const size_t crow = ((size_t)b * p.T + t0 + tid) * p.H + hh;
        if (live) zb = p.beta[crow];
        if (has_a) za = p.alpha[crow];
        if (has_l) zl = p.lam[crow];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = uniform(tmem_slot), T0 = tb, T1 = tb + 64;
    auto wait = [&](uint64_t* bar) { return mbar_try_wait(bar, 0) || wait_on(bar, 0, s_abort, p.status); };

    if (!p.beside) grid_dep_wait();
    grid_dep_launch();                // the kernel after this one may set itself up while the last CTAs of this one run
    if (warp == 4) {
        // ---------------------------------- copies and products ----------------------------------
        const uint32_t issue = elect_lane();
        const uint32_t aK = smem_u32(sK), aQ = smem_u32(sQ), aX = smem_u32(sX);
        const bool lead = lane == 0;
        wait(&bar_qk);
        __syncwarp();
        umma_product_w<false, false, 64>(T1, aQ, 8192, aK, 8192, C, D, false, issue);                // Q K^T
        umma_product_w<false, false, 64>(T0, aK, 8192, aK, 8192, C, D, false, issue);                // K K^T
        umma_commit_w(&bar_g, issue);
        wait(&bar_x);
        wait(&bar_g);
        const bool has_v = lead && !s_abort;
        if (has_v) {
            mbar_expect_tx(&bar_v, 16384);
            for (int blk = 0; blk < 2; ++blk) tma_load_3d(sQ + blk * 8192, &mapV, hh * D + blk * 64, t0, b, &bar_v);
        }
        __syncwarp();
        wait(&bar_t);
        wait(&bar_v);
        __syncwarp();
        tc_fence_after();
        umma_product_w<true, true>(T0, aQ, 8192, aK, 8192, C, C, false, issue);                      // Ut = V^T T^T
        umma_product_w<true, true>(T1, aX, 8192, aK + 8192, 8192, C, C, false, issue);               // Wt = X^T (T diag(gamma))^T
        umma_commit_w(&bar_w, issue);
        wait(&bar_o);
        tc_fence_after();
        if (lead) {
            const int y = (int)(((size_t)bh * p.Ns + n) * D);
            tma_store_2d(&mapUt, sX, 0, y);
            tma_store_2d(&mapWt, sQ, 0, y);
            tma_store_2d(&mapP, sK, 0, (int)wtok0);
            tma_store_commit();
            tma_store_wait_read();             // the staging tiles must outlive the reads; the writes complete with the grid
        }
        __syncwarp();
        // A wait has expired: the other warps may still be at their work, which they come to the end of by now without waiting, and what is
        // in flight has not been waited for
        if (s_abort) { mbar_drain(&bar_o, 0); mbar_drain(&bar_w, 0); mbar_drain(&bar_qk, 0); if (has_v) mbar_drain(&bar_v, 0); }
        __syncwarp();
        tmem_dealloc(tb, 128);
        if (blockIdx.x == 0) grid_dep_wait();            // when this kernel has completed, so has the one before it
        return;
    }
    // ---------------------------------- arithmetic ----------------------------------
    auto arrive = [&](uint64_t* bar) { __syncwarp(); if (lane == 0) mbar_arrive(bar); };
    // coefficients of token tid; in-chunk cumulative log-decay by a two-warp scan
    if (tid < C) {
        float g = has_a ? log_gate(__bfloat162float(za), LOGITS) : 0.f;
        sbeta[tid] = live ? gate(__bfloat162float(zb), LOGITS) : 0.f;
        slam[tid] = has_l ? gate(__bfloat162float(zl), LOGITS) : 0.f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float t = __shfl_up_sync(0xffffffffu, g, o);
            if (lane >= o) g += t;
        }
        if (tid == 31) swsum = g;
        asm volatile("bar.sync 2, 64;" ::: "memory");
        if (warp == 1) g += swsum;
        sg[tid] = g;
        p.g[wtok0 + tid] = g;
    }
    psync();
    wait(&bar_qk);
    // row-wise, 16 lanes to a 256-byte row (chunk `ch` of 16 bytes each): Qg = gamma Q to the workspace, and X
    {
        const int ch = tid & 15, rsub = tid >> 4;
        const uint32_t coff = (ch >> 3) * 8192;
        bf16* qg = p.Qg + wtok0 * D + ch * 8;
        const size_t nrows = (size_t)p.BH * p.Tp;
        const bool has_lam = p.lam != nullptr;
#pragma unroll
        for (int it = 0; it < 8; ++it) {
            const int row = it * 8 + rsub;
            const uint32_t off = coff + sw128_chunk(row, ch & 7);
            float qv[8], kv[8], rq = 1.f, rk = 1.f;
            load8(sQ + off, qv);
            load8(sK + off, kv);
            if (NORM) {
                // 1 / sqrt(|q|^2 + eps), 1 / sqrt(|k|^2 + eps)
                float sq = 0.f, sk = 0.f;
#pragma unroll
                for (int e = 0; e < 8; ++e) { sq = fmaf(qv[e], qv[e], sq); sk = fmaf(kv[e], kv[e], sk); }
#pragma unroll
                for (int o = 1; o < 16; o <<= 1) {
                    sq += __shfl_xor_sync(0xffffffffu, sq, o);
                    sk += __shfl_xor_sync(0xffffffffu, sk, o);
                }
                rq = rsqrtf(sq + kNormEps);
                rk = rsqrtf(sk + kNormEps);
                if (ch == 0) {
                    srq[row] = rq; srk[row] = rk;
                    p.rqk[wtok0 + row] = rq; p.rqk[nrows + wtok0 + row] = rk;
                }
            }
            const float gr = __expf(sg[row]) * rq, lm = slam[row] * rq;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if (NORM) kv[e] *= rk;
                if (NORM || has_lam) kv[e] = fmaf(lm, qv[e], kv[e]);      // lambda absent (the gated delta rule, Eq. 3): X = K
            }
            sts128(sX + off, pack8(kv));
#pragma unroll
            for (int e = 0; e < 8; ++e) qv[e] *= gr;
            *reinterpret_cast<uint4*>(qg + (size_t)row * D) = pack8(qv);
        }
    }
    fence_proxy_async();
    arrive(&bar_x);
    psync();                                             // K has been read, the factors of the normalisation are there
    wait(&bar_g);
    tc_fence_after();
    // A = strictLower(beta_r Gamma_ri (x_r . k_i)) -> shared fp32, transposed;  P = Gamma_ri (q_r . k_i), i <= r, kept in
    // registers until its staging tile is free.  My rows: r0, r0 + 8; of every 8 columns: ft, ft + 1.
    uint32_t pk[4][4];
    const int rw = 16 * warp, r0 = rw + (lane >> 2), ft = 2 * (lane & 3);
    {
        const uint32_t lane_base = (uint32_t)warp * 32;
        float gr[2], be[2], rq[2], rk[2], lm[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = r0 + 8 * j;
            gr[j] = sg[r]; be[j] = sbeta[r]; rq[j] = NORM ? srq[r] : 1.f; rk[j] = NORM ? srk[r] : 1.f; lm[j] = slam[r] * rq[j];
        }
#pragma unroll
        for (int cg = 0; cg < 4; ++cg) {
            float kk[8], qk[8];
            tmem_ld_frag2(tmem_addr(T0, lane_base, cg * 16), kk);
            tmem_ld_frag2(tmem_addr(T1, lane_base, cg * 16), qk);
            tmem_ld_wait();
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int j = m & 1, r = r0 + 8 * j, c = cg * 16 + 8 * (m >> 1) + ft;
                const float2 g2 = *reinterpret_cast<const float2*>(sg + c);
                const float2 k2 = NORM ? *reinterpret_cast<const float2*>(srk + c) : make_float2(1.f, 1.f);
                float pv[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int x = 4 * (m >> 1) + 2 * j + e;
                    float dec = c + e <= r ? __expf(gr[j] - (e ? g2.y : g2.x)) : 0.f;
                    if (NORM) dec *= e ? k2.y : k2.x;
                    sts32(sA + at_off(c + e, r), c + e < r ? be[j] * dec * fmaf(lm[j], qk[x], rk[j] * kk[x]) : 0.f);
                    pv[e] = dec * (rq[j] * qk[x]);
                }
                pk[cg][m] = pack_bf16(pv[0], pv[1]);
            }
        }
    }
    tc_fence_before();
    psync();
    invert(sA);
    // T = M diag(beta), T diag(gamma): line j of the MN-major tiles holds column j over the rows; thread = (column
    // j, block of eight rows), eight threads to a column.  The tiles take A's place: everything is read first.
    {
        float m[4][8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int id = k * kPrepCompute + tid, j = id >> 3, kb = id & 7;
#pragma unroll
            for (int e = 0; e < 8; e += 4)
                *reinterpret_cast<float4*>(m[k] + e) = *reinterpret_cast<const float4*>(sA + at_off(j, kb * 8 + e));
        }
        psync();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int id = k * kPrepCompute + tid, j = id >> 3, kb = id & 7;
            const float beta = sbeta[j], bg = beta * __expf(sg[j]);
            float a[8], bq[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) { a[e] = m[k][e] * beta; bq[e] = m[k][e] * bg; }
            sts128(sK + sw128_chunk(j, kb), pack8(a));
            sts128(sK + 8192 + sw128_chunk(j, kb), pack8(bq));
            if (p.Mt) *reinterpret_cast<uint4*>(p.Mt + (((size_t)bh * p.Ns + n) * C + j) * C + kb * 8) = pack8(m[k]);
        }
    }
    fence_proxy_async();
    arrive(&bar_t);
    wait(&bar_w);
    tc_fence_after();
    // P, [64 tokens][64], over the T tiles; row d = tid of U~^T over X and of W~^T over V; all written by TMA
#pragma unroll
    for (int cg = 0; cg < 4; ++cg) stsm4<false>(sK + sw128_chunk(rw + (lane & 15), cg * 2 + (lane >> 4)), pk[cg]);
#pragma unroll
    for (int q4 = 0; q4 < 4; ++q4) {
        float v[32];
        tmem_ld32(tmem_addr(tb, (uint32_t)warp * 32, q4 * 32), v);
        tmem_ld_wait();
        unsigned char* stage = q4 < 2 ? sX : sQ;
#pragma unroll
        for (int i = 0; i < 4; ++i) sts128(stage + sw128_chunk(tid, (q4 & 1) * 4 + i), pack8(v + i * 8));
    }
    fence_proxy_async();
    tc_fence_before();
    arrive(&bar_o);
}

// =================================================================================================
struct ChainParams {
    int Tp, H, N, Ns;          // N chunks of a sequence, from n0 on; Tp = 64 Ns rows per sequence in the workspace
    int n0;
    int h0_late;               // 1: h0 is what the chain of the chunks before has left
    const float* g;
    const float* h0;
    float* hT;
    int T;                     // tokens per sequence
    bf16* o;                   // [B][T][H][D], as mapO
    int scaled;                // 0: no forget gate and no key normalisation: every per-token factor on Delta is 1
    const float* rk;           // non-null (QD_NORM_QK): 1/|k_t| per workspace row; the keys are read un-normalised and
                               // the factor is folded into the per-token scale of Delta
    unsigned* status;
};

// Tiles of a chunk in shared memory.  Wt 16K | Ut 16K, three deep (Delta^T is staged over Ut and held until it has been
// read); Qg 16K | K 16K | P 8K, two deep; the exit state 32K; half an output tile 8K.
constexpr int kDeepA = 3, kStageA = 32768, kStageB = 40960;
constexpr int kOffB = kDeepA * kStageA, kOffH = kOffB + 2 * kStageB, kOffO = kOffH + 32768;
constexpr int kChainSmem = kOffO + 8192 + 1024;
constexpr int kChainCompute = 512;                 // 16 epilogue warps: 4 warpgroups split the accumulator columns
constexpr int kChainThreads = kChainCompute + 128 + 96;   // + the output warpgroup, 1 MMA-issue warp, 1 warp each for TMA loads and saves
constexpr int kOutWarp = kChainCompute / 32, kMmaWarp = kOutWarp + 4;

// named barriers: compute threads arrive, the MMA warp waits (they run in lock-step); kBarOut: the output warpgroup among itself
constexpr int kBarH = 1, kBarD = 2, kBarOut = 3;

// What the saving warp of a forward chain does, one lane of it: entry state of every chunk (two 64-column blocks, `block` bytes apart) and
// Delta^T, in the order in which they are staged; the state's tile is one deep, Delta^T's DEEP, `stage` bytes apart.
template <int DEEP, class Wait>
__device__ __forceinline__ void save_chunks(const CUtensorMap* mapHs, const CUtensorMap* mapDt, size_t row, int N, const unsigned char* sHs, int block,
                                            const unsigned char* sDt, int stage, uint64_t* ht, uint64_t* hf, uint64_t* dt, uint64_t* df, Wait wait) {
    int s = 0;
    for (int n = 0; n < N; ++n) {
        const int y = (int)(row + (size_t)n * D);
        wait(ht, n & 1);                                  // entry state of chunk n (rows = d_v index, columns = d_k index) is staged
        tma_store_2d(mapHs, sHs, 0, y);
        tma_store_2d(mapHs, sHs + block, 64, y);
        tma_store_commit();
        if (n > 0) {                                      // Delta^T of chunk n - 1 has been read
            tma_store_wait_read_n<1>();
            mbar_arrive(df + (s == 0 ? DEEP - 1 : s - 1));
        }
        wait(dt + s, (n / DEEP) & 1);                     // Delta^T of chunk n is staged
        tma_store_2d(mapDt, sDt + s * stage, 0, y);
        tma_store_commit();
        tma_store_wait_read_n<1>();                       // the entry state has been read
        mbar_arrive(hf);
        if (++s == DEEP) s = 0;
    }
    tma_store_wait_all();
}

// Forward state chain.  The only true dependency per chunk is
//   h ready -> Delta-accumulator = h^T Wt -> Delta^T -> H-accumulator = (scaled Delta^T) K -> h update;
// the output products (h^T Qg^T + Delta^T P^T, double-buffered accumulator), the output epilogue and
// every TMA copy run in its shadow on their own warps.
// With many sequences HBM bounds it: 75 of 256 chunks move 6.2 TB/s with saves.  With few, a chunk takes 2210 cycles when nothing is
// saved and 3330 with saves.  Three things were in the way of that sequence:
//  - the shared-memory port: with h^T and Delta^T as shared-memory operands it carried 368 KB per chunk, 2900 cycles.  They
//    are A operands, so they live in tensor memory (bf16 pairs, written by the epilogues with tcgen05.st): no operand copies,
//    no re-reading of A by every product;
//  - the issue of 24 products from a branch taken by one lane, 80 - 130 cycles each: the MMA warp stays converged;
//  - the TMA unit: from L2 it brings 98 - 113 bytes per cycle and SM (boxes of 8 and 16 KB), but takes out 32, and the two add up
//    (64 KB in 580 - 670 cycles, 64 KB out 2050, both 2570).  The 72 KB that a chunk loads and the 16 KB of its output are about 1200
//    cycles; the 48 KB of Delta^T and entry state that a forward saves for the backward make it 2750.  (Ordinary stores, by one or two warps from
//    the tiles or by the epilogue from its registers, were slower: 4500 - 5000 cycles per chunk.)  So with few heads the d_v rows of a
//    head, which evolve independently, are shared by two CTAs (k_tc_chain_fwd_half): each loads what both need, but only its half of
//    Ut, and stores its half of everything.
// SAVE: also store, per chunk, the bf16 entry state (mapHs) and Delta^T (mapDt).  Compile-time for the half chain's sake (4 sequences of
// 64 chunks with saves 76.6 us, with a flag 80.3); this kernel is indifferent (128 of 32: 160.8 / 161.1, with saves 202.2 / 202.0).
// Compute warpgroup w owns tokens [16w, 16w+16) of the 64-column accumulators and d_k columns
// [32w, 32w+32) of the state; thread l of a warpgroup owns TMEM lane l = d_v index.
template <bool SAVE>
__global__ void __launch_bounds__(kChainThreads) k_tc_chain_fwd(const __grid_constant__ CUtensorMap mapWt,
                                                                const __grid_constant__ CUtensorMap mapUt,
                                                                const __grid_constant__ CUtensorMap mapQg,
                                                                const __grid_constant__ CUtensorMap mapK,
                                                                const __grid_constant__ CUtensorMap mapP,
                                                                const __grid_constant__ CUtensorMap mapHs,
                                                                const __grid_constant__ CUtensorMap mapDt,
                                                                const __grid_constant__ CUtensorMap mapO,
                                                                ChainParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sHs = smem + kOffH;              // h^T [128 dv][128 dk] for its store, 2 blocks of [128 lines][64]
    unsigned char* sO = smem + kOffO;               // half an output tile: [32 tokens][128 dv], 2 blocks of [32 lines][64]
    // Where one side may run ahead of the other there is a barrier per buffer; it comes round only after the other side has
    // waited for it.  bar_e: every product of a chunk has finished; bar_dt, bar_ht: Delta^T / exit state staged for their stores
    // (one arrival per compute warp); bar_df, bar_hf: they have been read; bar_o, bar_of: an output accumulator is complete /
    // has been read.
    __shared__ uint64_t bar_la[kDeepA], bar_lb[2], bar_e[2], bar_dt[kDeepA], bar_df[kDeepA], bar_ht, bar_hf, bar_a, bar_b, bar_o[2], bar_of[2], bar_end;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    // per stage: gamma_C / gamma_t for the 64 tokens, then gamma_C; written by the TMA warp before it arrives on the
    // stage's load barrier, so no epilogue thread waits for a global load
    __shared__ __align__(16) float sG[kDeepA][68];

    const int tid = threadIdx.x, warp = warp_index(), wg = warp >> 2, l = tid & 127, wq = warp & 3;
    constexpr int nb = kChainCompute + 32;                            // participants of a named barrier
    const int bh = blockIdx.x, b = bh / p.H, hh = bh % p.H;

    if (tid == 0) {
        for (int i = 0; i < kDeepA; ++i) { mbar_init(&bar_la[i], 1); mbar_init(&bar_dt[i], 16); mbar_init(&bar_df[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&bar_lb[i], 1); mbar_init(&bar_e[i], 1); mbar_init(&bar_o[i], 1); mbar_init(&bar_of[i], 4); }
        mbar_init(&bar_a, 1); mbar_init(&bar_b, 1); mbar_init(&bar_end, 1);
        mbar_init(&bar_ht, 16); mbar_init(&bar_hf, 1);
        mbar_init_fence();
        s_abort = 0;
    }
    if (tid < 32) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = uniform(tmem_slot);
    // accumulators: Delta 64 columns, H 128, O 2 x 64; operands, two bf16 per column: h^T 64, Delta^T 32, scaled Delta^T 32
    const uint32_t tD = tbase, tH = tbase + 64, tO0 = tbase + 192, aH = tbase + 320, aD = tbase + 384;
    const uint32_t aDs = p.scaled ? tbase + 416 : aD;               // all factors 1: the scaled copy is Delta itself
    const uint32_t lane_base = (uint32_t)wq * 32;

    // bounded wait; once any wait has expired every later wait returns at once (the kernel drains)
    auto wait = [&](uint64_t* bar, uint32_t parity) { return mbar_try_wait(bar, parity) || wait_on(bar, parity, s_abort, p.status); };
    const int tok0 = p.n0 * C;                                       // first token; rows and tiles of the workspace start at
    const size_t row0 = (size_t)bh * p.Tp + tok0, tile0 = (size_t)bh * p.Ns + p.n0;

    if (warp < kOutWarp) {
        // ---------------------------------- compute warps ----------------------------------
        float h[32];      // h^T[j = l][32 wg .. 32 wg + 31], fp32
        if (p.h0_late) grid_dep_wait();
        if (p.h0) {
            const float* src = p.h0 + (size_t)bh * D * D + (size_t)(32 * wg) * D + l;
#pragma unroll
            for (int i = 0; i < 32; ++i) h[i] = __ldcg(src + (size_t)i * D);      // not from L1: it may be new
        } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) h[i] = 0.f;
        }
        grid_dep_wait();                  // the loads of h0 (an input) are in flight; everything below depends on the prep kernel
        grid_dep_launch();
        auto arrive = [&](uint64_t* bar) { __syncwarp(); if ((tid & 31) == 0) mbar_arrive(bar); };
        auto staged = [&](uint64_t* bar) { fence_proxy_async(); arrive(bar); };      // my part of a tile is in shared memory, for its store
        // the state as operand: my 32 columns are 16 packed columns of tensor memory
        auto put_h = [&]() {
            uint32_t r[8];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
#pragma unroll
                for (int e = 0; e < 8; ++e) r[e] = pack_bf16(h[q * 16 + 2 * e], h[q * 16 + 2 * e + 1]);
                tmem_st8(tmem_addr(aH, lane_base, wg * 16 + q * 8), r);
            }
            tmem_st_wait();
            tc_fence_before();
            nb_arrive(kBarH, nb);
        };
        // the state that chunk n begins with as a tile: 64-column block wg >> 1, 16-byte chunks 4 (wg & 1) ..
        auto save_h = [&](int n) {
            if (n > 0) wait(&bar_hf, (n - 1) & 1);
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) sts128(sHs + (wg >> 1) * 16384 + sw128_chunk(l, (wg & 1) * 4 + ch), pack8(h + ch * 8));
            staged(&bar_ht);
        };
        put_h();
        if (SAVE) save_h(0);
        int pending = 0;                  // barriers of the MMA warp that a warp which gives up has not been to
        int s = 0;
        for (int n = 0; n < p.N; ++n) {
            unsigned char* ut = smem + s * kStageA + 16384;
            wait(&bar_la[s], (n / kDeepA) & 1);
            const uint4 u0 = *reinterpret_cast<const uint4*>(ut + sw128_chunk(l, wg * 2));           // before the product is waited for
            const uint4 u1 = *reinterpret_cast<const uint4*>(ut + sw128_chunk(l, wg * 2 + 1));
            const float gamC = sG[s][64];
            if (!__all_sync(0xffffffffu, wait(&bar_a, n & 1))) { pending = 2 * (p.N - n); break; }
            tc_fence_after();
            // Delta^T = Ut - acc, my 16 tokens, as operands: plain, and scaled by gamma_C/gamma_r
            {
                float v[16];
                tmem_ld16(tmem_addr(tD, lane_base, wg * 16), v);
                const float4* gp = reinterpret_cast<const float4*>(&sG[s][wg * 16]);
                const uint32_t uw[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
                tmem_ld_wait();
                uint32_t r[8], rs[8];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 t = gp[q];
                    const float x0 = __uint_as_float(uw[2 * q] << 16) - v[4 * q], x1 = __uint_as_float(uw[2 * q] & 0xffff0000u) - v[4 * q + 1];
                    const float x2 = __uint_as_float(uw[2 * q + 1] << 16) - v[4 * q + 2], x3 = __uint_as_float(uw[2 * q + 1] & 0xffff0000u) - v[4 * q + 3];
                    r[2 * q] = pack_bf16(x0, x1); r[2 * q + 1] = pack_bf16(x2, x3);
                    rs[2 * q] = pack_bf16(x0 * t.x, x1 * t.y); rs[2 * q + 1] = pack_bf16(x2 * t.z, x3 * t.w);
                }
                if (p.scaled) tmem_st8(tmem_addr(aDs, lane_base, wg * 8), rs);
                tmem_st8(tmem_addr(aD, lane_base, wg * 8), r);
                tmem_st_wait();
                tc_fence_before();
                nb_arrive(kBarD, nb);
                if (SAVE) {
                    sts128(ut + sw128_chunk(l, wg * 2), make_uint4(r[0], r[1], r[2], r[3]));
                    sts128(ut + sw128_chunk(l, wg * 2 + 1), make_uint4(r[4], r[5], r[6], r[7]));
                    staged(&bar_dt[s]);
                }
            }
            // h^T <- gamma_C h^T + acc (my 32 d_k columns), refresh the operand
            if (!__all_sync(0xffffffffu, wait(&bar_b, n & 1))) { pending = 2 * (p.N - n) - 1; break; }
            tc_fence_after();
            {
                float v[32];
                tmem_ld32(tmem_addr(tH, lane_base, wg * 32), v);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; ++i) h[i] = fmaf(gamC, h[i], v[i]);
            }
            put_h();
            if (SAVE && n + 1 < p.N) save_h(n + 1);
            if (++s == kDeepA) s = 0;
        }
        // a wait has expired: keep step with the MMA warp, which comes to every one of them (odd counts: H is next)
        for (; pending > 0; --pending) nb_sync(pending & 1 ? kBarH : kBarD, nb);
        if (p.hT && !s_abort) {
            float* dst = p.hT + (size_t)bh * D * D + (size_t)(32 * wg) * D + l;
#pragma unroll
            for (int i = 0; i < 32; ++i) dst[(size_t)i * D] = h[i];
        }
    } else if (warp < kMmaWarp) {
        // ---------------------------------- output warpgroup ----------------------------------
        // O^T row j = l of a chunk -> token-major half tiles -> TMA; its first thread issues the stores
        const bool first = tid == kChainCompute;
        uint32_t xoff[8];                 // byte offsets of my (fixed) column inside a staging line, for the 8 possible (token & 7)
#pragma unroll
        for (int e = 0; e < 8; ++e)
            xoff[e] = (uint32_t)e * 128u + (((((uint32_t)l & 63u) >> 3) ^ (uint32_t)e) << 4) + ((uint32_t)l & 7u) * 2u;
        unsigned char* stg = sO + (l >> 6) * 4096;
        grid_dep_wait();                  // the chain before may take longer than a wait has (tc_fwd_parts)
        for (int n = 0; n < p.N; ++n) {
            const int ob = n & 1;
            wait(&bar_o[ob], (n >> 1) & 1);
            tc_fence_after();
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                float v[32];
                tmem_ld32(tmem_addr(tO0 + 64 * ob, lane_base, half * 32), v);
                tmem_ld_wait();
                if (half == 1) {                          // the accumulator may be written again
                    tc_fence_before();
                    __syncwarp();
                    if ((tid & 31) == 0) mbar_arrive(&bar_of[ob]);
                }
                if (first) tma_store_wait_read_n<0>();    // the half tile before has been read
                nb_sync(kBarOut, 128);
#pragma unroll
                for (int i = 0; i < 32; ++i) sts16(stg + (i >> 3) * 1024 + xoff[i & 7], __float2bfloat16_rn(v[i]));
                fence_proxy_async();
                nb_sync(kBarOut, 128);
                if (first) {                              // rows past the end of the sequence are skipped
                    tma_store_3d(&mapO, sO, hh * D, tok0 + n * C + half * 32, b);
                    tma_store_3d(&mapO, sO + 4096, hh * D + 64, tok0 + n * C + half * 32, b);
                    tma_store_commit();
                }
            }
        }
        if (first) tma_store_wait_all();
    } else if (warp == kMmaWarp) {
        // ---------------------------------- MMA-issue warp, converged ----------------------------------
        const uint32_t issue = elect_lane();
        grid_dep_wait();
        grid_dep_launch();
        int s = 0;
        for (int n = 0; n < p.N; ++n) {
            const int ob = n & 1;
            const uint32_t stA = smem_u32(smem) + s * kStageA, stB = smem_u32(smem) + kOffB + ob * kStageB;
            const uint32_t tO = tO0 + 64 * ob;
            wait(&bar_la[s], (n / kDeepA) & 1);
            nb_sync(kBarH, nb);                         // h^T operand of chunk n is in place
            tc_fence_after();
            // Delta-accumulator = h^T Wt (B: MN-major, lines = d_k)
            umma_product_ts_w<true>(tD, aH, stA, 8192, C, D, false, issue);
            umma_commit_w(&bar_a, issue);
            // O-accumulator = h^T Qg^T (B: K-major); it reads the operand that the h update rewrites, so the commit
            // behind the H product below (which releases that update) must cover it
            if (n > 1) wait(&bar_of[ob], ((n >> 1) - 1) & 1);
            wait(&bar_lb[ob], (n >> 1) & 1);
            tc_fence_after();
            umma_product_ts_w<false>(tO, aH, stB, 8192, C, D, false, issue);
            nb_sync(kBarD, nb);                         // Delta^T operands of chunk n are in place
            tc_fence_after();
            // H-accumulator = scaled Delta^T K (B: MN-major, lines = tokens)
            umma_product_ts_w<true>(tH, aDs, stB + 16384, 8192, D, C, false, issue);
            umma_commit_w(&bar_b, issue);
            // O-accumulator += Delta^T P^T (B: K-major [r][s])
            umma_product_ts_w<false>(tO, aD, stB + 32768, 8192, C, C, true, issue);
            umma_commit_w(&bar_o[ob], issue);
            umma_commit_w(&bar_e[ob], issue);
            if (++s == kDeepA) s = 0;
        }
        nb_sync(kBarH, nb);                               // final arrival of the compute warps
        umma_commit_w(&bar_end, issue);                   // leaves when its products have come to their end, whatever has expired
        mbar_drain(&bar_end, 0);
    } else if (warp == kMmaWarp + 1) {
        // ---------------------------------- saving warp ----------------------------------
        // apart from the loads, which would otherwise wait for what these wait for
        if ((tid & 31) == 0 && SAVE) {
            grid_dep_wait();
            save_chunks<kDeepA>(&mapHs, &mapDt, tile0 * D, p.N, sHs, 16384, smem + 16384, kStageA, &bar_ht, &bar_hf, bar_dt, bar_df, wait);
        }
    } else {
        // ---------------------------------- TMA load warp ----------------------------------
        const bool lead = (tid & 31) == 0;
        grid_dep_wait();                  // the tiles and the log-decays read below are written by the prep kernel
        grid_dep_launch();
        TokenScales ts(p.g, p.rk, row0, tid & 31);
        auto load_a = [&](int n, int s) {                // by the whole warp
            ts.put(sG[s]);
            __syncwarp();
            if (lead) {
                const int yc = (int)((tile0 + n) * D);
                mbar_expect_tx(&bar_la[s], 32768);
                tma_load_2d(smem + s * kStageA, &mapWt, 0, yc, &bar_la[s]);
                tma_load_2d(smem + s * kStageA + 16384, &mapUt, 0, yc, &bar_la[s]);
            }
            if (n + 1 < p.N) ts.fetch(n + 1);
        };
        auto load_b = [&](int n) {                       // by the leading lane
            unsigned char* st = smem + kOffB + (n & 1) * kStageB;
            uint64_t* bar = &bar_lb[n & 1];
            const int yt = (int)(row0 + (size_t)n * C);
            mbar_expect_tx(bar, kStageB);
            tma_load_2d(st, &mapQg, 0, yt, bar);
            tma_load_2d(st + 8192, &mapQg, 64, yt, bar);
            tma_load_3d(st + 16384, &mapK, hh * D, tok0 + n * C, b, bar);
            tma_load_3d(st + 16384 + 8192, &mapK, hh * D + 64, tok0 + n * C, b, bar);
            tma_load_2d(st + 32768, &mapP, 0, yt, bar);
        };
        ts.fetch(0);
        for (int n = 0; n < kDeepA && n < p.N; ++n) {
            load_a(n, n);
            if (lead && n < 2) load_b(n);
        }
        int s = 0, na = min(kDeepA, p.N), nb = min(2, p.N);
        for (int n = 0; n < p.N; ++n) {
            bool more = n + kDeepA < p.N;
            if (lead) {
                wait(&bar_e[n & 1], (n >> 1) & 1);        // every product of chunk n has finished: refill its buffers
                if (n + 2 < p.N && !s_abort) { load_b(n + 2); nb = n + 3; }
                if (more && SAVE) wait(&bar_df[s], (n / kDeepA) & 1);
            }
            more = __shfl_sync(0xffffffffu, more && !s_abort, 0);     // one answer for the warp
            if (more) { load_a(n + kDeepA, s); na = n + kDeepA + 1; }
            if (++s == kDeepA) s = 0;
        }
        // unless a wait has expired the products have been waited for, and so have the loads
        if (lead && s_abort) { mbar_drain_ring(bar_la, kDeepA, na); mbar_drain_ring(bar_lb, 2, nb); }
    }
    tc_fence_before();
    __syncthreads();
    if (tid < 32) tmem_dealloc(tbase, 512);
}

// Tiles of a chunk for 64 of the 128 d_v rows, all three deep: Wt 16K | Ut 8K; Qg 16K | K 16K | P 8K.  Then what goes out, one deep: the
// entry state 16K (2 blocks of [64 dv][64]) | Delta^T 8K | the output 8K ([64 tokens][64 dv]).
constexpr int kHalfDeep = 3, kHalfStageA = 24576, kHalfStageB = 40960;
constexpr int kHalfOffB = kHalfDeep * kHalfStageA, kHalfOffS = kHalfOffB + kHalfDeep * kHalfStageB, kHalfOffO = kHalfOffS + 24576;
constexpr int kHalfSmem = kHalfOffO + 8192 + 1024;
constexpr int kHalfThreads = kChainCompute + 128 + 128;      // + the output warpgroup, 1 warp each to issue MMAs, load, relay and save
constexpr int kBarA = 4, kBarB = 5;                          // the relay warp arrives, the compute warps wait

// The chain of 64 d_v rows, two CTAs to a sequence.  What bounds a chunk is the sequence of hand-offs: 772 cycles of the two
// products that depend on one another and twice the way from an accumulator to the next operand, 1560 - 1760 cycles in all with 1 - 32
// sequences, 1840 - 2090 with saves.  So that way is kept short:
//  - 64-row products put 16 rows on each of a warpgroup's four warps, so all four schedulers of the SM share the epilogues (as the
//    lower half of 128 rows they ran on two), and in fragment layout every thread has half as many elements; tiles are read and
//    staged by ldmatrix / stmatrix instead of element by element;
//  - the compute warps do not poll the products' barriers: a relay warp does, and raises a named barrier, at which they sleep;
//  - what does not depend on h is fetched, and waited for, under the product before: Ut and the scales by the compute warps, tiles
//    and the output accumulator by the MMA warp;
//  - tiles are three deep (the first group two deep: 1.30 times the time of a prompt of 8 x 128 chunks, the second 1.12 times), which
//    leaves room for one staged copy of what goes out.
// Entry state and Delta^T go out by TMA: stored by the compute warps from their fragments in 64-byte pieces, or by others in whole
// rows from the staged tiles, they delay every shared-memory access and wait of the SM (16 of 64: 104 us either way against 94).
// The output, a quarter of that, goes in whole rows of 128 bytes by ordinary stores.  The TMA unit, 64 KB in and 24 KB out a chunk with saves,
// is busy for 1310 - 1370 cycles of it, 580 - 670 without.
// us, as 64 of k_tc_chain_fwd's 128 rows and so, prompts and forwards with saves, both in turn on one box: 4 sequences of 16 chunks
// 27.2 / 24.2, 31.6 / 26.3; 4 of 64 77.6 / 65.0, 99.0 / 77.1; 16 of 64 91.5 / 81.0, 112 / 92.9; 8 of 128 155 / 133.6, 196.5 / 155.7; 32 of 64 115.3 /
// 111.3, 131.3 / 121.3; 72 of 16 54.1 / 54.2, 62.1 / 61.2.  With more sequences HBM takes over (64 of 256: 2120 and 2940 cycles a chunk).
template <bool SAVE>
__global__ void __launch_bounds__(kHalfThreads) k_tc_chain_fwd_half(const __grid_constant__ CUtensorMap mapWt,
                                                                    const __grid_constant__ CUtensorMap mapUt,
                                                                    const __grid_constant__ CUtensorMap mapQg,
                                                                    const __grid_constant__ CUtensorMap mapK,
                                                                    const __grid_constant__ CUtensorMap mapP,
                                                                    const __grid_constant__ CUtensorMap mapHs,
                                                                    const __grid_constant__ CUtensorMap mapDt, ChainParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    // bar_la, bar_lb: tiles loaded; bar_e: every product of a chunk has finished; bar_a, bar_b: products complete; bar_o, bar_of: an output
    // accumulator is complete / has been read; bar_ht, bar_dt: entry state / Delta^T staged (one arrival per compute warp); bar_hf, bar_df: read
    __shared__ uint64_t bar_la[kHalfDeep], bar_lb[kHalfDeep], bar_e[kHalfDeep], bar_a, bar_b, bar_o[2], bar_of[2], bar_ht, bar_dt, bar_hf, bar_df, bar_end;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    __shared__ __align__(16) float sG[kHalfDeep][68];        // per stage: gamma_C / gamma_t for the 64 tokens, then gamma_C

    const int tid = threadIdx.x, warp = warp_index(), wg = warp >> 2, wq = warp & 3, lane = tid & 31;
    constexpr int nb = kChainCompute + 32;                   // participants of a named barrier
    const int bh = blockIdx.x >> 1, v0 = (blockIdx.x & 1) * 64, b = bh / p.H, hh = bh % p.H;

    if (tid == 0) {
        for (int i = 0; i < kHalfDeep; ++i) { mbar_init(&bar_la[i], 1); mbar_init(&bar_lb[i], 1); mbar_init(&bar_e[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&bar_o[i], 1); mbar_init(&bar_of[i], 4); }
        mbar_init(&bar_a, 1); mbar_init(&bar_b, 1); mbar_init(&bar_end, 1);
        mbar_init(&bar_ht, 16); mbar_init(&bar_dt, 16); mbar_init(&bar_hf, 1); mbar_init(&bar_df, 1);
        mbar_init_fence();
        s_abort = 0;
    }
    if (tid < 32) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = uniform(tmem_slot);
    // accumulators: Delta 64 columns, H 128, O 2 x 64; operands, two bf16 per column: h^T 64, Delta^T 32, scaled Delta^T 32
    const uint32_t tD = tbase, tH = tbase + 64, tO0 = tbase + 192, aH = tbase + 320, aD = tbase + 384;
    const uint32_t aDs = p.scaled ? tbase + 416 : aD;        // all factors 1: the scaled copy is Delta itself
    const uint32_t lane_base = (uint32_t)wq * 32;

    // bounded wait; once any wait has expired every later wait returns at once: every warp still comes to every barrier, the results
    // are garbage, the status word says so.
    // The named barriers come in the order H, A, D, B, H, ...  Whoever arrives without waiting (bar.arrive) must not come to the same
    // barrier again before its phase is over: the second arrival would stand for that of a warp still to come, and that warp would
    // then wait for good.  It cannot, because the relay warp raises A of a chunk only when the MMA warp has passed H, and B when it has passed D:
    //  - a compute warp comes to D again behind the next A, so after the MMA warp has passed the next H and with it this D; to H
    //    again behind A and B of the chunk, so after the MMA warp has passed this H;
    //  - the relay warp comes to A (B) again after the MMA warp has passed the next H (D), to which every compute warp
    //    came from behind this A (B).
    // That a product is complete says that the MMA warp has passed the barrier before it, so the relay warp waits for the products of a
    // chunk whether a wait has expired or not: the MMA warp, which waits for nothing else by then, issues them all the same.
    auto wait = [&](uint64_t* bar, uint32_t parity) { return mbar_try_wait(bar, parity) || wait_on(bar, parity, s_abort, p.status); };
    const int tok0 = p.n0 * C;                               // first token; rows and tiles of the workspace start at
    const size_t row0 = (size_t)bh * p.Tp + tok0, tile0 = (size_t)bh * p.Ns + p.n0;

    if (warp < kOutWarp) {
        // ---------------------------------- compute warps ----------------------------------
        // fragments: rows r0, r0 + 8 of the CTA's 64; of every 8 columns two, ft and ft + 1
        const int ft = 2 * (lane & 3), r0 = 16 * wq + (lane >> 2);
        float h[16];          // h^T: [4 (8 d_k columns from 32 wg on)][2 (row)][2 (column)]
        const size_t hat = (size_t)bh * D * D + (size_t)(32 * wg + ft) * D + v0 + r0;
        auto at = [](int x) { return (size_t)(8 * (x >> 2) + (x & 1)) * D + 8 * ((x >> 1) & 1); };
        if (p.h0_late) grid_dep_wait();
#pragma unroll
        for (int x = 0; x < 16; ++x) h[x] = p.h0 ? __ldcg(p.h0 + hat + at(x)) : 0.f;        // not from L1: it may be new
        grid_dep_wait();                  // the loads of h0 (an input) are in flight; everything below depends on the prep kernel
        grid_dep_launch();
        const int rl = lane & 15, cl = lane >> 4;             // the row and the 16-byte chunk that this lane addresses for stsm4, ldsm4
        unsigned char *sHs = smem + kHalfOffS + (wg >> 1) * 8192, *sDt = smem + kHalfOffS + 16384;
        auto staged = [&](uint64_t* bar) { fence_proxy_async(); __syncwarp(); if (lane == 0) mbar_arrive(bar); };
        // the state as operand, and staged as the entry state of chunk n
        auto put_h = [&](int n) {
            uint32_t r[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) r[i] = pack_bf16(h[2 * i], h[2 * i + 1]);
            tmem_st_frag4(tmem_addr(aH, lane_base, wg * 16), r);
            tmem_st_wait();
            tc_fence_before();
            nb_arrive(kBarH, nb);
            if (SAVE && n < p.N) {
                if (n > 0) wait(&bar_hf, (n - 1) & 1);
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 2; ++i) stsm4<false>(sHs + sw128_chunk(16 * wq + rl, (wg & 1) * 4 + 2 * i + cl), r + 4 * i);
                staged(&bar_ht);
            }
        };
        put_h(0);
        int s = 0;
        uint32_t sp = 0;
        uint32_t u[4];                    // Ut of the chunk, [2 (8 tokens)][2 (row)], and its scales
        float2 f0, f1;
        float gamN;
        auto fetch = [&]() {
            wait(&bar_la[s], sp);
            __syncwarp();
            ldsm4<false>(smem + s * kHalfStageA + 16384 + sw128_chunk(16 * wq + rl, 2 * wg + cl), u);
            f0 = *reinterpret_cast<const float2*>(&sG[s][16 * wg + ft]);
            f1 = *reinterpret_cast<const float2*>(&sG[s][16 * wg + 8 + ft]);
            gamN = sG[s][64];
            if (++s == kHalfDeep) { s = 0; sp ^= 1; }
        };
        fetch();
        for (int n = 0; n < p.N; ++n) {
            const float gamC = gamN;
            nb_sync(kBarA, nb);
            tc_fence_after();
            // Delta^T = Ut - acc, my 16 tokens, as operands: plain, and scaled by gamma_C/gamma_r
            {
                float v[8];
                tmem_ld_frag2(tmem_addr(tD, lane_base, wg * 16), v);
                tmem_ld_wait();
                uint32_t r[4], rs[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float2 f = m < 2 ? f0 : f1;
                    const float x = __uint_as_float(u[m] << 16) - v[2 * m], y = __uint_as_float(u[m] & 0xffff0000u) - v[2 * m + 1];
                    r[m] = pack_bf16(x, y);
                    rs[m] = pack_bf16(x * f.x, y * f.y);
                }
                if (p.scaled) tmem_st_frag2(tmem_addr(aDs, lane_base, wg * 8), rs);
                tmem_st_frag2(tmem_addr(aD, lane_base, wg * 8), r);
                tmem_st_wait();
                tc_fence_before();
                nb_arrive(kBarD, nb);
                if (SAVE) {
                    if (n > 0) wait(&bar_df, (n - 1) & 1);
                    __syncwarp();
                    stsm4<false>(sDt + sw128_chunk(16 * wq + rl, 2 * wg + cl), r);
                    staged(&bar_dt);
                }
            }
            if (n + 1 < p.N) fetch();     // under the product
            // h^T <- gamma_C h^T + acc (my 32 d_k columns), refresh the operand
            nb_sync(kBarB, nb);
            tc_fence_after();
            {
                float v[16];
                tmem_ld_frag4(tmem_addr(tH, lane_base, wg * 32), v);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 16; ++i) h[i] = fmaf(gamC, h[i], v[i]);
            }
            put_h(n + 1);
        }
        if (p.hT && !s_abort) {
#pragma unroll
            for (int x = 0; x < 16; ++x) p.hT[hat + at(x)] = h[x];
        }
    } else if (warp < kMmaWarp) {
        // ---------------------------------- output warps ----------------------------------
        // O^T of a chunk, 16 rows to a warp -> token-major tile -> 16 tokens to a warp
        unsigned char* sO = smem + kHalfOffO;
        const size_t pitch = (size_t)p.H * D;
        bf16* o = p.o + (size_t)b * p.T * pitch + (size_t)hh * D + v0 + 8 * (lane & 7);
        grid_dep_wait();                  // the chain before may take longer than a wait has (tc_fwd_parts)
        for (int n = 0; n < p.N; ++n) {
            const int ob = n & 1;
            wait(&bar_o[ob], (n >> 1) & 1);
            __syncwarp();
            tc_fence_after();
            float v[2][16];
#pragma unroll
            for (int i = 0; i < 2; ++i) tmem_ld_frag4(tmem_addr(tO0 + 64 * ob, lane_base, 32 * i), v[i]);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_of[ob]);          // the accumulator may be written again
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t r[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) r[m] = pack_bf16(v[i >> 1][8 * (i & 1) + 2 * m], v[i >> 1][8 * (i & 1) + 2 * m + 1]);
                stsm4<true>(sO + sw128_chunk(16 * i + 8 * (lane >> 4) + (lane & 7), 2 * wq + ((lane >> 3) & 1)), r);
            }
            nb_sync(kBarOut, 128);
            uint4 x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const uint4*>(sO + sw128_chunk(16 * wq + 4 * i + (lane >> 3), lane & 7));
            nb_sync(kBarOut, 128);                            // the tile may be written again
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = tok0 + n * C + 16 * wq + 4 * i + (lane >> 3);
                if (t < p.T) *reinterpret_cast<uint4*>(o + t * pitch) = x[i];      // rows past the end of the sequence are skipped
            }
        }
    } else if (warp == kMmaWarp) {
        // ---------------------------------- MMA-issue warp, converged ----------------------------------
        const uint32_t issue = elect_lane();
        grid_dep_wait();
        grid_dep_launch();
        int s = 0;
        uint32_t sp = 0;
        wait(&bar_la[0], 0);
        for (int n = 0; n < p.N; ++n) {
            const int ob = n & 1, st = s;
            const uint32_t stA = smem_u32(smem) + s * kHalfStageA, stB = smem_u32(smem) + kHalfOffB + s * kHalfStageB;
            const uint32_t tO = tO0 + 64 * ob;
            nb_sync(kBarH, nb);                               // h^T operand of chunk n is in place
            tc_fence_after();
            // Delta-accumulator = h^T Wt (B: MN-major, lines = d_k)
            umma_product_ts_w<true, 64>(tD, aH, stA, 8192, C, D, false, issue);
            umma_commit_w(&bar_a, issue);
            // O-accumulator = h^T Qg^T (B: K-major); it reads the operand that the h update rewrites, so the commit
            // behind the H product below (which releases that update) must cover it
            wait(&bar_lb[s], sp);
            umma_product_ts_w<false, 64>(tO, aH, stB, 8192, C, D, false, issue);
            if (++s == kHalfDeep) { s = 0; sp ^= 1; }
            if (n + 1 < p.N) {                                // what the next chunk needs besides h^T, while there is time
                wait(&bar_la[s], sp);
                if (n > 0) wait(&bar_of[ob ^ 1], ((n - 1) >> 1) & 1);
            }
            nb_sync(kBarD, nb);                               // Delta^T operands of chunk n are in place
            tc_fence_after();
            // H-accumulator = scaled Delta^T K (B: MN-major, lines = tokens)
            umma_product_ts_w<true, 64>(tH, aDs, stB + 16384, 8192, D, C, false, issue);
            umma_commit_w(&bar_b, issue);
            // O-accumulator += Delta^T P^T (B: K-major [r][s])
            umma_product_ts_w<false, 64>(tO, aD, stB + 32768, 8192, C, C, true, issue);
            umma_commit_w(&bar_o[ob], issue);
            if (n + kHalfDeep < p.N) umma_commit_w(&bar_e[st], issue);      // the load warp waits for these: nothing arrives in a CTA that has left
        }
        nb_sync(kBarH, nb);                                   // final arrival of the compute warps
        umma_commit_w(&bar_end, issue);                       // leaves when its products have come to their end, whatever has expired
        mbar_drain(&bar_end, 0);
    } else if (warp == kMmaWarp + 1) {
        // ---------------------------------- TMA load warp ----------------------------------
        const bool lead = lane == 0;
        grid_dep_wait();                  // the tiles and the log-decays read below are written by the prep kernel
        grid_dep_launch();
        TokenScales ts(p.g, p.rk, row0, lane);
        auto load = [&](int n, int s) {                       // by the whole warp
            ts.put(sG[s]);
            __syncwarp();
            if (lead) {
                const int yc = (int)((tile0 + n) * D), yt = (int)(row0 + (size_t)n * C);
                unsigned char *sa = smem + s * kHalfStageA, *sb = smem + kHalfOffB + s * kHalfStageB;
                mbar_expect_tx(&bar_la[s], kHalfStageA);
                tma_load_2d(sa, &mapWt, 0, yc, &bar_la[s]);
                tma_load_2d(sa + 16384, &mapUt, 0, yc + v0, &bar_la[s]);
                mbar_expect_tx(&bar_lb[s], kHalfStageB);
                tma_load_2d(sb, &mapQg, 0, yt, &bar_lb[s]);
                tma_load_2d(sb + 8192, &mapQg, 64, yt, &bar_lb[s]);
                tma_load_3d(sb + 16384, &mapK, hh * D, tok0 + n * C, b, &bar_lb[s]);
                tma_load_3d(sb + 16384 + 8192, &mapK, hh * D + 64, tok0 + n * C, b, &bar_lb[s]);
                tma_load_2d(sb + 32768, &mapP, 0, yt, &bar_lb[s]);
            }
            if (n + 1 < p.N) ts.fetch(n + 1);
        };
        ts.fetch(0);
        int loads = 0;
        for (; loads < kHalfDeep && loads < p.N; ++loads) load(loads, loads);
        int s = 0;
        uint32_t sp = 0;
        for (; loads < p.N; ++loads) {
            wait(&bar_e[s], sp);                              // every product of the chunk three before has finished: refill its buffers
            if (!__all_sync(0xffffffffu, !s_abort)) break;    // one answer for the warp
            load(loads, s);
            if (++s == kHalfDeep) { s = 0; sp ^= 1; }
        }
        if (lead) { mbar_drain_ring(bar_la, kHalfDeep, loads); mbar_drain_ring(bar_lb, kHalfDeep, loads); }      // leaves when its loads have come
    } else if (warp == kMmaWarp + 2) {
        // ---------------------------------- relay warp ----------------------------------
        grid_dep_wait();
        auto relay = [&](uint64_t* bar, uint32_t parity, int id) {
            if (!wait(bar, parity)) mbar_drain(bar, parity);
            tc_fence_after();
            tc_fence_before();
            __syncwarp();
            nb_arrive(id, nb);
        };
        for (int n = 0; n < p.N; ++n) {
            relay(&bar_a, n & 1, kBarA);
            relay(&bar_b, n & 1, kBarB);
        }
    } else {
        // ---------------------------------- saving warp ----------------------------------
        if (lane == 0 && SAVE) {
            grid_dep_wait();
            save_chunks<1>(&mapHs, &mapDt, tile0 * D + v0, p.N, smem + kHalfOffS, 8192, smem + kHalfOffS + 16384, 0, &bar_ht, &bar_hf, &bar_dt, &bar_df, wait);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid < 32) tmem_dealloc(tbase, 512);
}

template <class K>
cudaError_t set_smem(K kern, size_t bytes) { return set_max_smem_once(reinterpret_cast<const void*>(kern), bytes); }

}  // namespace

bool tc_supported(const qd_shape& s) {
    return s.dtype == QD_BF16 && s.dk == 128 && s.dv == 128 && s.chunk == kChunk &&
           (long long)s.B * s.H * tc_padded_T(s) * 128 < 0x7fffffffLL * 64;
}

// Two CTAs per sequence while every CTA still gets an SM of its own.  us, two against one, prompt / with saves / backward: 74
// sequences of 8 chunks 29.7 31.4 / 32.5 36.9 / 45.1 48.8, of 64 203 209 / 230 249 / 298 313; 75 of 8 42.2 35.3 / 46.0 41.7 / 59.2 53.5,
// of 64 245 199 / 284 236 / 351 299.
int chain_rows(uint64_t BH) { return 2 * BH <= kSMs ? 64 : 128; }

TcLayout tc_layout(const qd_shape& s) {
    TcLayout L{};
    const size_t BH = (size_t)s.B * s.H, T = (size_t)tc_padded_T(s);
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = (off + bytes + 1023) & ~(size_t)1023; return o; };
    L.status = take(256);
    L.next = L.status + 128;
    L.g = take(BH * T * 4);
    L.Qg = take(BH * T * s.dk * 2);
    L.P = take(BH * T * kChunk * 2);
    L.Wt = take(BH * T * s.dk * 2);
    L.Ut = take(BH * T * s.dv * 2);
    L.rqk = take(2 * BH * T * 4);
    L.fwd_end = off;
    const size_t N = T / kChunk;
    L.Mt = take(BH * T * kChunk * 2);
    L.hsT = take(BH * N * s.dk * s.dv * 2);
    L.Dt = take(BH * T * s.dv * 2);
    L.dhsT = take(BH * N * s.dk * s.dv * 2);
    L.dDt = take(BH * T * s.dv * 2);
    L.bwd_end = off;
    return L;
}

namespace {

struct PrepCall { CUtensorMap mQ, mK, mV, mUt, mWt, mP; PrepParams p; };
struct ChainCall { CUtensorMap mWt, mUt, mQg, mK, mP, mHs, mDt, mO; ChainParams p; };

bool setup(const ChunkArgs& a, PrepCall& c) {
    const qd_shape& s = a.s;
    const int Tp = tc_padded_T(s);
    const uint64_t trows = (uint64_t)s.B * s.H * (Tp / kChunk) * D;          // rows of the [chunk][d][64] tiles
    if (!make_tmap_tokens(&c.mQ, a.q, s.B, s.T, s.H, D, 64) || !make_tmap_tokens(&c.mK, a.k, s.B, s.T, s.H, D, 64) ||
        !make_tmap_tokens(&c.mV, a.v, s.B, s.T, s.H, D, 64) ||
        !make_tmap_bf16_2d(&c.mUt, a.ws + a.TL.Ut, 64, trows, 128, 128) ||
        !make_tmap_bf16_2d(&c.mWt, a.ws + a.TL.Wt, 64, trows, 128, 128) ||
        !make_tmap_bf16_2d(&c.mP, a.ws + a.TL.P, 64, (uint64_t)s.B * s.H * Tp, 128, 64))
        return false;
    PrepParams& p = c.p;
    p = PrepParams{};
    p.T = s.T; p.Tp = Tp; p.H = s.H; p.N = (s.T + kChunk - 1) / kChunk; p.Ns = Tp / kChunk; p.BH = s.B * s.H;
    p.rqk = a.norm ? (float*)(a.ws + a.TL.rqk) : nullptr;
    p.beta = (const bf16*)a.beta; p.alpha = (const bf16*)a.alpha; p.lam = (const bf16*)a.lam;
    p.g = (float*)(a.ws + a.TL.g);
    p.Qg = (bf16*)(a.ws + a.TL.Qg);
    p.Mt = a.save ? (bf16*)(a.ws + a.TL.Mt) : nullptr;
    p.status = (unsigned*)(a.ws + a.TL.status);
    return true;
}
cudaError_t launch(const ChunkArgs& a, const PrepCall& c) {
    auto kern = a.norm ? (a.logits ? k_tc_prep<true, true> : k_tc_prep<true, false>)
                       : (a.logits ? k_tc_prep<false, true> : k_tc_prep<false, false>);
    cudaError_t e = set_smem(kern, kPrepSmem);
    if (e != cudaSuccess) return e;
    return launch_overlapped(kern, dim3((unsigned)(c.p.BH * c.p.N)), dim3(kPrepThreads), kPrepSmem, a.stream, c.mQ, c.mK, c.mV, c.mUt,
                             c.mWt, c.mP, c.p);
}

bool setup(const ChunkArgs& a, ChainCall& c) {
    const qd_shape& s = a.s;
    const int Tp = tc_padded_T(s);
    const uint64_t BH = (uint64_t)s.B * s.H, Ns = Tp / kChunk, N = (s.T + kChunk - 1) / kChunk;
    const int rows = chain_rows(BH);
    if (!make_tmap_bf16_2d(&c.mHs, a.ws + a.TL.hsT, D, BH * Ns * D, D * 2, rows) ||
        !make_tmap_bf16_2d(&c.mDt, a.ws + a.TL.Dt, 64, BH * Ns * D, 128, rows) ||
        (rows == D && !make_tmap_tokens(&c.mO, a.o, s.B, s.T, s.H, D, 32)) ||
        !make_tmap_bf16_2d(&c.mWt, a.ws + a.TL.Wt, 64, BH * Ns * D, 128, 128) ||
        !make_tmap_bf16_2d(&c.mUt, a.ws + a.TL.Ut, 64, BH * Ns * D, 128, rows) ||
        !make_tmap_bf16_2d(&c.mQg, a.ws + a.TL.Qg, D, BH * Tp, D * 2, 64) ||
        !make_tmap_tokens(&c.mK, a.k, s.B, s.T, s.H, D, 64) ||
        !make_tmap_bf16_2d(&c.mP, a.ws + a.TL.P, 64, BH * Tp, 128, 64))
        return false;
    ChainParams& p = c.p;
    p = ChainParams{};
    p.Tp = Tp; p.H = s.H; p.N = (int)N; p.Ns = (int)Ns;
    p.g = (const float*)(a.ws + a.TL.g);
    p.h0 = a.h0; p.hT = a.hT;
    p.T = s.T; p.o = (bf16*)a.o;
    p.scaled = (a.alpha || a.norm) ? 1 : 0;
    p.rk = a.norm ? (const float*)(a.ws + a.TL.rqk) + BH * Tp : nullptr;
    p.status = (unsigned*)(a.ws + a.TL.status);
    return true;
}
cudaError_t launch(const ChunkArgs& a, const ChainCall& c) {
    const uint64_t BH = (uint64_t)a.s.B * a.s.H;
    const int rows = chain_rows(BH);
    if (rows != D) {
        const auto half = a.save ? k_tc_chain_fwd_half<true> : k_tc_chain_fwd_half<false>;
        cudaError_t e = set_smem(half, kHalfSmem);
        if (e != cudaSuccess) return e;
        return launch_overlapped(half, dim3((unsigned)(2 * BH)), dim3(kHalfThreads), kHalfSmem, a.stream, c.mWt, c.mUt, c.mQg, c.mK, c.mP,
                                 c.mHs, c.mDt, c.p);
    }
    const auto kern = a.save ? k_tc_chain_fwd<true> : k_tc_chain_fwd<false>;
    cudaError_t e = set_smem(kern, kChainSmem);
    if (e != cudaSuccess) return e;
    return launch_overlapped(kern, dim3((unsigned)BH), dim3(kChainThreads), kChainSmem, a.stream, c.mWt, c.mUt, c.mQg,
                             c.mK, c.mP, c.mHs, c.mDt, c.mO, c.p);
}

}  // namespace

cudaError_t tc_prep(const ChunkArgs& a) {
    PrepCall c;
    return setup(a, c) ? launch(a, c) : cudaErrorInvalidValue;
}

cudaError_t tc_chain_fwd(const ChunkArgs& a) {
    ChainCall c;
    return setup(a, c) ? launch(a, c) : cudaErrorInvalidValue;
}

// With few sequences the forward chain, two CTAs to a sequence, leaves SMs idle for as long as its dependent chunks take.  A
// sequence is then taken in parts, and the preparation of a part runs beside the chain of the part before it:
//     prep 0, chain 0, prep 1, chain 1, ...
// in one stream, by programmatic launch alone.  prep i + 1 may start when every CTA of chain i has begun its work, which it does
// when prep i has completed (and so everything before that); it reads inputs and writes the workspace rows of its own chunks, so
// it need not wait.  Its first CTA waits for chain i before it leaves, so when prep i + 1 has completed chain i has too, and
// chain i + 1, which waits for prep i + 1, finds the state that chain i left: in h_T, or without one in the section that the
// reverse chain fills later.  The state is passed on in fp32, so the results are those of one part, bit for bit.
// Where: with up to 40 sequences (68 SMs idle), from 64 chunks and 1.7 loads of the GPU with preparations (1024 chunks) on.  One, two, three
// parts, us, prompts; with saves: 16 sequences of 64 chunks 88.8 / 82.8 / 84.3; 98.8 / 93.3 / 96.4.  32 of 64 116.7 / 111.7 / 113.3; 128.4 / 121.3 /
// 122.9.  40 of 64 129.3 / 126.0 / 130.9; 143.9 / 139.4 / 146.3.  8 of 128 140.5 / 133.9 / 133.9; 161.5 / 155.7 / 157.4.  But 8 of 64 71.0 / 70.6; 83.4 /
// 83.7.  40 of 32 69.3 / 71.4; 76.8 / 78.6.  44 of 64 136.7 / 137.1; 155.0 / 152.6.  48 of 64 143.0 / 146.1; 162.1 / 163.9.  64 of 256 744 / 757;
// 859 / 867.  (From 128 chunks on 41 to 48 sequences would gain 2 - 5 %: 48 of 128 287 / 281; 326 / 316, 48 of 256 593 / 576; 672 / 646.)  Three of them
// from 256 chunks on: 32 of 512 877 / 779 / 749; 990 / 891 / 854.  16 of 512 637 / 578 / 564; 715 / 659 / 646.  40 of 256 521 / 489 / 487; 585 / 545 /
// 542.  4 of 256 246 / 239 / 240; 287 / 280 / 284.  With 128 chunks the third part gives 0 - 2 % (32 sequences 221 / 201 / 200, 40 247 / 235 / 239).
// The parts are equal.  A third of 32 x 512 chunks takes the chain about 190 us, and the preparation beside it, on 84 SMs, 240 - 250.
int tc_fwd_parts(const ChunkArgs& a) {
    const long long BH = (long long)a.s.B * a.s.H, N = (a.s.T + kChunk - 1) / kChunk;
    if (BH > 40 || N < 64 || BH * N < 1024 || !(a.hT || a.save)) return 1;
    return N < 256 ? 2 : 3;
}

cudaError_t tc_fwd(const ChunkArgs& a, int parts) {
    PrepCall pc;
    ChainCall cc;
    if (!setup(a, pc) || !setup(a, cc)) return cudaErrorInvalidValue;
    const int N = pc.p.N;
    float* carry = a.hT ? a.hT : (float*)(a.ws + a.TL.dhsT);             // [BH][D][D]; dhsT has as much from two chunks on
    for (int i = 0; i < parts; ++i) {
        const int n0 = (int)((long long)N * i / parts), n1 = (int)((long long)N * (i + 1) / parts);
        const bool last = i + 1 == parts;
        pc.p.n0 = cc.p.n0 = n0;
        pc.p.N = cc.p.N = n1 - n0;
        pc.p.beside = cc.p.h0_late = i > 0;
        if (i > 0) cc.p.h0 = carry;
        cc.p.hT = last ? a.hT : carry;
        cudaError_t e = launch(a, pc);
        if (e == cudaSuccess) e = launch(a, cc);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace qd
