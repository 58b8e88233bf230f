// Tensor-core (tcgen05 / TMEM / TMA) chunkwise backward for bf16, d_k = d_v = 128, chunk 64.
//
// The paper prints no backward pass; these kernels evaluate the exact gradient of the chunk
// equations of Section 3.3.2 (see the forward kernels for the notation):
//   k_tc_chain_bwd  one CTA per (batch, head), or two that share its d_v rows (chain_rows), chunks in REVERSE order, dh^T
//                   (fp32) in registers:
//                     dDelta^T = dO^T P + diag-scaled (dh^T K^T)          (scale gamma_C/gamma_s per token s)
//                     dh^T <- gamma_C dh^T + dO^T Qg - dDelta^T W<-
//                   leaves per chunk dDelta^T and the bf16 dh^T at the chunk's exit.
//   k_tc_chunk_bwd  one CTA per SM, a chunk at a time: every remaining product (dP, dT, dA = -M^T dM M^T, dX, ...),
//                   d_k/d_v-shaped results transposed (d index on the 128 TMEM lanes), 64 x 64-shaped
//                   ones in natural orientation as 64-row instructions, 16 rows on each warp of a warpgroup;
//                   row dot-products that run across lanes use a warp-shuffle column reduction.
// All waits are bounded (see tc_fwd.cu).
#include "chain.cuh"
#include "internal.h"
#include "sm100.cuh"

namespace qd {
namespace {
using namespace sm100;
typedef __nv_bfloat16 bf16;

constexpr int C = kChunk;      // 64
constexpr int D = 128;         // d_k = d_v

// One halving step of a column sum across the lanes of a warp: lanes whose `off` bit is set keep the upper half
// of the N values, the others the lower half; each adds what its partner sends.
template <int N>
__device__ __forceinline__ void fold(float* v, int lane, int off) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
        const float keep = up ? v[N / 2 + k] : v[k];
        const float send = up ? v[k] : v[N / 2 + k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
}

// =================================================================================================
struct ChainBwdParams {
    int Tp, H, N, Ns;          // N chunks of a sequence, from n0 on; Tp = 64 Ns rows per sequence in the workspace
    int n0;
    int dhT_early;             // the kernel before this one in the stream is the library's own: dhT is older than it
    const float* rk;           // non-null (QD_NORM_QK): 1/|k_t| per workspace row, folded into the per-token scale
    const float* g;
    const float* dhT;
    float* dh0;
    unsigned* status;
    unsigned* next;            // three counters, zeroed here for k_tc_chunk_bwd; null: they are already
};

// Tiles of a chain's chunk in shared memory: K 16K | P 8K, three deep; Qg 16K | dO 16K and Wt 16K, two deep; staged for their
// stores, one deep: dh^T 32K | dDelta^T 16K; with 64 rows dO, dh^T and dDelta^T have half the size, and are staged two deep; then
// the per-token scales.
constexpr int kDeepK = 3, kBytesK = 24576;
constexpr int kOffQ = kDeepK * kBytesK, kOffG = kOffQ + 2 * (32768 + 16384) + 32768 + 16384;
constexpr int kChainSmem = kOffG + (kDeepK + 1) * 68 * 4 + 1024;
constexpr int kChainCompute = 512;                 // 16 epilogue warps: 4 warpgroups split the accumulator columns
constexpr int kChainThreads = kChainCompute + 96;  // + 1 MMA-issue warp, 1 warp each for saves and TMA loads
constexpr int kMmaWarp = kChainCompute / 32;

// named barriers of the chain: compute threads arrive, the MMA warp waits (they run in lock-step)
constexpr int kBarH = 1, kBarD = 2;

// A barrier per buffer where one side may run ahead.  k, q, w: tiles loaded; fk, fq, fw: read by their last product; ht, dt:
// staged (one arrival per compute warp); hf, df: read by their store (two deep: hf alone, for both); a, b: products complete;
// end: all of them.
struct ChainBars { uint64_t k[kDeepK], fk[kDeepK], q[2], fq[2], w[2], fw[2], hf[2], df, a, b, end, ht[2], dt[2]; };

// Reverse state chain.  Per chunk the dependency is
//   dh ready -> A2 = dh^T K^T -> dDelta^T -> H-accumulator -= dDelta^T W<- -> dh update;
// A1 = dO^T P and the dO^T Qg part of the H-accumulator do not depend on dh and are issued a chunk ahead (double-buffered
// H-accumulator).  As in the forward chain, the dependent operands (dh^T, -dDelta^T) live in tensor memory and the issuing
// warp stays converged.  With few sequences two CTAs share the d_v rows of one (ROWS = 64).
// With 128 rows what bounds a chunk is HBM if there are many sequences; with few (2500 cycles) the SM's TMA unit, which is busy for
// 2200 of them: 72 KB in at 98 - 113 bytes per cycle and 48 KB out at 32, which add up.  With 64 it is the sequence of hand-offs (1930
// cycles with 1 - 32 sequences, of which TMA 1310 - 1370), so nothing that can be elsewhere is on it: a wait that has long been
// satisfied costs 100 - 200 cycles, so the next chunk's scales are waited for under the last product, one barrier stands for both
// staged tiles, the tiles are staged two deep, and a wait polls before it looks at the abort flag (4 sequences of 64 chunks, backward,
// 92 -> 85 us when that was done).
// Compute warpgroup w owns tokens [16w, 16w+16) of the 64-column accumulators and d_k columns
// [32w, 32w+32) of dh^T; thread l of a warpgroup owns TMEM lane l = d_v index.
template <int ROWS>
__global__ void __launch_bounds__(kChainThreads) k_tc_chain_bwd(const __grid_constant__ CUtensorMap mapWt,
                                                                const __grid_constant__ CUtensorMap mapdO,
                                                                const __grid_constant__ CUtensorMap mapQg,
                                                                const __grid_constant__ CUtensorMap mapK,
                                                                const __grid_constant__ CUtensorMap mapP,
                                                                const __grid_constant__ CUtensorMap mapdHs,
                                                                const __grid_constant__ CUtensorMap mapdDt,
                                                                ChainBwdParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    constexpr int rows = ROWS, bytesQ = 16384 + rows * 128, offW = kOffQ + 2 * bytesQ;
    constexpr int two = rows == D ? 0 : 1, bytesS = rows * 384;       // staged tiles: two deep or not
    unsigned char* stg = smem + offW + 2 * 16384;      // dh^T [rows dv][128 dk], 2 blocks of [rows lines][64]; dDelta^T [rows dv][64 tokens]
    __shared__ ChainBars bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    // gamma_C / gamma_t for the 64 tokens, then gamma_C; written by the load warp before it arrives on bar.k.  One deeper than
    // K and P: those are dead when A2 is complete, but the epilogue reads these after that
    float (*sG)[68] = reinterpret_cast<float (*)[68]>(smem + kOffG);

    const int tid = threadIdx.x, warp = warp_index(), wg = warp >> 2, l = tid & 127, wq = warp & 3;
    constexpr int nwq = rows / 32, nb = 4 * rows + 32;               // warps of a warpgroup that have rows; barrier participants
    constexpr int parts = D / rows;
    const int bh = blockIdx.x / parts, v0 = (blockIdx.x % parts) * rows, b = bh / p.H, hh = bh % p.H;

    if (tid == 0) {
        uint64_t* all = bar.k;
        for (int i = 0; i < (int)(sizeof(ChainBars) / 8); ++i) mbar_init(all + i, all + i >= bar.ht ? 4 * nwq : 1);
        mbar_init_fence();
        s_abort = 0;
    }
    if (tid < 32) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = uniform(tmem_slot);
    // accumulators: A1, A2 64 columns each, H 2 x 128; operands, two bf16 per column: dh^T 64, -dDelta^T 32
    const uint32_t tA1 = tbase, tA2 = tbase + 64, tH0 = tbase + 128, aH = tbase + 384, aD = tbase + 448;
    const uint32_t lane_base = (uint32_t)wq * 32;

    // bounded wait; once any wait has expired every later wait returns at once (the kernel drains)
    auto wait = [&](uint64_t* br, uint32_t parity) { return mbar_try_wait(br, parity) || wait_on(br, parity, s_abort, p.status); };
    const int tok0 = p.n0 * C;                                       // first token; rows and tiles of the workspace start at
    const size_t row0 = (size_t)bh * p.Tp + tok0, tile0 = (size_t)bh * p.Ns + p.n0;

    if (warp < kMmaWarp && wq >= nwq) {
        // lanes without a row: straight to the end
    } else if (warp < kMmaWarp) {
        // ---------------------------------- compute warps ----------------------------------
        float dh[32];     // dh^T[j = l][32 wg .. 32 wg + 31]
        // dhT is an input of the call.  When the kernel before this one is the library's own forward chain, dhT is older
        // than that kernel and may be read while it drains; otherwise the predecessor may be the very kernel that wrote
        // dhT, whose writes are only guaranteed visible after the wait.
        if (!p.dhT_early) grid_dep_wait();
        const size_t at = (size_t)bh * D * D + (size_t)(32 * wg) * D + v0 + l;
#pragma unroll
        for (int i = 0; i < 32; ++i) dh[i] = p.dhT ? __ldcg(p.dhT + at + (size_t)i * D) : 0.f;      // not from L1: it may be new
        if (p.dhT_early) grid_dep_wait();  // the loads of dhT are in flight; everything below depends on earlier kernels
        grid_dep_launch();
        auto arrive = [&](uint64_t* b) { __syncwarp(); if ((tid & 31) == 0) mbar_arrive(b); };
        auto staged = [&](uint64_t* b) { fence_proxy_async(); arrive(b); };      // my part of a tile is in shared memory, for its store
        // dh as operand: my 32 columns are 16 packed columns of tensor memory; then as a tile for its store
        auto put_h = [&]() {
            uint32_t r[8];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
#pragma unroll
                for (int e = 0; e < 8; ++e) r[e] = pack_bf16(dh[q * 16 + 2 * e], dh[q * 16 + 2 * e + 1]);
                tmem_st8(tmem_addr(aH, lane_base, wg * 16 + q * 8), r);
            }
            tmem_st_wait();
            tc_fence_before();
            nb_arrive(kBarH, nb);
        };
        int pending = 0;                  // barriers of the MMA warp that a warp which gives up has not been to
        int s = 0;
        uint32_t sp = 0;
        wait(&bar.k[0], 0);
        for (int it = 0; it < p.N; ++it) {
            put_h();
            const int sb = it & two;
            unsigned char* sdH = stg + sb * bytesS;
            if (it > two) wait(&bar.hf[sb], ((it >> two) - 1) & 1);       // the tile (two deep: both) has been read by the store before
            // 64-column block wg >> 1, 16-byte chunks 4 (wg & 1) ..
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) sts128(sdH + (wg >> 1) * (rows * 128) + sw128_chunk(l, (wg & 1) * 4 + ch), pack8(dh + ch * 8));
            staged(&bar.ht[sb]);
            const float gamC = sG[it & 3][64];
            if (!__all_sync(0xffffffffu, wait(&bar.a, it & 1))) { pending = 2 * (p.N - it) - 1; break; }
            tc_fence_after();
            // dDelta^T = A1 + gamma_C/gamma_s A2, my 16 tokens; negated as operand
            {
                float a1[16], a2[16];
                tmem_ld16(tmem_addr(tA1, lane_base, wg * 16), a1);
                tmem_ld16(tmem_addr(tA2, lane_base, wg * 16), a2);
                const float4* gp = reinterpret_cast<const float4*>(&sG[it & 3][wg * 16]);
                tmem_ld_wait();
                uint32_t r[8], rn[8];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 t = gp[q];
                    r[2 * q] = pack_bf16(fmaf(t.x, a2[4 * q], a1[4 * q]), fmaf(t.y, a2[4 * q + 1], a1[4 * q + 1]));
                    r[2 * q + 1] = pack_bf16(fmaf(t.z, a2[4 * q + 2], a1[4 * q + 2]), fmaf(t.w, a2[4 * q + 3], a1[4 * q + 3]));
                    rn[2 * q] = r[2 * q] ^ 0x80008000u; rn[2 * q + 1] = r[2 * q + 1] ^ 0x80008000u;
                }
                tmem_st8(tmem_addr(aD, lane_base, wg * 8), rn);
                tmem_st_wait();
                tc_fence_before();
                nb_arrive(kBarD, nb);
                unsigned char* sdD = sdH + rows * 256;
                if (!two && it > 0) wait(&bar.df, (it - 1) & 1);
                sts128(sdD + sw128_chunk(l, wg * 2), make_uint4(r[0], r[1], r[2], r[3]));
                sts128(sdD + sw128_chunk(l, wg * 2 + 1), make_uint4(r[4], r[5], r[6], r[7]));
                staged(&bar.dt[sb]);
            }
            // A chunk's K and P may be reloaded as soon as A2 is complete, which the announcement of its dh^T sets off: so
            // the scales of the next chunk are waited for before that, not after (where the barrier could have come round)
            if (++s == kDeepK) { s = 0; sp ^= 1; }
            if (it + 1 < p.N) wait(&bar.k[s], sp);
            if (!__all_sync(0xffffffffu, wait(&bar.b, it & 1))) { pending = 2 * (p.N - it) - 2; break; }
            tc_fence_after();
            {
                float v[32];
                tmem_ld32(tmem_addr(tH0 + 128 * (it & 1), lane_base, wg * 32), v);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; ++i) dh[i] = fmaf(gamC, dh[i], v[i]);
            }
        }
        // a wait has expired: keep step with the MMA warp, which comes to every one of them (odd counts: D is next)
        for (; pending > 0; --pending) nb_sync(pending & 1 ? kBarD : kBarH, nb);
        if (p.dh0 && !s_abort) {
#pragma unroll
            for (int i = 0; i < 32; ++i) p.dh0[at + (size_t)i * D] = dh[i];
        }
    } else if (warp == kMmaWarp) {
        // ---------------------------------- MMA-issue warp, converged ----------------------------------
        const uint32_t issue = elect_lane();
        grid_dep_wait();
        grid_dep_launch();
        const uint32_t sb = smem_u32(smem);
        // A1 = dO^T P (A, B MN-major: lines = token r), H-accumulator = dO^T Qg (B MN-major, two blocks of d_k)
        // stage of the ring of K and P, and the parity of its present round
        int s = 0;
        uint32_t sp = 0;
        auto ahead = [&](int it) {
            const int t = it & 1;
            const uint32_t sq = sb + kOffQ + t * bytesQ;
            wait(&bar.k[s], sp);
            wait(&bar.q[t], (it >> 1) & 1);
            tc_fence_after();
            umma_product_w<true, true>(tA1, sq + 16384, 8192, sb + s * kBytesK + 16384, 8192, C, C, false, issue);
            umma_product_w<true, true>(tH0 + 128 * (it & 1), sq + 16384, 8192, sq, 8192, D, C, false, issue);
            umma_commit_w(&bar.fq[t], issue);
        };
        ahead(0);
        for (int it = 0; it < p.N; ++it) {
            nb_sync(kBarH, nb);                         // dh^T operand (exit state of this chunk) is in place
            tc_fence_after();
            // A2 = dh^T K^T (B K-major)
            umma_product_ts_w<false>(tA2, aH, sb + s * kBytesK, 8192, C, D, false, issue);
            umma_commit_w(&bar.a, issue);
            umma_commit_w(&bar.fk[s], issue);
            const int t = it & 1;
            wait(&bar.w[t], (it >> 1) & 1);
            nb_sync(kBarD, nb);                         // -dDelta^T operand is in place, A1 has been read
            tc_fence_after();
            // H-accumulator -= dDelta^T W<-   (B K-major: lines = d_k index, contraction over tokens)
            umma_product_ts_w<false>(tH0 + 128 * (it & 1), aD, sb + offW + t * 16384, 16384, D, C, true, issue);
            umma_commit_w(&bar.b, issue);
            umma_commit_w(&bar.fw[t], issue);
            if (++s == kDeepK) { s = 0; sp ^= 1; }
            if (it + 1 < p.N) ahead(it + 1);            // in the shadow of the dh update
        }
        umma_commit_w(&bar.end, issue);                 // leaves when its products have come to their end, whatever has expired
        mbar_drain(&bar.end, 0);
    } else if (warp == kMmaWarp + 1) {
        // ---------------------------------- saving warp ----------------------------------
        if ((tid & 31) == 0) {
            grid_dep_wait();
            if (blockIdx.x == 0 && p.next) p.next[0] = p.next[1] = p.next[2] = 0;
            for (int it = 0; it < p.N; ++it) {
                const int y = (int)((tile0 + (p.N - 1 - it)) * D) + v0, sb = it & two;
                unsigned char *sdH = stg + sb * bytesS, *sdD = sdH + rows * 256;
                wait(&bar.ht[sb], (it >> two) & 1);       // gradient w.r.t. the exit state (rows = d_v, columns = d_k) is staged
                tma_store_2d(&mapdHs, sdH, 0, y);
                tma_store_2d(&mapdHs, sdH + rows * 128, 64, y);
                tma_store_commit();
                if (!two && it > 0) { tma_store_wait_read_n<1>(); mbar_arrive(&bar.df); }        // dDelta^T of the chunk before has been read
                wait(&bar.dt[sb], (it >> two) & 1);       // dDelta^T is staged
                tma_store_2d(&mapdDt, sdD, 0, y);
                tma_store_commit();
                if (!two) {
                    tma_store_wait_read_n<1>();
                    mbar_arrive(&bar.hf[0]);              // the dh^T tile has been read
                } else if (it > 0) {
                    tma_store_wait_read_n<2>();
                    mbar_arrive(&bar.hf[sb ^ 1]);         // both tiles of the chunk before have been read
                }
            }
            tma_store_wait_all();
        }
    } else {
        // ---------------------------------- TMA load warp ----------------------------------
        const bool lead = (tid & 31) == 0;
        grid_dep_wait();
        grid_dep_launch();
        // iteration `it` processes chunk n = N-1-it
        TokenScales ts(p.g, p.rk, row0, tid & 31);
        auto load_k = [&](int it, int s) {               // by the whole warp
            ts.put(sG[it & 3]);
            __syncwarp();
            if (lead) {
                const int n = p.N - 1 - it;
                unsigned char* st = smem + s * kBytesK;
                mbar_expect_tx(&bar.k[s], kBytesK);
                tma_load_3d(st, &mapK, hh * D, tok0 + n * C, b, &bar.k[s]);
                tma_load_3d(st + 8192, &mapK, hh * D + 64, tok0 + n * C, b, &bar.k[s]);
                tma_load_2d(st + 16384, &mapP, 0, (int)(row0 + (size_t)n * C), &bar.k[s]);
            }
            if (it + 1 < p.N) ts.fetch(p.N - 2 - it);
        };
        auto load_q = [&](int it) {                      // by the leading lane
            const int n = p.N - 1 - it;
            unsigned char* st = smem + kOffQ + (it & 1) * bytesQ;
            uint64_t* br = &bar.q[it & 1];
            const int yt = (int)(row0 + (size_t)n * C);
            mbar_expect_tx(br, bytesQ);
            tma_load_3d(st + 16384, &mapdO, hh * D + v0, tok0 + n * C, b, br);             // rows past the end of the sequence: zeros
            if (rows == D) tma_load_3d(st + 16384 + 8192, &mapdO, hh * D + 64, tok0 + n * C, b, br);
            tma_load_2d(st, &mapQg, 0, yt, br);
            tma_load_2d(st + 8192, &mapQg, 64, yt, br);
        };
        auto load_w = [&](int it) {
            mbar_expect_tx(&bar.w[it & 1], 16384);
            tma_load_2d(smem + offW + (it & 1) * 16384, &mapWt, 0, (int)((tile0 + (p.N - 1 - it)) * D), &bar.w[it & 1]);
        };
        ts.fetch(p.N - 1);
        for (int it = 0; it < kDeepK && it < p.N; ++it) {
            load_k(it, it);
            if (lead && it < 2) { load_q(it); load_w(it); }
        }
        int s = 0;                                        // stage of chunk it's K and P, and the parity of its present round
        uint32_t sp = 0;
        int nk = min(kDeepK, p.N), nq = min(2, p.N), nw = nq;
        for (int it = 0; it < p.N; ++it) {
            bool more = it + kDeepK < p.N;
            if (lead) {
                wait(&bar.fq[it & 1], (it >> 1) & 1);
                if (it + 2 < p.N && !s_abort) { load_q(it + 2); nq = it + 3; }
                wait(&bar.fk[s], sp);
            }
            more = __shfl_sync(0xffffffffu, more && !s_abort, 0);     // one answer for the warp
            if (more) { load_k(it + kDeepK, s); nk = it + kDeepK + 1; }
            if (lead) {
                wait(&bar.fw[it & 1], (it >> 1) & 1);
                if (it + 2 < p.N && !s_abort) { load_w(it + 2); nw = it + 3; }
            }
            __syncwarp();
            if (++s == kDeepK) { s = 0; sp ^= 1; }
        }
        // unless a wait has expired the products have been waited for, and so have the loads
        if (lead && s_abort) { mbar_drain_ring(bar.k, kDeepK, nk); mbar_drain_ring(bar.q, 2, nq); mbar_drain_ring(bar.w, 2, nw); }
    }
    tc_fence_before();
    __syncthreads();
    if (tid < 32) tmem_dealloc(tbase, 512);
}

// =================================================================================================
struct ChunkBwdMaps { CUtensorMap Q, K, V, dO, Mt, P, Dt, dDt, Hs, dHs, dQ, dK, dV; };
struct ChunkBwdParams {
    int logits;                // beta, alpha, lambda are logits of sigmoid gates; their gradients are taken w.r.t. the logits
    const float* rqk;          // QD_NORM_QK: 1/|q_t| per workspace row, then (BH*Tp further) 1/|k_t|
    int group;                 // sequences per group of work items
    int T, Tp, H, N, Ns, BH, total;   // T tokens per sequence, of which the N chunks from n0 on; Tp = 64 Ns rows per sequence in the workspace; total = BH*N
    int n0;
    int beside;                // 1: runs beside the reverse chain launched before it (tc_bwd), so it waits for that at its end
    const bf16 *beta, *alpha, *lam;
    const float* g;
    float *dbeta, *dalpha, *dlam;
    unsigned* status;
    unsigned* next;            // work items taken beyond the first of every CTA; zero when the kernel begins
};

// =================================================================================================
// shared-memory map of a chunk's tiles (bytes from the 1024-aligned base)
constexpr int oQ = 0, oK = 16384, oV = 32768, odO = 49152, oX = 65536, oMt = 81920, oP = 90112, oDt = 98304,
              odDt = 114688, oH = 131072, odH = 163840;                            // TMA-loaded tiles (X is built)
constexpr int kBwdEarlyBytes = 3 * 16384 + 2 * 8192;
// tiles built later reuse regions whose contents are dead by then
constexpr int odPG = oV, odTb = oV + 8192, odW = 196608, oN = oDt, odXK = oDt + 8192, oStDv = odDt, oStDk = oX, oStDq = odW;
constexpr int kTileBytes = 196608 + 16384;     // with the dW<-^T tile, written while dO is still an operand
constexpr int kNWG = 4;                       // warpgroups; each owns 64/kNWG columns of every 64-column accumulator
constexpr int kCW = C / kNWG, kG8 = kCW / 8;    // columns per warpgroup, groups of 8 columns
constexpr int kBwdCompute = 128 * kNWG;                 // epilogue threads
// + a warp that issues every MMA, a warp that issues every TMA copy, and two whose threads own a token each: coefficients
// and the sums over rows and columns that become d beta, d lambda and d alpha
constexpr int kBwdTail = kBwdCompute + 64, kBwdThreads = kBwdTail + C;
constexpr int kBwdNb = kBwdCompute + 32;                 // participants of a named barrier: the epilogue threads and a waiting warp
// named barriers: 1 = the epilogue threads among themselves; the others are raised by the
// epilogue threads (bar.arrive) when a tile is complete and awaited by the MMA warp or the TMA warp (bar.sync); Sum: row
// and column sums complete, awaited by the token threads; Tok: among themselves; End: everybody, the
// TMA warp only arrives
constexpr int kNbC = 1, kNbX = 2, kNbDW = 3, kNbDTb = 4, kNbN = 5, kNbDXK = 6, kNbOut = 7, kNbDV = 8, kNbDVt = 10, kNbSum = 11, kNbTok = 12, kNbEnd = 13;
constexpr int kNbSumN = kBwdCompute + C;

struct ChunkBars { uint64_t load, d, h, qk, st, a, b, c, m2, m3, m4, m5, end; };
// What the warps tell each other; `_` arrays by parity of the chunk, so that the token threads can publish a chunk
// ahead and take their sums a chunk late.
struct ChunkShared {
    float4 scf_[2][C];     // per token: {gamma beta, gamma_C / gamma, gamma, lambda}, one load in the last epilogue
    float sbeta_[2][C], sg_[2][C], slam_[2][C], sgam_[2][C];
    float2 srn_[2][C];     // NORM: {1/|k_t|, 1/|q_t|}
    float sred_[2][2][4][C];   // per-warp column sums: [0] rowsum(dQ1 o Q) - <(K-> dh)_r, Delta_r>, [1] d lambda
    float swk_[2][kBwdCompute / 32];        // per-warp sums of <(K-> dh)_r, Delta_r>
    float scol[2][4][C];   // column sums of dP o P, dA o A by quarters of the rows
    float srow[4][kNWG][C];   // per-row partial sums over each warpgroup's columns: rPP, d beta, t2, rAA
    float swp[kBwdCompute / 32], stot[2];
    int2 item[4];          // {chunk, sequence} of iterations it .. it + 2, by it mod 4; chunk < 0: no more
};
constexpr int kBwdSmem = kTileBytes + (int)sizeof(ChunkShared) + 1024;

// Four epilogue warpgroups: warpgroup w (threads 128w..128w+127) owns TMEM columns [16w, 16w+16) of every 64-column
// accumulator; inside a warpgroup, warp wq owns TMEM lanes [32 wq, 32 wq + 32), i.e. rows 32 wq .. of a 128-row product and
// rows 16 wq .. of a 64-row one.
// HAS_LAM = false: lambda is absent and d lambda is not asked for (the gated delta rule, Eq. 3): X = K, nothing is built,
// no column sum for d lambda.  HAS_ALPHA = false: alpha is absent and d alpha is not asked for (no forget gate; with
// HAS_LAM = false too this is DeltaNet, Eq. 2): every decay factor is 1 and none of the sums that only feed d alpha is
// taken.  The <true, true> instances serve every other case (an absent input then reads as lambda = 0, alpha = 1).
// NORM (QD_NORM_QK): the Q and K tiles arrive un-normalised and are normalised in place with the factors the forward
// left in the workspace; dq and dk are taken through the normalisation, dx = r (dx^ - x^ <x^, dx^>), which needs the
// row sums <x^, dx^>: dk^ and dq^ are staged in bf16 like dk and dq without NORM, and a second pass over the staged tiles, a
// row to 16 lanes, takes the sums and rewrites them.
// Work items: a chunk of a sequence.  They come in groups of p.group sequences, inside a group chunk by chunk from the first on
// (which the reverse chain has left last, so its tiles are still in L2), the sequences of a chunk index next to each other.  Every
// CTA takes the next one from a counter, two chunks ahead of its work.  Backward of 128 sequences of 32 chunks: 255 us; every
// gridDim.x-th item to a CTA 264 - 270; from the last chunk on 258; groups of 32 sequences 263, all at a time 259.  Training passes
// against items in sequence order with every gridDim.x-th to a CTA (and the reverse chain of then): 531 -> 514, one long
// group of 32 sequences of 512 chunks 2549 -> 2464.
template <bool HAS_LAM, bool HAS_ALPHA, bool NORM>
__global__ void __launch_bounds__(kBwdThreads) k_tc_chunk_bwd(const __grid_constant__ ChunkBwdMaps m, ChunkBwdParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ ChunkBars bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort, s_latch[2];                  // s_latch[it % 2]: a wait had expired before iteration it
    ChunkShared& sh = *reinterpret_cast<ChunkShared*>(sm + kTileBytes);
    auto &sbeta_ = sh.sbeta_, &sg_ = sh.sg_, &slam_ = sh.slam_, &sgam_ = sh.sgam_;
    auto& scf_ = sh.scf_;
    auto& srn_ = sh.srn_;
    auto& sred_ = sh.sred_;
    auto& swk_ = sh.swk_;
    auto& scol = sh.scol;
    auto& srow = sh.srow;
    auto& swp = sh.swp;
    auto& stot = sh.stot;
    volatile int2* const item = sh.item;
    const int tid = threadIdx.x, wg = tid >> 7, l = tid & 127, lane = tid & 31, wq = (tid >> 5) & 3;
    const int c0 = wg * kCW;                                      // my columns of a 64-column accumulator

    if (tid == 0) {
        uint64_t* all = &bar.load;
        for (int i = 0; i < (int)(sizeof(ChunkBars) / 8); ++i) mbar_init(all + i, 1);
        mbar_init_fence();
        s_abort = 0;
        s_latch[0] = s_latch[1] = 0;
    }
    if (tid < 32) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = tmem_slot;
    const uint32_t T0 = tb, T1 = tb + 64, T2 = tb + 128, T3 = tb + 192, T4 = tb + 256, T5 = tb + 320, T6 = tb + 384,
                   T7 = tb + 448;
    const uint32_t lane_base = (uint32_t)wq * 32;
    auto my = [&](uint32_t t) { return tmem_addr(t, lane_base, (uint32_t)c0); };

    // The tiles of a chunk arrive in three groups, as their regions fall free in the chunk before: V, dO, M^T, P, Delta^T,
    // dDelta^T after its last products; h^T, dh^T in the middle; Q, K, which the last epilogue
    // reads, at its end.  The first products need only the first two.
    struct Item { int n, bh; };                                  // chunk n of sequence bh; n < 0: none
    auto slot = [&](int it) { return Item{item[it & 3].x, item[it & 3].y}; };
    auto nth = [&](int i) {
        if (i >= p.total) return Item{-1, 0};
        const int per = p.group * p.N, grp = i / per, r = i - grp * per;
        const int g0 = grp * p.group, gs = min(p.group, p.BH - g0);       // the last group may be smaller
        return Item{p.n0 + r / gs, g0 + r % gs};
    };
    auto claim = [&]() { return nth((int)gridDim.x + (int)atomicAdd(p.next, 1u)); };      // a CTA's first item goes by its number
    auto put = [&](int it, Item x) { item[it & 3].x = x.n; item[it & 3].y = x.bh; };
    auto issue_dd = [&](Item x) {                 // dDelta^T on its own: the first product waits for it
        mbar_expect_tx(&bar.d, 16384);
        tma_load_2d(sm + odDt, &m.dDt, 0, (int)(((size_t)x.bh * p.Ns + x.n) * D), &bar.d);
    };
    auto issue_early = [&](Item x) {
        const int b_ = x.bh / p.H, hh_ = x.bh % p.H;
        const int yt = (int)((size_t)x.bh * p.Tp + (size_t)x.n * C);
        const int yc = (int)(((size_t)x.bh * p.Ns + x.n) * D);
        mbar_expect_tx(&bar.load, kBwdEarlyBytes);
        tma_load_2d(sm + oMt, &m.Mt, 0, yt, &bar.load);
        for (int blk = 0; blk < 2; ++blk)         // token rows past the end of the sequence arrive as zeros
            tma_load_3d(sm + oV + blk * 8192, &m.V, hh_ * D + blk * 64, x.n * C, b_, &bar.load);
        tma_load_2d(sm + oDt, &m.Dt, 0, yc, &bar.load);
        for (int blk = 0; blk < 2; ++blk)
            tma_load_3d(sm + odO + blk * 8192, &m.dO, hh_ * D + blk * 64, x.n * C, b_, &bar.load);
        tma_load_2d(sm + oP, &m.P, 0, yt, &bar.load);
    };
    auto issue_h = [&](Item x) {                  // half of bar.h
        const int yc = (int)(((size_t)x.bh * p.Ns + x.n) * D);
        mbar_expect_tx(&bar.h, 2 * 32768);
        for (int blk = 0; blk < 2; ++blk) tma_load_2d(sm + oH + blk * 16384, &m.Hs, blk * 64, yc, &bar.h);
    };
    auto issue_dh = [&](Item x) {                 // the other half
        const int yc = (int)(((size_t)x.bh * p.Ns + x.n) * D);
        for (int blk = 0; blk < 2; ++blk) tma_load_2d(sm + odH + blk * 16384, &m.dHs, blk * 64, yc, &bar.h);
    };
    auto issue_qk = [&](Item x) {
        const int b_ = x.bh / p.H, hh_ = x.bh % p.H;
        mbar_expect_tx(&bar.qk, 2 * 16384);
        for (int blk = 0; blk < 2; ++blk) {
            tma_load_3d(sm + oQ + blk * 8192, &m.Q, hh_ * D + blk * 64, x.n * C, b_, &bar.qk);
            tma_load_3d(sm + oK + blk * 8192, &m.K, hh_ * D + blk * 64, x.n * C, b_, &bar.qk);
        }
    };
    // of the tiles of a chunk, those that are waited for most into L2 only, a chunk time ahead
    auto prefetch_late = [&](Item x) {
        const int b_ = x.bh / p.H, hh_ = x.bh % p.H;
        const int yc = (int)(((size_t)x.bh * p.Ns + x.n) * D);
        for (int blk = 0; blk < 2; ++blk) {
            tma_prefetch_3d(&m.Q, hh_ * D + blk * 64, x.n * C, b_);
            tma_prefetch_3d(&m.K, hh_ * D + blk * 64, x.n * C, b_);
            tma_prefetch_2d(&m.Hs, blk * 64, yc);
            tma_prefetch_2d(&m.dHs, blk * 64, yc);
        }
        tma_prefetch_2d(&m.Dt, 0, yc);
        tma_prefetch_2d(&m.dDt, 0, yc);
    };
    // bounded wait; once any wait has expired every later wait returns at once and the kernel drains: all
    // threads still pass every barrier, results are garbage, the status word says so
    auto wait = [&](uint64_t* bar, uint32_t parity) {
        if (mbar_try_wait(bar, parity) || s_abort) return;
        if (!mbar_wait(bar, parity)) { s_abort = 1; *p.status = QD_ERR_TIMEOUT; }
    };
    const uint32_t aQ = smem_u32(sm + oQ), aK = smem_u32(sm + oK), aV = smem_u32(sm + oV), adO = smem_u32(sm + odO),
                   aX = smem_u32(sm + oX), aMt = smem_u32(sm + oMt), aDt = smem_u32(sm + oDt),
                   adDt = smem_u32(sm + odDt), aH = smem_u32(sm + oH), adH = smem_u32(sm + odH);
    const uint32_t adPG = smem_u32(sm + odPG), adTb = smem_u32(sm + odTb), adW = smem_u32(sm + odW),
                   aN = smem_u32(sm + oN), adXK = smem_u32(sm + odXK);
    constexpr bool has_lam = HAS_LAM, has_alpha = HAS_ALPHA, want_dl = HAS_LAM, want_da = HAS_ALPHA;
    const uint32_t aXe = has_lam ? aX : aK;

    if (tid >= kBwdCompute && tid < kBwdNb) {
        // =============================== MMA warp ===============================
        // Nothing here is done by one lane alone but the issue itself, so that descriptors and their increments stay in
        // uniform registers (see umma_product_w); copies have a warp of their own.
        const uint32_t issue = elect_lane();
        const uint32_t tbu = uniform(tb);
        const uint32_t T0 = tbu, T1 = tbu + 64, T2 = tbu + 128, T3 = tbu + 192, T4 = tbu + 256, T5 = tbu + 320, T6 = tbu + 384, T7 = tbu + 448;
        __syncthreads();                                                 // the first item is known
        if (!p.beside) grid_dep_wait();
        __syncthreads();                                                 // the first chunk's coefficients have been published
        for (int it = 0; (int)uniform((uint32_t)slot(it).n) >= 0; ++it) {
            const uint32_t ph = it & 1;
            if (__any_sync(0xffffffffu, s_latch[ph])) break;
            wait(&bar.d, ph);
            wait(&bar.h, ph);
            __syncwarp();
            tc_fence_after();
            umma_product_w<true, true>(T3, aH, 16384, adDt, 8192, C, D, false, issue, true);     // -h dDelta^T      [i][r] = dW<-^T
            umma_commit_w(&bar.a, issue);
            wait(&bar.load, ph);
            umma_product_w<false, false>(T6, adDt, 16384, aMt, 8192, C, C, false, issue);        // dDelta^T M       [j][s]
            umma_product_w<false, true, 64>(T2, aV, 8192, adDt, 8192, C, D, false, issue);       // V dDelta^T       [s][r]
            umma_commit_w(&bar.b, issue);                // from here on no product reads V or dDelta^T any more
            umma_product_w<false, true, 64>(T1, adO, 8192, aDt, 8192, C, D, false, issue);       // dO Delta^T       [r][s]
            umma_commit_w(&bar.c, issue);
            umma_product_w<true, false>(T4, aH, 16384, adO, 8192, C, D, false, issue);           // h dO^T           [i][r]
            wait(&bar.qk, ph);
            nb_sync(kNbDW, kBwdNb);                                      // the dW<-^T tile is complete
            nb_sync(kNbX, kBwdNb);                                       // X has been built
            tc_fence_after();
            // the product that the dependent chain waits for goes first, those that are needed late after it
            umma_product_w<false, true, 64>(T3, aXe, 8192, adW, 8192, C, D, false, issue);       // X dW<-^T         [s][r]
            umma_commit_w(&bar.m2, issue);
            umma_product_w<false, false, 64>(T0, aXe, 8192, aK, 8192, C, D, false, issue);       // X K^T            [r][i]
            umma_product_w<true, true>(T5, adH, 16384, aDt, 8192, C, D, false, issue);           // dh Delta^T       [i][s]
            nb_sync(kNbDTb, kBwdNb);
            tc_fence_after();
            umma_product_w<true, true, 64>(T3, adTb, 8192, aMt, 8192, C, C, false, issue);       // N~ = dT diag(beta) M^T   [r][u]
            umma_commit_w(&bar.m3, issue);                // from here on nobody reads h, dh or Delta^T
            nb_sync(kNbN, kBwdNb);                                       // N~ is a tile, and so is dP o Gamma
            tc_fence_after();
            umma_product_w<false, true, 64>(T2, aMt, 8192, aN, 8192, C, C, false, issue, true);  // dA = -M^T N~     [r][s]
            umma_commit_w(&bar.m4, issue);
            umma_product_w<true, true>(T1, aQ, 8192, adPG, 8192, C, C, false, issue);            // (dPG^T Q)^T      [i][s]
            umma_product_w<true, false>(T3, aK, 8192, adPG, 8192, C, C, false, issue);           // (dPG K)^T        [i][r]
            nb_sync(kNbDV, kBwdNb);                                      // T6 has been read
            tc_fence_after();
            umma_product_w<false, false>(T6, adW, 16384, aMt, 8192, C, C, false, issue);         // dW<-^T M         [i][s]
            nb_sync(kNbDXK, kBwdNb);
            tc_fence_after();
            umma_product_w<true, false>(T7, aK, 8192, adXK, 8192, C, C, false, issue);           // (dXK K)^T        [i][r]
            umma_product_w<true, true>(T1, aXe, 8192, adXK, 8192, C, C, true, issue);            // + (dXK^T X)^T    [i][s]
            umma_commit_w(&bar.m5, issue);
            nb_sync(kNbEnd, kBwdThreads);                                // every read of this chunk's tiles and accumulators is done
        }
        umma_commit_w(&bar.end, issue);                                  // leaves when its products have come to their end, whatever has expired
        mbar_drain(&bar.end, 0);
    } else if (tid >= kBwdNb && tid < kBwdTail) {
        // =============================== TMA warp ===============================
        const bool lead = lane == 0;
        if (lead) put(0, nth((int)blockIdx.x));
        __syncthreads();                                                 // the first item is known
        if (lead) {
            // first chunk: everything that the reverse chain (the kernel before this one) does not write is fetched
            // before waiting for it -- inputs, and tiles of kernels that had finished before the reverse chain began
            const Item x = slot(0);
            issue_qk(x);
            issue_early(x);
            issue_h(x);
            if (!p.beside) grid_dep_wait();
            issue_dh(x);
            issue_dd(x);
            put(1, claim());
            mbar_arrive(&bar.st);                                        // nothing is staged yet
        }
        __syncthreads();                                                 // the first chunk's coefficients have been published
        int ne = 1, nh = 1, nqk = 1;
        for (int it = 0; slot(it).n >= 0; ++it) {
            const Item cur = slot(it), next = slot(it + 1);
            const int n = cur.n, b = cur.bh / p.H, hh = cur.bh % p.H;
            const bool more = next.n >= 0;
            const uint32_t ph = it & 1;
            if (__any_sync(0xffffffffu, s_latch[ph])) break;
            if (lead) {
                if (more) prefetch_late(next);
                put(it + 2, more ? claim() : next);
                wait(&bar.m3, ph);                                       // from here on nobody reads h or dh
                if (more && !s_abort) { issue_h(next); issue_dh(next); ++nh; }
            }
            nb_sync(kNbDVt, kBwdNb);                                     // the dv staging tile is complete
            if (lead) {
                tma_store_3d(&m.dV, sm + oStDv, hh * D, n * C, b);          // rows past the end of the sequence are skipped
                tma_store_3d(&m.dV, sm + oStDv + 8192, hh * D + 64, n * C, b);
                tma_store_commit();
                tma_store_wait_read();
                wait(&bar.m5, ph);                                         // from here on nobody reads anything but Q, K
                fence_proxy_async();
                if (more && !s_abort) { issue_dd(next); issue_early(next); ++ne; }
            }
            nb_sync(kNbOut, kBwdNb);                                     // the dk and dq staging tiles are complete
            // Everybody has to leave in the same iteration.  This one's latch may not have been read by every warp yet: once a wait has
            // expired the epilogue comes here without the others.  The next one's was read before the End barrier that the epilogue has passed
            // since.  An expiry that this misses is seen one chunk later (waits return at once meanwhile).
            if (lead) s_latch[ph ^ 1] = s_abort;
            __syncwarp();
            nb_arrive(kNbEnd, kBwdThreads);                              // nobody waits for the copies to be issued
            if (lead) {
                tma_store_3d(&m.dK, sm + oStDk, hh * D, n * C, b);
                tma_store_3d(&m.dK, sm + oStDk + 8192, hh * D + 64, n * C, b);
                tma_store_3d(&m.dQ, sm + oStDq, hh * D, n * C, b);
                tma_store_3d(&m.dQ, sm + oStDq + 8192, hh * D + 64, n * C, b);
                tma_store_commit();
                fence_proxy_async();                                     // the epilogue's reads of Q precede the copy into its region
                if (more && !s_abort) { issue_qk(next); ++nqk; }
            }
            if (lead) {
                tma_store_wait_read();                                   // the staging tiles have been read by the stores
                mbar_arrive(&bar.st);
            }
            __syncwarp();
        }
        if (lead && s_abort) {        // otherwise the products have been waited for, and so have the loads
            mbar_drain_ring(&bar.load, 1, ne); mbar_drain_ring(&bar.d, 1, ne); mbar_drain_ring(&bar.h, 1, nh); mbar_drain_ring(&bar.qk, 1, nqk);
        }
        if (lead) tma_store_wait_all();
    } else if (tid >= kBwdTail) {
        // =============================== token threads ===============================
        // thread r owns token r of the chunk
        const int r = tid - kBwdTail;
        bf16 zb = __float2bfloat16_rn(0.f), zl = zb, za = zb;                // as stored, converted a chunk later: nothing waits for the loads
        float cg = 0.f, cgC = 0.f, rq = 1.f, rk = 1.f;
        bool tok = false;
        auto fetch = [&](Item x) {
            const int n_ = x.n, bh_ = x.bh;
            const int b_ = bh_ / p.H, hh_ = bh_ % p.H;
            tok = n_ * C + r < p.T;                               // tokens past the end of the sequence: beta = 0, alpha = 1
            const size_t cr = ((size_t)b_ * p.T + (size_t)n_ * C + r) * p.H + hh_, wr = (size_t)bh_ * p.Tp + (size_t)n_ * C;
            if (tok) {
                zb = p.beta[cr];
                if (p.lam) zl = p.lam[cr];
                if (p.alpha) za = p.alpha[cr];
            }
            cg = p.g[wr + r];
            cgC = p.g[wr + C - 1];
            if (NORM) { rq = p.rqk[wr + r]; rk = p.rqk[(size_t)p.BH * p.Tp + wr + r]; }
        };
        float be = 0.f, lm = 0.f, al = 1.f;
        auto publish = [&](int par) {
            be = tok ? gate(__bfloat162float(zb), p.logits) : 0.f;
            lm = (tok && p.lam) ? gate(__bfloat162float(zl), p.logits) : 0.f;
            al = (tok && p.alpha) ? gate(__bfloat162float(za), p.logits) : 1.f;
            const float gm = __expf(cg);
            sbeta_[par][r] = be; slam_[par][r] = lm; sg_[par][r] = cg; sgam_[par][r] = gm;
            scf_[par][r] = make_float4(gm * be, __expf(cgC - cg), gm, lm);
            if (NORM) srn_[par][r] = make_float2(rk, rq);
        };
        __syncthreads();                                                 // the first item is known
        if (slot(0).n >= 0) { fetch(slot(0)); publish(0); }
        if (!p.beside) grid_dep_wait();
        __syncthreads();
        // what the sums at the end of a chunk need of it, taken up a chunk later
        float dg_pre = 0.f, dhh = 0.f, be0 = 0.f, lm0 = 0.f, al0 = 1.f, gmC = 1.f;
        auto finish = [&](Item x, int par) {
            const int n = x.n, bh = x.bh;
            const size_t at = ((size_t)(bh / p.H) * p.T + (size_t)n * C + r) * p.H + bh % p.H;
            const bool in = n * C + r < p.T;
            float dg = dg_pre, dl = 0.f;
#pragma unroll
            for (int w4 = 0; w4 < 4; ++w4) {
                if (want_da) dg += sred_[par][0][w4][r];
                if (want_dl) dl += sred_[par][1][w4][r];
            }
            if (want_dl && in) p.dlam[at] = p.logits ? dl * lm0 * (1.f - lm0) : dl;
            if (want_da) {
                if (r == C - 1) {
                    float kds = 0.f;
#pragma unroll
                    for (int w = 0; w < kBwdCompute / 32; ++w) kds += swk_[par][w];
                    dg += gmC * dhh + kds;
                }
                // d log alpha_i = sum_{r >= i} dg_r (suffix sums over 64 tokens, two warps)
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float t = __shfl_down_sync(0xffffffffu, dg, o);
                    if (lane + o < 32) dg += t;
                }
                if (lane == 0) stot[r >> 5] = dg;
                nb_sync(kNbTok, C);
                if (r < 32) dg += stot[1];
                // d log alpha -> d alpha = d log alpha / alpha;  with logit inputs d/dz log sigmoid(z) = 1 - sigmoid(z)
                if (in && p.dalpha) p.dalpha[at] = p.logits ? dg * (1.f - al0) : dg / al0;
            }
        };
        Item prev{-1, 0};
        uint32_t last_ph = 0;
        for (int it = 0; slot(it).n >= 0; ++it) {
            const Item cur = slot(it), next = slot(it + 1);
            const int n = cur.n, bh = cur.bh;
            const uint32_t ph = it & 1;
            if (__any_sync(0xffffffffu, s_latch[ph])) { prev.n = -1; break; }
            if (prev.n >= 0) finish(prev, ph ^ 1);
            const float gm = sgam_[ph][C - 1];
            be0 = be; lm0 = lm; al0 = al; gmC = gm;
            if (next.n >= 0) fetch(next);
            nb_sync(kNbSum, kNbSumN);                                    // row sums and scratch are complete
            float rPP = 0.f, t2 = 0.f, rAA = 0.f, dbt = 0.f;
#pragma unroll
            for (int w4 = 0; w4 < kNWG; ++w4) {
                rPP += srow[0][w4][r]; dbt += srow[1][w4][r]; t2 += srow[2][w4][r]; rAA += srow[3][w4][r];
            }
            dg_pre = rPP + t2 + rAA;
            if (want_da) {
#pragma unroll
                for (int w4 = 0; w4 < 4; ++w4) dg_pre -= scol[0][w4][r] + scol[1][w4][r];
            }
            // with logit inputs: d/dz of sigmoid(z) is sigmoid(z) (1 - sigmoid(z))
            if (n * C + r < p.T) p.dbeta[((size_t)(bh / p.H) * p.T + (size_t)n * C + r) * p.H + bh % p.H] = p.logits ? dbt * be0 * (1.f - be0) : dbt;
            if (want_da) {
                dhh = 0.f;
#pragma unroll
                for (int w = 0; w < kBwdCompute / 32; ++w) dhh += swp[w];
            }
            if (next.n >= 0) publish(ph ^ 1);
            nb_sync(kNbEnd, kBwdThreads);                                // every read of this chunk's tiles and accumulators is done
            prev = cur;
            last_ph = ph;
        }
        if (prev.n >= 0) finish(prev, last_ph);
    } else {
    // ======================================== epilogue threads ========================================
    auto csync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(kNbC), "r"(kBwdCompute) : "memory"); };   // warps arrive converged
    // fragment layout (tmem_ld_frag): columns c0 + 8 g + ft + {0, 1} of 16-row halves hf; the matching rows of a token-major
    // tile, transposed: lane l addresses token c0 + 8 g + l % 8, rows 32 wq + 8 (l / 8) ..
    const int ft = 2 * (lane & 3);
    auto frag = [&](uint32_t t, int g, int hf) { return tmem_addr(t, lane_base + 16 * hf, (uint32_t)c0 + 8 * g); };
    uint32_t foff[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) foff[g] = (wq >> 1) * 8192 + sw128_chunk(c0 + 8 * g + (lane & 7), (wq & 1) * 4 + (lane >> 3));
    __syncthreads();                    // the first item is known
    if (!p.beside) grid_dep_wait();
    __syncthreads();                    // the first chunk's coefficients have been published

    for (int it = 0; slot(it).n >= 0; ++it) {
    const uint32_t ph = it & 1;
    if (s_latch[ph]) break;
    const float *sbeta = sbeta_[ph], *slam = slam_[ph], *sg = sg_[ph], *sgam = sgam_[ph];
    const float4* scf = scf_[ph];
    const float2* srn = srn_[ph];
    // ---- partial <dh,h>_F, under the first products ---------------------------------------------------
    wait(&bar.h, ph);
    float dhh_part = 0.f;
    if (want_da)
#pragma unroll
    for (int cc = 0; cc < 16 / kNWG; ++cc) {
        const int ci = wg * (16 / kNWG) + cc;                // chunk 0..15 of line l
        const uint32_t off = (ci >> 3) * 16384 + sw128_chunk(l, ci & 7);
        float a[8], c8[8];
        load8(sm + oH + off, a);
        load8(sm + odH + off, c8);
#pragma unroll
        for (int e = 0; e < 8; ++e) dhh_part = fmaf(a[e], c8[e], dhh_part);
    }
    if (want_da) {
        dhh_part += __shfl_xor_sync(0xffffffffu, dhh_part, 16);
        dhh_part += __shfl_xor_sync(0xffffffffu, dhh_part, 8);
        dhh_part += __shfl_xor_sync(0xffffffffu, dhh_part, 4);
        dhh_part += __shfl_xor_sync(0xffffffffu, dhh_part, 2);
        dhh_part += __shfl_xor_sync(0xffffffffu, dhh_part, 1);
        if (lane == 0) swp[tid >> 5] = dhh_part;
    }
    // ---- dW<-^T = -h dDelta^T: row i = l as an operand tile (region of its own: dO is still being read) -----
    wait(&bar.st, ph);                                    // the staged dk, dq of the chunk before lie over X and this tile
    wait(&bar.a, ph);
    tc_fence_after();
#pragma unroll
    for (int g8 = 0; g8 < kG8; ++g8) {
        float dw[8];
        tmem_ld8(my(T3) + g8 * 8, dw);
        tmem_ld_wait();
        sts128(sm + odW + sw128_chunk(l, wg * kG8 + g8), pack8(dw));
    }
    fence_proxy_async();
    tc_fence_before();
    nb_arrive(kNbDW, kBwdNb);
    wait(&bar.load, ph);
    wait(&bar.qk, ph);
    // ---- X = K + lambda Q (the products that do not read X are already running) ------------------------
    if (has_lam || NORM) {
        constexpr int kPer = 16 / (kBwdCompute / 64);     // 16-byte chunks of a row per thread
        const int r = tid & 63, part = tid >> 6;
        const float lm = slam[r];
        const float rq = NORM ? srn[r].y : 1.f, rk = NORM ? srn[r].x : 1.f;
#pragma unroll
        for (int cc = 0; cc < kPer; ++cc) {
            const int ci = part * kPer + cc;              // chunk 0..15 of the row: block ci>>3, chunk ci&7
            const uint32_t off = (ci >> 3) * 8192 + sw128_chunk(r, ci & 7);
            float qv[8], kv[8];
            load8(sm + oQ + off, qv);
            load8(sm + oK + off, kv);
            if (NORM) {                                   // q^ and k^ in place: no product has read Q or K yet
#pragma unroll
                for (int e = 0; e < 8; ++e) { qv[e] *= rq; kv[e] *= rk; }
                sts128(sm + oQ + off, pack8(qv));
                sts128(sm + oK + off, pack8(kv));
            }
            if (has_lam) {
#pragma unroll
                for (int e = 0; e < 8; ++e) kv[e] = fmaf(lm, qv[e], kv[e]);
                sts128(sm + oX + off, pack8(kv));
            }
        }
    }
    fence_proxy_async();
    nb_arrive(kNbX, kBwdNb);
    // The 64-row accumulators: this thread's rows are rw + 8 j + lane / 4, j = 0, 1, its columns c0 + 8 g + ft + {0, 1}.  Of a
    // sum over columns, the lane ends up with that of row `mine`, of a sum over the warp's 16 rows with that of column `ours`.
    const int rw = 16 * wq, mine = rw + 4 * (lane & 2) + (lane >> 2), ours = c0 + ((lane & 16) ? 8 : 0) + ft + ((lane & 8) ? 1 : 0);
    const bool my_row = !(lane & 1), our_col = !(lane & 4);
    auto row_sum = [&](float* v) { fold<2>(v, lane, 2); return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1); };
    auto col_sum = [&](float* v) { fold<4>(v, lane, 16); fold<2>(v, lane, 8); return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 4); };
    const int r0 = rw + (lane >> 2);                       // rows r0, r0 + 8
    // of a [64 rows][64] tile: matrix m = 2 g + j, rows rw + 8 j .., columns c0 + 8 g ..
    const uint32_t at = sw128_chunk(rw + (lane & 15), wg * 2 + (lane >> 4));
    const float gr[2] = {sg[r0], sg[r0 + 8]};
    float gm[8];                                           // Gamma_rs, s <= r
    {
        float gs[4];
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const float2 t = *reinterpret_cast<const float2*>(sg + c0 + 8 * g + ft);
            gs[2 * g] = t.x; gs[2 * g + 1] = t.y;
        }
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const int s = c0 + 8 * (x >> 2) + ft + (x & 1), r = r0 + 8 * ((x >> 1) & 1);
            gm[x] = s <= r ? (has_alpha ? __expf(gr[(x >> 1) & 1] - gs[2 * (x >> 2) + (x & 1)]) : 1.f) : 0.f;
        }
    }
    // ---- dT^T row s, columns r;  M[r][s] = line s of Mt ------------------------------------------------
    wait(&bar.b, ph);
    wait(&bar.m2, ph);
    tc_fence_after();
    {
        float a[8], bq[8], db[2] = {}, mb[2] = {};
        uint32_t mr[4], o[4];
        tmem_ld_frag2(frag(T2, 0, 0), a);
        tmem_ld_frag2(frag(T3, 0, 0), bq);
        ldsm4<false>(sm + oMt + at, mr);
        const float gs[2] = {sgam[r0], sgam[r0 + 8]}, bs[2] = {sbeta[r0], sbeta[r0 + 8]};
        tmem_ld_wait();
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = m & 1;
            float tb8[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int x = 4 * (m >> 1) + 2 * j + e;
                const float mv = __uint_as_float(e ? mr[m] & 0xffff0000u : mr[m] << 16), dt = fmaf(gs[j], bq[x], a[x]);
                db[j] = fmaf(dt, mv, db[j]);
                mb[j] = fmaf(mv, bq[x], mb[j]);
                tb8[e] = bs[j] * dt;
            }
            o[m] = pack_bf16(tb8[0], tb8[1]);
        }
        stsm4<false>(sm + odTb + at, o);
        fence_proxy_async();
        tc_fence_before();
        nb_arrive(kNbDTb, kBwdNb);
        const float d = row_sum(db), t2 = sgam[mine] * sbeta[mine] * row_sum(mb);
        if (my_row) { srow[1][wg][mine] = d; srow[2][wg][mine] = t2; }
    }
    // ---- dP, under N~: causal mask, dP o P (row and column sums), dP o Gamma as an operand tile ----------
    wait(&bar.c, ph);
    tc_fence_after();
    {
        float v[8], rPP[2] = {}, cP[4] = {};
        uint32_t pr[4], o[4];
        tmem_ld_frag2(frag(T1, 0, 0), v);
        ldsm4<false>(sm + oP + at, pr);                    // causal: zero above the diagonal
        tmem_ld_wait();
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = m & 1;
            float pg[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int x = 4 * (m >> 1) + 2 * j + e;
                const float pp = v[x] * __uint_as_float(e ? pr[m] & 0xffff0000u : pr[m] << 16);
                rPP[j] += pp;
                cP[2 * (m >> 1) + e] += pp;
                pg[e] = gm[x] * v[x];
            }
            o[m] = pack_bf16(pg[0], pg[1]);
        }
        stsm4<false>(sm + odPG + at, o);
        const float d = row_sum(rPP);
        if (my_row) srow[0][wg][mine] = d;
        if (want_da) {
            const float x = col_sum(cP);
            if (our_col) scol[0][wq][ours] = x;
        }
    }
    // ---- N~ = dT diag(beta) M^T, copied out as an operand tile --------------------------------------
    wait(&bar.m3, ph);
    tc_fence_after();
    {
        float v[8];
        uint32_t o[4];
        tmem_ld_frag2(frag(T3, 0, 0), v);
        tmem_ld_wait();
#pragma unroll
        for (int m = 0; m < 4; ++m) o[m] = pack_bf16(v[4 * (m >> 1) + 2 * (m & 1)], v[4 * (m >> 1) + 2 * (m & 1) + 1]);
        stsm4<false>(sm + oN + at, o);
    }
    fence_proxy_async();
    tc_fence_before();
    nb_arrive(kNbN, kBwdNb);
    // ---- dV, under dA ---------------------------------------------------------------------------------
    {
        // dV^T [j][s], scaled by beta_s, transposed into the staging tile
        float dvv[2][2][4];                               // [8 columns][16 rows]
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) tmem_ld_frag(frag(T6, g, hf), dvv[g][hf]);
        tmem_ld_wait();
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const float2 be = *reinterpret_cast<const float2*>(sbeta + c0 + 8 * g + ft);
            uint32_t r[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) r[m] = pack_bf16(be.x * dvv[g][m >> 1][2 * (m & 1)], be.y * dvv[g][m >> 1][2 * (m & 1) + 1]);
            stsm4<true>(sm + oStDv + foff[g], r);
        }
    }
    fence_proxy_async();
    tc_fence_before();
    nb_arrive(kNbDV, kBwdNb);
    nb_arrive(kNbDVt, kBwdNb);
    // ---- dA = -M^T N~ -----------------------------------------------------------------------------
    wait(&bar.m4, ph);
    tc_fence_after();
    {
        float da[8], xk[8], dbr[2] = {}, cA[4] = {};
        uint32_t o[4];
        tmem_ld_frag2(frag(T2, 0, 0), da);
        tmem_ld_frag2(frag(T0, 0, 0), xk);
        const float br[2] = {sbeta[r0], sbeta[r0 + 8]};
        tmem_ld_wait();
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = m & 1;
            float out[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int x = 4 * (m >> 1) + 2 * j + e;
                const float d = c0 + 8 * (m >> 1) + ft + e < r0 + 8 * j ? da[x] * gm[x] : 0.f, dgx = d * xk[x];
                dbr[j] += dgx;
                cA[2 * (m >> 1) + e] = fmaf(br[j], dgx, cA[2 * (m >> 1) + e]);
                out[e] = br[j] * d;                        // dXK
            }
            o[m] = pack_bf16(out[0], out[1]);
        }
        stsm4<false>(sm + odXK + at, o);
        fence_proxy_async();
        tc_fence_before();
        nb_arrive(kNbDXK, kBwdNb);
        const float d = row_sum(dbr);
        if (my_row) { srow[1][wg][mine] += d; srow[3][wg][mine] = sbeta[mine] * d; }
        if (want_da) {
            const float x = col_sum(cA);
            if (our_col) scol[1][wq][ours] = x;
        }
    }
    nb_arrive(kNbSum, kNbSumN);
    wait(&bar.m5, ph);
    tc_fence_after();
    // The last epilogue: dk and dq, transposed, into their staging tiles, and the column sums (over the d_k index i, i.e.
    // down the fragments and across eight lanes) that d lambda and the decay gradient need.
    {
        float ksum = 0.f, t1[4], dl[4];                   // [2 (8 columns) + column of the pair]
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const int t = c0 + 8 * g + ft;
            float dx[2][4], v[2][4], w[2][4], u[2][4], z[2][4], y[2][4];
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                tmem_ld_frag(frag(T6, g, hf), dx[hf]); tmem_ld_frag(frag(T7, g, hf), v[hf]); tmem_ld_frag(frag(T1, g, hf), w[hf]);
                tmem_ld_frag(frag(T5, g, hf), u[hf]); tmem_ld_frag(frag(T4, g, hf), z[hf]); tmem_ld_frag(frag(T3, g, hf), y[hf]);
            }
            uint32_t qr[4], kr[4], dkr[4], dqr[4];
            ldsm4<true>(sm + oQ + foff[g], qr);
            ldsm4<true>(sm + oK + foff[g], kr);
            const float4 cf[2] = {scf[t], scf[t + 1]};
            tmem_ld_wait();
            float s0[2] = {}, s1[2] = {}, s2[2] = {};      // sums of U k, Z q, dX q
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                float dkv[2], dqv[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int hf = m >> 1, x = 2 * (m & 1) + e;
                    const float qv = __uint_as_float(e ? qr[m] & 0xffff0000u : qr[m] << 16), kv = __uint_as_float(e ? kr[m] & 0xffff0000u : kr[m] << 16);
                    const float dxe = fmaf(cf[e].x, dx[hf][x], v[hf][x]);                       // dX^T[i][t]
                    dkv[e] = fmaf(cf[e].y, u[hf][x], w[hf][x] + dxe);                           // d k  (d k^ with NORM)
                    dqv[e] = fmaf(cf[e].w, dxe, fmaf(cf[e].z, z[hf][x], y[hf][x]));             // d q  (d q^ with NORM)
                    s0[e] = fmaf(u[hf][x], kv, s0[e]);
                    s1[e] = fmaf(z[hf][x], qv, s1[e]);
                    s2[e] = fmaf(dxe, qv, s2[e]);
                }
                dkr[m] = pack_bf16(dkv[0], dkv[1]);
                dqr[m] = pack_bf16(dqv[0], dqv[1]);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                // <(K-> dh)_t, Delta_t> = gamma_C/gamma_t sum_i K[t][i] (dh Delta^T)[i][t], all of it in fp32
                const float kd = cf[e].y * s0[e];
                ksum += kd;
                t1[2 * g + e] = fmaf(cf[e].z, s1[e], -kd);
                dl[2 * g + e] = s2[e];
            }
            stsm4<true>(sm + oStDk + foff[g], dkr);
            stsm4<true>(sm + oStDq + foff[g], dqr);
        }
        // lane: column 8 (bit 4) + 2 (lane % 4) + (bit 3)
        const int col = c0 + ((lane & 16) ? 8 : 0) + ft + ((lane & 8) ? 1 : 0);
        if (want_dl) {
            fold<4>(dl, lane, 16); fold<2>(dl, lane, 8);
            const float x = dl[0] + __shfl_xor_sync(0xffffffffu, dl[0], 4);
            if (!(lane & 4)) sred_[ph][1][wq][col] = x;
        }
        if (want_da) {
            fold<4>(t1, lane, 16); fold<2>(t1, lane, 8);
            const float x = t1[0] + __shfl_xor_sync(0xffffffffu, t1[0], 4);
            if (!(lane & 4)) sred_[ph][0][wq][col] = x;
        }
        if (want_da) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ksum += __shfl_xor_sync(0xffffffffu, ksum, o);
            if (lane == 0) swk_[ph][tid >> 5] = ksum;
        }
    }
    if (NORM) {
        // Through the normalisation: dx = r (dx^ - x^ <x^, dx^>).  The staged tiles hold dk^ and dq^ token-major, like the
        // K^ and Q^ tiles: 16 lanes to a row, one 16-byte chunk each, the row's dot product by shuffles.
        csync();                             // the staged tiles are complete
        const int ci = tid & 15;
#pragma unroll
        for (int r = tid >> 4; r < C; r += kBwdCompute / 16) {
            const uint32_t off = (ci >> 3) * 8192 + sw128_chunk(r, ci & 7);
            float a8[8], x8[8], b8[8], y8[8], ck = 0.f, cq = 0.f;
            load8(sm + oStDk + off, a8);
            load8(sm + oK + off, x8);
            load8(sm + oStDq + off, b8);
            load8(sm + oQ + off, y8);
#pragma unroll
            for (int e = 0; e < 8; ++e) { ck = fmaf(a8[e], x8[e], ck); cq = fmaf(b8[e], y8[e], cq); }
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) {
                ck += __shfl_xor_sync(0xffffffffu, ck, o);
                cq += __shfl_xor_sync(0xffffffffu, cq, o);
            }
            const float2 rn = srn[r];        // {1/|k|, 1/|q|}
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                a8[e] = rn.x * fmaf(-ck, x8[e], a8[e]);
                b8[e] = rn.y * fmaf(-cq, y8[e], b8[e]);
            }
            sts128(sm + oStDk + off, pack8(a8));
            sts128(sm + oStDq + off, pack8(b8));
        }
    }
    fence_proxy_async();
    tc_fence_before();
    nb_arrive(kNbOut, kBwdNb);
    nb_sync(kNbEnd, kBwdThreads);        // every read of this chunk's tiles and accumulators is done
    }  // chunk loop
    }  // epilogue threads
    tc_fence_before();
    __syncthreads();
    if (tid < 32) tmem_dealloc(tb, 512);
    if (tid == 0 && blockIdx.x == 0) grid_dep_wait();            // when this kernel has completed, so has the one before it
}

template <class K>
cudaError_t set_smem(K kern, size_t bytes) { return set_max_smem_once(reinterpret_cast<const void*>(kern), bytes); }

}  // namespace

namespace {

// Chunks [n0, n1) of every sequence; what comes after them is in dhT, what goes before them to dh0.
cudaError_t chain_bwd(const ChunkArgs& a, int n0, int n1, const float* dhT, float* dh0) {
    const qd_shape& s = a.s;
    const int Tp = tc_padded_T(s);
    const uint64_t BH = (uint64_t)s.B * s.H, Ns = Tp / kChunk;
    const int rows = chain_rows(BH);
    CUtensorMap mWt, mdO, mQg, mK, mP, mdHs, mdDt;
    if (!make_tmap_bf16_2d(&mWt, a.ws + a.TL.Wt, 64, BH * Ns * D, 128, 128) ||
        !make_tmap_tokens(&mdO, a.dO, s.B, s.T, s.H, D, 64) ||
        !make_tmap_bf16_2d(&mQg, a.ws + a.TL.Qg, D, BH * Tp, D * 2, 64) ||
        !make_tmap_tokens(&mK, a.k, s.B, s.T, s.H, D, 64) ||
        !make_tmap_bf16_2d(&mP, a.ws + a.TL.P, 64, BH * Tp, 128, 64) ||
        !make_tmap_bf16_2d(&mdHs, a.ws + a.TL.dhsT, D, BH * Ns * D, D * 2, rows) ||
        !make_tmap_bf16_2d(&mdDt, a.ws + a.TL.dDt, 64, BH * Ns * D, 128, rows))
        return cudaErrorInvalidValue;
    ChainBwdParams p{};
    const bool first = dhT == a.dhT;
    p.Tp = Tp; p.H = s.H; p.N = n1 - n0; p.n0 = n0; p.Ns = (int)Ns;
    p.dhT_early = first && a.own_predecessor ? 1 : 0;
    p.rk = a.norm ? (const float*)(a.ws + a.TL.rqk) + BH * Tp : nullptr;
    p.g = (const float*)(a.ws + a.TL.g);
    p.dhT = dhT; p.dh0 = dh0;
    p.status = (unsigned*)(a.ws + a.TL.status);
    p.next = first ? (unsigned*)(a.ws + a.TL.next) : nullptr;
    const auto kern = rows == D ? k_tc_chain_bwd<D> : k_tc_chain_bwd<D / 2>;
    cudaError_t e = set_smem(kern, kChainSmem);
    if (e != cudaSuccess) return e;
    return launch_overlapped(kern, dim3((unsigned)(BH * (D / rows))), dim3(kChainThreads), kChainSmem, a.stream,
                             mWt, mdO, mQg, mK, mP, mdHs, mdDt, p);
}

cudaError_t chunk_bwd(const ChunkArgs& a, int n0, int n1, bool beside, int counter) {
    const qd_shape& s = a.s;
    const int Tp = tc_padded_T(s);
    const uint64_t BH = (uint64_t)s.B * s.H, Ns = Tp / kChunk, N = n1 - n0;
    ChunkBwdMaps m;
    if (!make_tmap_tokens(&m.dQ, a.dq, s.B, s.T, s.H, D, 64) ||
        !make_tmap_tokens(&m.dK, a.dk, s.B, s.T, s.H, D, 64) ||
        !make_tmap_tokens(&m.dV, a.dv, s.B, s.T, s.H, D, 64) ||
        !make_tmap_tokens(&m.Q, a.q, s.B, s.T, s.H, D, 64) ||
        !make_tmap_tokens(&m.K, a.k, s.B, s.T, s.H, D, 64) ||
        !make_tmap_tokens(&m.V, a.v, s.B, s.T, s.H, D, 64) ||
        !make_tmap_tokens(&m.dO, a.dO, s.B, s.T, s.H, D, 64) ||
        !make_tmap_bf16_2d(&m.Mt, a.ws + a.TL.Mt, 64, BH * Tp, 128, 64) ||
        !make_tmap_bf16_2d(&m.P, a.ws + a.TL.P, 64, BH * Tp, 128, 64) ||
        !make_tmap_bf16_2d(&m.Dt, a.ws + a.TL.Dt, 64, BH * Ns * D, 128, 128) ||
        !make_tmap_bf16_2d(&m.dDt, a.ws + a.TL.dDt, 64, BH * Ns * D, 128, 128) ||
        !make_tmap_bf16_2d(&m.Hs, a.ws + a.TL.hsT, D, BH * Ns * D, D * 2, 128) ||
        !make_tmap_bf16_2d(&m.dHs, a.ws + a.TL.dhsT, D, BH * Ns * D, D * 2, 128))
        return cudaErrorInvalidValue;
    ChunkBwdParams p{};
    p.T = s.T; p.Tp = Tp; p.H = s.H; p.N = (int)N; p.n0 = n0; p.beside = beside; p.Ns = (int)Ns; p.BH = (int)BH; p.total = (int)(BH * N);
    p.group = (int)std::min<uint64_t>(BH, 64);
    p.beta = (const bf16*)a.beta; p.alpha = (const bf16*)a.alpha; p.lam = (const bf16*)a.lam;
    p.g = (const float*)(a.ws + a.TL.g);
    p.dbeta = a.dbeta; p.dalpha = a.dalpha; p.dlam = a.dlam;
    p.logits = a.logits ? 1 : 0;
    p.rqk = a.norm ? (const float*)(a.ws + a.TL.rqk) : nullptr;
    p.status = (unsigned*)(a.ws + a.TL.status);
    p.next = (unsigned*)(a.ws + a.TL.next) + counter;
    // the instance without lambda / without the forget gate needs the input AND its gradient to be absent
    const bool lam = a.lam || a.dlam, alpha = a.alpha || a.dalpha;
    using Kern = decltype(&k_tc_chunk_bwd<true, true, false>);
    static const Kern table[8] = {
        k_tc_chunk_bwd<false, false, false>, k_tc_chunk_bwd<false, false, true>, k_tc_chunk_bwd<false, true, false>,
        k_tc_chunk_bwd<false, true, true>,   k_tc_chunk_bwd<true, false, false>, k_tc_chunk_bwd<true, false, true>,
        k_tc_chunk_bwd<true, true, false>,   k_tc_chunk_bwd<true, true, true>,
    };
    const Kern kern = table[(lam ? 4 : 0) + (alpha ? 2 : 0) + (a.norm ? 1 : 0)];
    cudaError_t e = set_smem(kern, kBwdSmem);
    if (e != cudaSuccess) return e;
    // persistent: one CTA per SM
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<uint64_t>(BH * N, (uint64_t)sms);
    return launch_overlapped(kern, dim3(grid), dim3(kBwdThreads), kBwdSmem, a.stream, m, p);
}

int chunks(const ChunkArgs& a) { return (a.s.T + kChunk - 1) / kChunk; }

}  // namespace

cudaError_t tc_chain_bwd(const ChunkArgs& a) { return chain_bwd(a, 0, chunks(a), a.dhT, a.dh0); }
cudaError_t tc_chunk_bwd(const ChunkArgs& a) { return chunk_bwd(a, 0, chunks(a), false, 0); }

// With few long sequences the reverse chain leaves SMs idle, as the forward chain does (tc_fwd_parts).  Its chunks are then taken
// in two parts or three, and those of a part, the later ones of every sequence first, are differentiated beside the chain of the next:
//     chain [n, N), chain [0, n), chunks [n, N), chunks [0, n)
//     chain [n2, N), chain [n1, n2), chunks [n2, N), chain [0, n1), chunks [n1, n2), chunks [0, n1)
// in one stream, by programmatic launch alone.  Chunks that stand after a chain that they do not depend on may start when every CTA
// of that chain has begun its work, which it does when all before it has completed; they touch the rows of their own chunks, so
// they need not wait, and what remains of their work when the chain leaves its SMs is taken by further CTAs.  Their first CTA
// waits for the chain before it leaves, so whatever is launched next and waits for them comes after the chain too.
// dh passes on in fp32, through U~'s section, which no kernel of the backward reads (a CTA of the chain has read its part of it
// when it writes it); results are those of one part, bit for bit.
// Where the line n lies: the fewer sequences, the more SMs for the chunks beside a chain and the more they are given:
// n = N (20 + sequences) / 88.  Backward, us, one part / halves / this: 32 sequences of 512 chunks 1332 / 1191 / 1160, 16 of 512
// 854 / 728 / 709, 8 of 128 179 / 169 / 166, 40 of 128 389 / 384 / 374.  Where it is used: 48 of 256 899 / 856, but 48 of 128 446 / 443, 64
// of 256 1159 / 1164; 40 of 96 292 / 285, 32 of 96 247 / 243, 24 of 64 136 / 133, 4 of 64 80.3 / 78.2; but 40 of 64 196 / 201, 32 of 32
// 85.6 / 90.9, 16 of 32 63.9 / 64.3, 2 of 64 72.9 / 77.1.
// Three parts let the first chain, beside which nothing runs, be a third to a half as long, for one more pair of launches: n1 = N sequences
// / 56 (34 at most), n2 = n1 + 5 N / 16, near the best of a sweep over both.  Two parts / three: 32 sequences of 512 chunks 1117 / 1074, 16 of
// 512 731 / 694, 12 of 1024 1258 / 1210, 12 of 256 334 / 329, 12 of 171 233 / 228, 16 of 128 196 / 192, 32 of 128 288 / 281, 36 of 128
// 312 / 309; but 32 of 112 257 / 256, 12 of 128 178.6 / 180.2, 40 of 140 369 / 370, 40 of 256 645 / 642, and the sweep had 8 of 512
// 596 / 604, 48 of 256 853 / 862.
int tc_bwd_parts(const ChunkArgs& a) {
    const long long BH = (long long)a.s.B * a.s.H, N = chunks(a);
    if (BH > 48 || N < 64 || N < 3 * BH || BH * N < 256) return 1;
    return BH >= 12 && BH <= 36 && N >= 128 && BH * N >= 2048 ? 3 : 2;
}

cudaError_t tc_bwd(const ChunkArgs& a, int parts) {
    const int N = chunks(a), BH = a.s.B * a.s.H;
    float* carry = (float*)(a.ws + a.TL.Ut);                 // [BH][D][D], from four chunks on
    const int lo = parts == 2 ? (int)((long long)N * (20 + BH) / 88) : (int)((long long)N * std::min(BH, 34) / 56);
    const int hi = parts == 2 ? lo : lo + (int)((long long)N * 5 / 16);
    cudaError_t e = chain_bwd(a, hi, N, a.dhT, carry);
    int n1 = N;                                              // the chunks from here on are differentiated; chains have come to n0
    for (int i = 0, n0 = hi; i + 1 < parts; ++i) {
        const int to = i + 2 == parts ? 0 : lo;
        if (e == cudaSuccess) e = chain_bwd(a, to, n0, carry, to ? carry : a.dh0);
        if (e == cudaSuccess) e = chunk_bwd(a, n0, n1, true, i);
        n1 = n0;
        n0 = to;
    }
    return e == cudaSuccess ? chunk_bwd(a, 0, n1, false, parts - 1) : e;
}

}  // namespace qd
