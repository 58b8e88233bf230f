// What the kernels of the accurate path share: arguments, accumulator tiles, the triangular inverse, per-token sums, launches.
// The path serves fp32 storage (1e-4 parity needs full fp32 products, split_chunk.cu) and, in bf16, the head dimensions that the
// tcgen05 kernels do not cover (split_bf16.cu).  It follows the chunk equations of Section 3.3.2:
//   g_r = sum_{i<=r} log alpha_i,  gamma_r = e^{g_r},  Gamma_ri = e^{g_r-g_i} (r >= i)
//   X = K + diag(lambda) Q
//   A = strictLower(diag(beta)(Gamma o X K^T)),  M = (I+A)^-1,  T = M diag(beta)     (UT transform)
//   U~ = T V,  W<- = T diag(gamma) X                                                  (extended WY)
//   Delta = U~ - W<- h;  O = diag(gamma) Q h + (Gamma o Q K^T o causal) Delta
//   h <- gamma_C h + (diag(gamma_C/gamma) K)^T Delta                                  (chunk-level update)
// and, for the backward, the exact gradient of those equations (the paper prints none).
// Every decay factor is formed as exp of a non-positive difference of cumulative logs; no
// quotient of cumulative products is ever taken.
#pragma once
#include "internal.h"
#include "sm100.cuh"
#include "tf32.cuh"

namespace qd {
namespace {

constexpr int C = kChunk;
constexpr int NT = 256;            // threads of most kernels here: 8 warps
constexpr int LDC = C + 4;         // leading dimension of the C x C matrices in shared memory
constexpr int LDI = C / 2 + 4;     // of the inverse's scratch

struct Ptrs {
    int B, T, Tp, H, N;              // the workspace holds Tp = 64 N >= T rows per sequence; rows past T are tokens with
                                     // beta = 0, alpha = 1, q = k = v = dO = 0 (exact no-ops of the recurrence)
    const void *q, *k, *v, *beta, *alpha, *lam, *dO;
    const float *h0, *dhT;
    void *o, *dq, *dk_, *dv_;
    float *hT, *dbeta, *dalpha, *dlam, *dh0;
    float* g;
    void *P, *W, *U, *D, *dD;
    float *M, *hs, *dhs, *kdhd, *dhh;
    int nslices, save;
    int logits;                      // beta, alpha, lambda are logits of sigmoid gates
    float* rqk;                      // non-null (QD_NORM_QK): q and k are L2-normalised in here; [0, BH*Tp) 1/|q_t|, then 1/|k_t|
    unsigned* status;                // cleared by the preparation kernel
};

// ---- products -----------------------------------------------------------------------------------------------------
// acc += A B for the (16 MT) x (8 NTL) tile of this warp at row m0, column n0: contraction over [kb, k1), a(m, k) and b(k, n)
// fetch the operands.  Lane (g = lane / 4, t = lane % 4) holds, of every
// 16 x 8 piece, rows g and g + 8, columns 2t and 2t + 1.
// The tensor instruction truncates as it accumulates, which over a long contraction biases the sum by 1e-6 of itself; so it
// only sums 16 terms at a time, from zero, the small products (lo hi, hi lo) of all of them before the large ones, and those sums
// are added with rounded fp32 additions.  Measured against fp64 on 1024 tokens, d = 64, slowly forgetting gates, rms error of the
// outputs: 1.2e-6 with one running sum, 3.0e-7 with the three products of 8 terms after those of the 8 before, 2.5e-7 so, 2.3e-7
// with plain fp32 FMAs.
__device__ __forceinline__ void add2(float& x, float& y, float a, float b) {
    asm("{\n\t.reg .b64 u, v;\n\tmov.b64 u, {%0, %1};\n\tmov.b64 v, {%2, %3};\n\tadd.rn.f32x2 u, u, v;\n\tmov.b64 {%0, %1}, u;\n\t}"
        : "+f"(x), "+f"(y) : "f"(a), "f"(b));
}
template <int MT, int NTL, class FA, class FB>
__device__ __forceinline__ void wmm(float (&acc)[MT][NTL][4], int m0, int n0, int k1, FA a, FB b, int kb = 0) {
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
    constexpr int KS = 2, JN = NTL > 2 ? 2 : NTL;      // k steps per group; columns whose sums are open at a time
#pragma unroll 1
    for (int k0 = kb; k0 < k1; k0 += 8 * KS) {
        uint32_t ah[KS][MT][4], al[KS][MT][4];
#pragma unroll
        for (int s = 0; s < KS; ++s)
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float x = a(m0 + 16 * i + g + 8 * (e & 1), k0 + 8 * s + t + 4 * (e >> 1));
                    tf32_split(x, ah[s][i][e], al[s][i][e]);
                }
#pragma unroll
        for (int jb = 0; jb < NTL; jb += JN) {
            float part[MT][JN][4];
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int j = 0; j < JN; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) part[i][j][e] = 0.f;
            uint32_t bh[KS][JN][2], bl[KS][JN][2];
#pragma unroll
            for (int s = 0; s < KS; ++s)
#pragma unroll
                for (int j = 0; j < JN; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float x = b(k0 + 8 * s + t + 4 * e, n0 + 8 * (jb + j) + g);
                        tf32_split(x, bh[s][j][e], bl[s][j][e]);
                    }
            auto add = [&](int s, const uint32_t (&x)[KS][MT][4], const uint32_t (&y)[KS][JN][2]) {
#pragma unroll
                for (int i = 0; i < MT; ++i)
#pragma unroll
                    for (int j = 0; j < JN; ++j) mma_tf32(part[i][j], x[s][i], y[s][j]);
            };
#pragma unroll
            for (int s = 0; s < KS; ++s) { add(s, al, bh); add(s, ah, bl); }
#pragma unroll
            for (int s = 0; s < KS; ++s) add(s, ah, bh);
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int j = 0; j < JN; ++j) {
                    add2(acc[i][jb + j][0], acc[i][jb + j][1], part[i][j][0], part[i][j][1]);
                    add2(acc[i][jb + j][2], acc[i][jb + j][3], part[i][j][2], part[i][j][3]);
                }
        }
    }
}
// ---- accumulator tiles of a warp --------------------------------------------------------------------------------------
template <int MT, int NTL>
__device__ __forceinline__ void zero(float (&acc)[MT][NTL][4]) {
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NTL; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
}
// f(row, column, value pair) over the accumulator of a warp: values at (row, column) and (row, column + 1)
template <int MT, int NTL, class F>
__device__ __forceinline__ void each(float (&acc)[MT][NTL][4], int m0, int n0, F f) {
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < NTL; ++j) f(m0 + 16 * i + 8 * h + g, n0 + 8 * j + 2 * t, acc[i][j][2 * h], acc[i][j][2 * h + 1]);
}
// f(row, column, value pair of a, value pair of b) over two accumulators of the same tile
template <int MT, int NTL, class F>
__device__ __forceinline__ void each2(float (&a)[MT][NTL][4], float (&b)[MT][NTL][4], int m0, int n0, F f) {
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < NTL; ++j)
                f(m0 + 16 * i + 8 * h + g, n0 + 8 * j + 2 * t, a[i][j][2 * h], a[i][j][2 * h + 1], b[i][j][2 * h], b[i][j][2 * h + 1]);
}
// Row sums over a warp's tile: f(row, column, x0, x1) gives what the pair adds; the sum over the warp's columns of row r
// goes to dst[r] (one lane of four writes).
template <int MT, int NTL, class F>
__device__ __forceinline__ void row_sums(float (&acc)[MT][NTL][4], int m0, int n0, float* dst, F f) {
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float s = 0.f;
#pragma unroll
            for (int j = 0; j < NTL; ++j) s += f(m0 + 16 * i + 8 * h + g, n0 + 8 * j + 2 * t, acc[i][j][2 * h], acc[i][j][2 * h + 1]);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (t == 0) dst[m0 + 16 * i + 8 * h + g] = s;
        }
}

__device__ __forceinline__ void st2(float* p, float x, float y) { *reinterpret_cast<float2*>(p) = make_float2(x, y); }
__device__ __forceinline__ void st2(__nv_bfloat16* p, float x, float y) {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(x, y);
}
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 ld2(const __nv_bfloat16* p) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// M = (I + A)^-1 of a unit lower-triangular 64 x 64 matrix (A strictly lower, sA, untouched above its diagonal), into sM.
// The four 16 x 16 diagonal blocks are inverted by right-looking substitution, a column in the registers of a lane; then
// blocks are joined twice, M21 = -M22 (A21 M11), on the tensor instruction with the inner product in sS.  The chain of dependent
// steps is 16 + 4 products long; a column per thread over all 64 rows took 30 us here, joins by FMAs 5 of 50 us more on 1024 chunks
// of d = 64, 2 of 27 on 128 chunks of fp32, d = 128.
__device__ __forceinline__ void invert_unit_lower(const float* sA, float* sM, float* sS) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int e = tid; e < C * C / 2; e += NT) {                  // zeros above the diagonal blocks
        const int r = e / (C / 2), c = e % (C / 2);              // every row r, columns from its block's end on
        const int col = (r / 16 + 1) * 16 + c;
        if (col < C) sM[r * LDC + col] = 0.f;
    }
    for (int e = tid; e < 16 * 16; e += NT) sM[(e / 16) * LDC + 48 + e % 16] = 0.f;
    if (warp < 4 && lane < 16) {
        const float* Ab = sA + warp * 16 * LDC + warp * 16;
        float m[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) m[r] = r == lane ? 1.f : 0.f;
#pragma unroll
        for (int i = 0; i < 15; ++i)
#pragma unroll
            for (int r = i + 1; r < 16; ++r) m[r] = fmaf(-Ab[r * LDC + i], m[i], m[r]);
#pragma unroll
        for (int r = 0; r < 16; ++r) sM[(warp * 16 + r) * LDC + warp * 16 + lane] = m[r];
    }
    __syncthreads();
#pragma unroll
    for (int S = 16; S <= 32; S *= 2) {                          // join pairs of S x S blocks, a 16 x 8 piece per warp
        const int o = S == 16 ? (warp >> 1) * 32 : 0, m0 = S == 16 ? 0 : (warp & 1) * 16, n0 = S == 16 ? (warp & 1) * 8 : (warp >> 1) * 8;
        const bool mine = S == 32 || warp < 4;
        float x[1][1][4];
        zero(x);
        if (mine) {
            wmm(x, m0, n0, S, [&](int m, int k) { return sA[(o + S + m) * LDC + o + k]; }, [&](int k, int n) { return sM[(o + k) * LDC + o + n]; });
            each(x, m0, n0, [&](int m, int n, float u, float v) { st2(sS + (o + m) * LDI + n, u, v); });
        }
        __syncthreads();
        zero(x);
        if (mine) {
            wmm(x, m0, n0, S, [&](int m, int k) { return sM[(o + S + m) * LDC + o + S + k]; }, [&](int k, int n) { return sS[(o + k) * LDI + n]; });
            each(x, m0, n0, [&](int m, int n, float u, float v) { st2(sM + (o + S + m) * LDC + o + n, -u, -v); });
        }
        __syncthreads();
    }
}

// In-chunk cumulative log-decays of 64 tokens by the first two warps: thread t < 64 passes log alpha_t, sg[t] becomes g_t.
// One thread adds them up in order, under the tile loads: neighbours then share their rounding errors, which cancel in the
// differences g_r - g_i that the decays are made of; a tree of sums costs half as much again in the error of the outputs.
__device__ __forceinline__ void scan64(float x, float* sg) {
    sg[threadIdx.x] = x;
    asm volatile("bar.sync 1, 64;" ::: "memory");
    if (threadIdx.x == 0) {
        float acc = 0.f;
#pragma unroll
        for (int r = 0; r < C; r += 4) {
            float4 v = *reinterpret_cast<float4*>(sg + r);
            v.x += acc; v.y += v.x; v.z += v.y; v.w += v.z; acc = v.w;
            *reinterpret_cast<float4*>(sg + r) = v;
        }
    }
    asm volatile("bar.sync 1, 64;" ::: "memory");
}

// Copies of the state chains: by four extra warps, which issue them while the others compute.  Issued by the warps that compute, the
// copies and the decay factors of a chunk were 800 - 1100 of its 3500 - 4500 cycles.  Forward and backward, before and with them:
// fp32 16 sequences of 512 tokens, 128 x 128 170 -> 161 us, 8 of 1024, 64 x 128 183 -> 161, 128 of 1024, 64 x 64 947 -> 901; bf16 64 x 64,
// 64 of 1024 247 -> 240, 8 of 1024 102 -> 91, 2 of 4096 287 -> 246.  A warp's share of the output moved to further warps as well: 2 %
// more on narrow slices, 2 % less on wide ones.
constexpr int kLoaders = 128;
template <int N> __device__ __forceinline__ void fetch_wait_but() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void fetch_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// decay factors of a chunk's tokens, thread `me` < 64 token `me`: fetched a chunk ahead, written before the barrier that ends the present one
struct ChainCoef {
    float g = 0.f, gC = 0.f, rq = 1.f, rk = 1.f;
    __device__ __forceinline__ void get(const Ptrs& p, size_t wrow0, size_t nrows, int me = threadIdx.x) {
        if (me >= C) return;
        g = p.g[wrow0 + me]; gC = p.g[wrow0 + C - 1];
        if (p.rqk) { rq = p.rqk[wrow0 + me]; rk = p.rqk[nrows + wrow0 + me]; }
    }
    __device__ __forceinline__ void put(float* gq, float* gk, float* gc, int me = threadIdx.x) const {
        if (me >= C) return;
        gq[me] = expf(g) * rq; gk[me] = expf(gC - g) * rk;
        if (me == 0) *gc = expf(gC);
    }
};
// Per token, from the row sums (prow: dP o P, t1, t2, d beta, d lambda) and the column sums (cP: dP o P, cA: dA o A; db1: dT o M,
// of token threadIdx.x): d beta, d lambda, and the decay gradient: dg, its reverse in-chunk cumulative sum,
// d alpha = d log alpha / alpha.  sdg and skd are scratch.
template <typename IO, int NC>
__device__ __forceinline__ void token_gradients(const Ptrs& p, const float (&prow)[5][4][C], const float (&cP)[NC][C],
                                                const float (&cA)[NC][C], float db1, const float* sbeta, const float* slam,
                                                const float* salpha, const float* sgam, float* sdg, float* skd, size_t row0,
                                                size_t wrow0, int bh, int n, int live) {
    const int tid = threadIdx.x, H = p.H;
    const size_t nrows = (size_t)p.B * H * p.Tp, BHN = (size_t)p.B * H * p.N;
    if (tid < C) {
        auto rows = [&](int w) { return prow[w][0][tid] + prow[w][1][tid] + prow[w][2][tid] + prow[w][3][tid]; };
        const float be = sbeta[tid], la = slam[tid], db2 = rows(3), dl = rows(4);
        float kd = 0.f;
        for (int s = 0; s < p.nslices; ++s) kd += p.kdhd[(size_t)s * nrows + wrow0 + tid];
        float sP = 0.f, sA = 0.f;
#pragma unroll
        for (int c = 0; c < NC; ++c) { sP += cP[c][tid]; sA += cA[c][tid]; }
        sdg[tid] = rows(0) - sP + be * db2 - sA + rows(1) + rows(2) - kd;
        skd[tid] = kd;
        if (tid < live) {
            const size_t r = row0 + (size_t)tid * H;
            // with logit inputs the gradients are taken w.r.t. the logits: sigmoid' = s (1 - s), (log sigmoid)' = 1 - s
            const float db = db1 + db2;
            p.dbeta[r] = p.logits ? db * be * (1.f - be) : db;
            if (p.dlam) p.dlam[r] = p.logits ? dl * la * (1.f - la) : dl;
        }
    }
    __syncthreads();
    if (tid < 32 && p.dalpha) {
        // lane owns tokens 2 lane, 2 lane + 1; d log alpha_i = sum_{r >= i} dg_r (suffix sums)
        float dhh = 0.f, kds = skd[2 * tid] + skd[2 * tid + 1];
        if (tid < p.nslices) dhh = p.dhh[(size_t)tid * BHN + (size_t)bh * p.N + n];
        dhh = warp_sum(dhh);
        kds = warp_sum(kds);
        const float a = sdg[2 * tid];
        float b2 = sdg[2 * tid + 1];
        if (tid == 31) b2 += sgam[C - 1] * dhh + kds;
        float sfx = a + b2;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float t = __shfl_down_sync(0xffffffffu, sfx, o);
            if (tid + o < 32) sfx += t;
        }
        const size_t r = row0 + (size_t)(2 * tid) * H;
        const float a0 = salpha[2 * tid], a1 = salpha[2 * tid + 1];
        if (2 * tid < live) p.dalpha[r] = p.logits ? sfx * (1.f - a0) : sfx / a0;
        if (2 * tid + 1 < live) p.dalpha[r + H] = p.logits ? (sfx - a) * (1.f - a1) : (sfx - a) / a1;
    }
}

inline Ptrs make_ptrs(const ChunkArgs& a) {
    Ptrs p{};
    p.B = a.s.B; p.T = a.s.T; p.Tp = split_padded_T(a.s); p.H = a.s.H; p.N = p.Tp / kChunk;
    p.q = a.q; p.k = a.k; p.v = a.v; p.beta = a.beta; p.alpha = a.alpha; p.lam = a.lam; p.dO = a.dO;
    p.h0 = a.h0; p.dhT = a.dhT; p.o = a.o; p.dq = a.dq; p.dk_ = a.dk; p.dv_ = a.dv;
    p.hT = a.hT; p.dbeta = a.dbeta; p.dalpha = a.dalpha; p.dlam = a.dlam; p.dh0 = a.dh0;
    p.g = (float*)(a.ws + a.L.g);
    p.P = a.ws + a.L.P; p.W = a.ws + a.L.W; p.U = a.ws + a.L.U;
    p.D = a.ws + a.L.D; p.dD = a.ws + a.L.dD;
    p.M = (float*)(a.ws + a.L.M);
    p.hs = (float*)(a.ws + a.L.hs); p.dhs = (float*)(a.ws + a.L.dhs);
    p.kdhd = (float*)(a.ws + a.L.kdhd); p.dhh = (float*)(a.ws + a.L.dhh);
    p.nslices = a.s.dv / a.L.slice; p.save = a.save ? 1 : 0; p.logits = a.logits ? 1 : 0;
    p.rqk = a.norm ? (float*)(a.ws + a.L.rqk) : nullptr;
    p.status = (unsigned*)(a.ws + a.L.status);
    return p;
}

// Small grids, where the gap between two kernels is a tenth of the time, are launched while the kernel before them drains.
// Larger ones are not: CTAs that come early take the SMs that are free first instead of one each.  Measured with this line at 0,
// 16, 32, 64, 96, 128, 148 and 296 on eleven sizes of fp32 64 x 64 and 128 x 128 and bf16 64 x 64 and 128 x 64, training passes:
// up to 64 every step gains or changes nothing (2 sequences of 256 tokens: 82 -> 74, 127 -> 120, 57 -> 50, 68 -> 60 us; grids of
// 64, 8 sequences of 512: 109 -> 107, 170 -> 165, 70 -> 70, 88 -> 87), but for fp32 128 x 128 on 8 sequences of 1024 (262 -> 266); at
// 128 the same sizes lose (16 sequences of 512: 109 -> 112, 176 -> 187, 72 -> 80, 89 -> 92; 64 of 1024, bf16 64 x 64: 250 -> 302)
// except bf16 128 x 64 on 32 and 64 sequences (121 -> 118, 363 -> 358).
template <class K, class... Args>
cudaError_t launch(K kern, int grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaError_t e = set_max_smem_once(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
    if (grid <= 64) return launch_overlapped(kern, dim3((unsigned)grid), dim3(threads), smem, stream, args...);
    kern<<<grid, threads, smem, stream>>>(args...);
    return cudaGetLastError();
}

}  // namespace
}  // namespace qd
