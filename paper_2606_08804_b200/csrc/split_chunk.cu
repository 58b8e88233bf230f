// Chunkwise Q-Delta forward and backward with fp32-accurate products on the warp-level tensor instructions.
//
// This is the path for fp32 storage (1e-4 parity needs full fp32 products) and for the head dimensions the tcgen05
// kernels do not cover.  It follows the chunk equations of Section 3.3.2:
//   g_r = sum_{i<=r} log alpha_i,  gamma_r = e^{g_r},  Gamma_ri = e^{g_r-g_i} (r >= i)
//   X = K + diag(lambda) Q
//   A = strictLower(diag(beta)(Gamma o X K^T)),  M = (I+A)^-1,  T = M diag(beta)     (UT transform)
//   U~ = T V,  W<- = T diag(gamma) X                                                  (extended WY)
//   Delta = U~ - W<- h;  O = diag(gamma) Q h + (Gamma o Q K^T o causal) Delta
//   h <- gamma_C h + (diag(gamma_C/gamma) K)^T Delta                                  (chunk-level update)
// and, for the backward, the exact gradient of those equations (the paper prints none).
// Every decay factor is formed as exp of a non-positive difference of cumulative logs; no
// quotient of cumulative products is ever taken.
//
// Arithmetic.  A product of two fp32 matrices is three m16n8k8 tf32 products of their 11-bit halves, x = hi + lo, both
// halves rounded: hi hi + hi lo + lo hi, accumulated in fp32 (the dropped lo lo term is below 2^-22 of the product).  A
// bf16 operand is exact in one tf32 half, so bf16 storage needs two products, or one when both operands are stored.
// Measured on a B200: m16n8k8 runs at 276 TFLOP/s, i.e. 92 as three products, against 68 for packed fp32 FMAs and 39 for
// scalar ones; the difference that counts more is operand traffic, 16 shared-memory loads for 24 instructions of 1024
// multiply-adds here.  Operands live in shared memory as fp32 tiles with padded rows; each kernel reads every global
// operand once.
#include "internal.h"
#include "sm100.cuh"
#include "tf32.cuh"
#include "planes.cuh"

namespace qd {
namespace {

constexpr int C = kChunk;
constexpr int NT = 256;            // threads of the kernels that take a chunk each: 8 warps
constexpr int LDC = C + 4;         // leading dimension of the C x C matrices in shared memory
constexpr int LDI = C / 2 + 4;    // of the inverse's scratch
constexpr int kPad = 4;            // of a d-wide tile: rows g, columns t of a fragment fall on banks 4 g + t

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

template <typename IO> constexpr int kTerms = 2;                 // tf32 halves that a stored value needs
template <> constexpr int kTerms<__nv_bfloat16> = 1;

// ---- products -----------------------------------------------------------------------------------------------------
// acc += A B for the (16 MT) x (8 NTL) tile of this warp at row m0, column n0: contraction extent K, a(m, k) and b(k, n)
// fetch the operands, TA / TB say how many tf32 halves they need.  Lane (g = lane / 4, t = lane % 4) holds, of every
// 16 x 8 piece, rows g and g + 8, columns 2t and 2t + 1.
// EX: the tensor instruction truncates as it accumulates, which over a long contraction biases the sum by 1e-6 of itself;
// with EX (fp32 storage) it only sums 16 terms at a time, from zero, and those sums are added with rounded fp32 additions.
// Measured against fp64 on 1024 tokens: slowly forgetting gates, rms error of the outputs 1.2e-6 without, 2.9e-7 with, 2.6e-7 for plain fp32 FMAs.
__device__ __forceinline__ void add2(float& x, float& y, float a, float b) {
    asm("{\n\t.reg .b64 u, v;\n\tmov.b64 u, {%0, %1};\n\tmov.b64 v, {%2, %3};\n\tadd.rn.f32x2 u, u, v;\n\tmov.b64 {%0, %1}, u;\n\t}"
        : "+f"(x), "+f"(y) : "f"(a), "f"(b));
}
template <int MT, int NTL, int TA, int TB, bool EX, class FA, class FB>
__device__ __forceinline__ void wmm(float (&acc)[MT][NTL][4], int m0, int n0, int K, FA a, FB b) {
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
    constexpr int KS = EX ? 2 : 1, JN = EX && NTL > 2 ? 2 : NTL;      // k steps per group; columns whose sums are open at a time
#pragma unroll EX ? 1 : 2
    for (int k0 = 0; k0 < K; k0 += 8 * KS) {
        uint32_t ah[KS][MT][4], al[KS][MT][4];
#pragma unroll
        for (int s = 0; s < KS; ++s)
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float x = a(m0 + 16 * i + g + 8 * (e & 1), k0 + 8 * s + t + 4 * (e >> 1));
                    if (TA == 2) tf32_split(x, ah[s][i][e], al[s][i][e]);
                    else ah[s][i][e] = __float_as_uint(x);
                }
#pragma unroll
        for (int jb = 0; jb < NTL; jb += JN) {
            float part[MT][JN][4];
            float (*c)[JN][4] = part;
            if (EX) {
#pragma unroll
                for (int i = 0; i < MT; ++i)
#pragma unroll
                    for (int j = 0; j < JN; ++j)
#pragma unroll
                        for (int e = 0; e < 4; ++e) part[i][j][e] = 0.f;
            }
#pragma unroll
            for (int s = 0; s < KS; ++s) {
                uint32_t bh[JN][2], bl[JN][2];
#pragma unroll
                for (int j = 0; j < JN; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float x = b(k0 + 8 * s + t + 4 * e, n0 + 8 * (jb + j) + g);
                        if (TB == 2) tf32_split(x, bh[j][e], bl[j][e]);
                        else bh[j][e] = __float_as_uint(x);
                    }
#pragma unroll
                for (int term = (TA == 2 ? 0 : 1); term < 3; ++term) {       // lo hi, hi lo, hi hi
                    if (term == 1 && TB == 1) continue;
#pragma unroll
                    for (int i = 0; i < MT; ++i)
#pragma unroll
                        for (int j = 0; j < JN; ++j)
                            mma_tf32(EX ? c[i][j] : acc[i][jb + j], term == 0 ? al[s][i] : ah[s][i], term == 1 ? bl[j] : bh[j]);
                }
            }
            if (EX) {
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
}
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

// ---- tiles --------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void st2(float* p, float x, float y) { *reinterpret_cast<float2*>(p) = make_float2(x, y); }
__device__ __forceinline__ void st2(__nv_bfloat16* p, float x, float y) {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(x, y);
}
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 ld2(const __nv_bfloat16* p) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
}

// A ROWS x W tile on its way from global memory (rows `stride` elements apart, rows >= live read as zeros) through
// registers into shared memory as fp32 with leading dimension LD.  All loads of a tile are in flight together, and a
// caller may put work between get() and put().
template <typename IO, int ROWS, int W, int LD, int TH = NT>
struct Tile {
    static constexpr int kPer = 16 / (int)sizeof(IO), kChunks = W / kPer, kTotal = ROWS * kChunks;
    static constexpr int kN = (kTotal + TH - 1) / TH;
    uint4 r[kN];
    __device__ __forceinline__ void get(const IO* src, size_t stride, int live) {
#pragma unroll
        for (int i = 0; i < kN; ++i) {
            const int id = i * TH + threadIdx.x, row = id / kChunks, c = id % kChunks;
            r[i] = make_uint4(0, 0, 0, 0);
            if ((kTotal % TH == 0 || id < kTotal) && row < live)
                r[i] = *reinterpret_cast<const uint4*>(src + (size_t)row * stride + c * kPer);
        }
    }
    __device__ __forceinline__ void put(float* dst) const {
#pragma unroll
        for (int i = 0; i < kN; ++i) {
            const int id = i * TH + threadIdx.x, row = id / kChunks, c = id % kChunks;
            if (kTotal % TH != 0 && id >= kTotal) continue;
            float4* d = reinterpret_cast<float4*>(dst + row * LD + c * kPer);
            if (sizeof(IO) == 4) {
                d[0] = make_float4(__uint_as_float(r[i].x), __uint_as_float(r[i].y), __uint_as_float(r[i].z), __uint_as_float(r[i].w));
            } else {
                d[0] = make_float4(__uint_as_float(r[i].x << 16), __uint_as_float(r[i].x & 0xffff0000u),
                                   __uint_as_float(r[i].y << 16), __uint_as_float(r[i].y & 0xffff0000u));
                d[1] = make_float4(__uint_as_float(r[i].z << 16), __uint_as_float(r[i].z & 0xffff0000u),
                                   __uint_as_float(r[i].w << 16), __uint_as_float(r[i].w & 0xffff0000u));
            }
        }
    }
};
template <typename IO, int ROWS, int W, int LD>
__device__ __forceinline__ void load_tile(float* dst, const IO* src, size_t stride, int live) {
    Tile<IO, ROWS, W, LD> t;
    t.get(src, stride, live);
    t.put(dst);
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// M = (I + A)^-1 of a unit lower-triangular 64 x 64 matrix (A strictly lower, sA, untouched above its diagonal), into sM.
// The four 16 x 16 diagonal blocks are inverted by right-looking substitution, a column in the registers of a lane; then
// blocks are joined twice, M21 = -M22 (A21 M11), over all threads, with the inner product in sS.  The chain of dependent
// steps is 16 + 4 products long; a column per thread over all 64 rows took 30 us here.
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
    for (int S = 16; S <= 32; S *= 2) {                          // join pairs of S x S blocks
        const int pairs = C / (2 * S), quads = S * S / 4;        // four neighbouring columns per item
        for (int e = tid; e < pairs * quads; e += NT) {
            const int p = e / quads, r = (e % quads) / (S / 4), c = (e % (S / 4)) * 4, o = p * 2 * S;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
            for (int k = 0; k < S; ++k) {
                const float av = sA[(o + S + r) * LDC + o + k];
                const float4 b = *reinterpret_cast<const float4*>(sM + (o + k) * LDC + o + c);
                x.x = fmaf(av, b.x, x.x); x.y = fmaf(av, b.y, x.y); x.z = fmaf(av, b.z, x.z); x.w = fmaf(av, b.w, x.w);
            }
            *reinterpret_cast<float4*>(sS + (o + r) * LDI + c) = x;
        }
        __syncthreads();
        for (int e = tid; e < pairs * quads; e += NT) {
            const int p = e / quads, r = (e % quads) / (S / 4), c = (e % (S / 4)) * 4, o = p * 2 * S;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
            for (int k = 0; k < S; ++k) {
                const float av = -sM[(o + S + r) * LDC + o + S + k];
                const float4 b = *reinterpret_cast<const float4*>(sS + (o + k) * LDI + c);
                x.x = fmaf(av, b.x, x.x); x.y = fmaf(av, b.y, x.y); x.z = fmaf(av, b.z, x.z); x.w = fmaf(av, b.w, x.w);
            }
            *reinterpret_cast<float4*>(sM + (o + S + r) * LDC + o + c) = x;
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

// ---------------------------------------------------------------------------------------------
// K1: per chunk-head, state-independent part: g, P, W<-, U~ (and M for the backward).
template <int DK, int DV>
__global__ void __launch_bounds__(NT) k_prep(Ptrs p) {
    typedef float IO;
    extern __shared__ float sm[];
    constexpr int LK = DK + kPad, LV = DV + kPad, TI = kTerms<IO>;
    constexpr bool EX = TI == 2;
    float *sQ = sm, *sK = sQ + C * LK, *sV = sK + C * LK, *sA = sV + C * LV, *sM = sA + C * LDC;
    __shared__ __align__(16) float sg[C];
    __shared__ float sbeta[C], scq[C], sck[C], srq[C], srk[C];
    const int ch = blockIdx.x, n = ch % p.N, bh = ch / p.N, b = bh / p.H, hh = bh % p.H, H = p.H, tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh;   // token row of local r: row0 + r*H
    const size_t wrow0 = (size_t)bh * p.Tp + (size_t)n * C;           // workspace row of local r: wrow0 + r
    const int live = min(C, p.T - n * C);                             // tokens of this chunk inside the sequence
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    if (ch == 0 && tid == 0) *p.status = 0;
    {
        Tile<IO, C, DK, LK> tq, tk;
        Tile<IO, C, DV, LV> tv;
        tq.get((const IO*)p.q + row0 * DK, (size_t)H * DK, live);
        tk.get((const IO*)p.k + row0 * DK, (size_t)H * DK, live);
        tv.get((const IO*)p.v + row0 * DV, (size_t)H * DV, live);
        if (tid < C) {
            const size_t r = row0 + (size_t)tid * H;
            const bool in = tid < live;
            const float la = (in && p.alpha) ? log_gate(ld((const IO*)p.alpha, r), p.logits) : 0.f;
            const float be = in ? gate(ld((const IO*)p.beta, r), p.logits) : 0.f;
            const float lm = (in && p.lam) ? gate(ld((const IO*)p.lam, r), p.logits) : 0.f;
            scan64(la, sg);
            p.g[wrow0 + tid] = sg[tid];
            sbeta[tid] = be;
            scq[tid] = lm; sck[tid] = 1.f; srq[tid] = 1.f; srk[tid] = 1.f;
        }
        tq.put(sQ); tk.put(sK); tv.put(sV);
    }
    __syncthreads();
    if (p.rqk) {
        const size_t nrows = (size_t)p.B * H * p.Tp;
        for (int r = warp; r < C; r += NT / 32) {
            float sq = 0.f, sk = 0.f;
#pragma unroll
            for (int d = lane; d < DK; d += 32) {
                sq = fmaf(sQ[r * LK + d], sQ[r * LK + d], sq);
                sk = fmaf(sK[r * LK + d], sK[r * LK + d], sk);
            }
            sq = warp_sum(sq); sk = warp_sum(sk);
            if (lane == 0) {
                const float rq = 1.f / sqrtf(sq + kNormEps), rk = 1.f / sqrtf(sk + kNormEps);
                srq[r] = rq; srk[r] = rk;
                scq[r] *= rq; sck[r] = rk;
                p.rqk[wrow0 + r] = rq; p.rqk[nrows + wrow0 + r] = rk;
            }
        }
        __syncthreads();
    }
    // x_r = (1/|k_r|) k_r + (lambda_r / |q_r|) q_r; the stored rows stay as they are, exact in their storage type
    auto Xf = [&](int r, int d) { return fmaf(scq[r], sQ[r * LK + d], sck[r] * sK[r * LK + d]); };
    const int wm = (warp & 1) * 32, wn = warp >> 1;
    {
        float a1[2][2][4], a2[2][2][4];
        zero(a1); zero(a2);
        auto Kt = [&](int d, int i) { return sK[i * LK + d]; };
        wmm<2, 2, 2, TI, EX>(a1, wm, wn * 16, DK, Xf, Kt);
        wmm<2, 2, TI, TI, EX>(a2, wm, wn * 16, DK, [&](int r, int d) { return sQ[r * LK + d]; }, Kt);
        // A = strictLower(beta_r Gamma_ri (x_r . k_i)),  P = Gamma o (Q K^T), causal including the diagonal
        each(a1, wm, wn * 16, [&](int r, int i, float x, float y) {
            const float f = sbeta[r];
            x = i < r ? f * expf(sg[r] - sg[i]) * srk[i] * x : 0.f;
            y = i + 1 < r ? f * expf(sg[r] - sg[i + 1]) * srk[i + 1] * y : 0.f;
            st2(sA + r * LDC + i, x, y);
        });
        each(a2, wm, wn * 16, [&](int r, int i, float x, float y) {
            const float f = srq[r];
            x = i <= r ? f * expf(sg[r] - sg[i]) * srk[i] * x : 0.f;
            y = i + 1 <= r ? f * expf(sg[r] - sg[i + 1]) * srk[i + 1] * y : 0.f;
            st2((IO*)p.P + (wrow0 + r) * C + i, x, y);
        });
    }
    __syncthreads();
    float* sS = sM + C * LDC;
    invert_unit_lower(sA, sM, sS);
    for (int e = tid; e < C * C; e += NT) {                            // T = M diag(beta), over A
        const int r = e / C, i = e % C;
        const float m = sM[r * LDC + i];
        sA[r * LDC + i] = m * sbeta[i];
        if (p.save) p.M[wrow0 * C + e] = m;
    }
    if (tid < C) { const float gm = expf(sg[tid]); scq[tid] *= gm; sck[tid] *= gm; }     // X becomes diag(gamma) X
    __syncthreads();
    auto Tf = [&](int r, int i) { return sA[r * LDC + i]; };
    {
        float u[2][DV / 32][4];
        zero(u);
        wmm<2, DV / 32, 2, TI, EX>(u, wm, wn * (DV / 4), C, Tf, [&](int i, int j) { return sV[i * LV + j]; });
        each(u, wm, wn * (DV / 4), [&](int r, int j, float x, float y) { st2((IO*)p.U + (wrow0 + r) * DV + j, x, y); });
    }
    {
        float w[2][DK / 32][4];
        zero(w);
        wmm<2, DK / 32, 2, 2, EX>(w, wm, wn * (DK / 4), C, Tf, Xf);
        each(w, wm, wn * (DK / 4), [&](int r, int d, float x, float y) { st2((IO*)p.W + (wrow0 + r) * DK + d, x, y); });
    }
}

// The same for bf16 storage, on bf16 planes: X is never formed, X K^T and T diag(gamma) X are each a product with K and one
// with Q, their coefficients applied to the result or to T.  One set of planes holds T, T diag(gamma / |k|) and
// T diag(lambda gamma / |q|) in turn, over what the inverse needed; at d_k = d_v = 64 three CTAs fit an SM.
// 1024 chunks of 64 x 64: 72 us with tf32 halves and two CTAs, 56 so (d_k 128, d_v 64: 119 and 70), bound by the latency of its
// chain of small steps.
template <int DK, int DV>
struct PrepPlanes {
    typedef Planes<C, DK, 1> TQ;
    typedef Planes<C, DV, 1> TV;
    typedef Planes<C, C, 3> TC;
    static constexpr int kT = 2 * TQ::kBytes + TV::kBytes, kM = kT + TC::kBytes, kBytes = kM + C * LDC * 4, kCtas = kBytes <= 74 * 1024 ? 3 : 2;
    static_assert(C * (LDC + LDI) * 4 <= TC::kBytes, "A and the inverse's scratch");
};
template <int DK, int DV>
__global__ void __launch_bounds__(NT, PrepPlanes<DK, DV>::kCtas) k_prep_planes(Ptrs p) {
    extern __shared__ __align__(16) unsigned char smb[];
    typedef PrepPlanes<DK, DV> L;
    typedef __nv_bfloat16 IO;
    const typename L::TQ mQ(smb), mK(smb + L::TQ::kBytes);
    const typename L::TV mV(smb + 2 * L::TQ::kBytes);
    const typename L::TC mT(smb + L::kT);
    float *sA = reinterpret_cast<float*>(smb + L::kT), *sS = sA + C * LDC, *sM = reinterpret_cast<float*>(smb + L::kM);
    __shared__ __align__(16) float sg[C], sbeta[C], scq[C], sck[C], srq[C], srk[C];
    const int ch = blockIdx.x, n = ch % p.N, bh = ch / p.N, b = bh / p.H, hh = bh % p.H, H = p.H, tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh;
    const size_t wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
    const int live = min(C, p.T - n * C);
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    if (ch == 0 && tid == 0) *p.status = 0;
    mQ.template fetch<NT>((const IO*)p.q + row0 * DK, (size_t)H * DK, live);
    mK.template fetch<NT>((const IO*)p.k + row0 * DK, (size_t)H * DK, live);
    mV.template fetch<NT>((const IO*)p.v + row0 * DV, (size_t)H * DV, live);
    if (tid < C) {
        const size_t r = row0 + (size_t)tid * H;
        const bool in = tid < live;
        const float la = (in && p.alpha) ? log_gate(ld((const IO*)p.alpha, r), p.logits) : 0.f;
        const float be = in ? gate(ld((const IO*)p.beta, r), p.logits) : 0.f;
        const float lm = (in && p.lam) ? gate(ld((const IO*)p.lam, r), p.logits) : 0.f;
        scan64(la, sg);
        p.g[wrow0 + tid] = sg[tid];
        sbeta[tid] = be;
        scq[tid] = lm; sck[tid] = 1.f; srq[tid] = 1.f; srk[tid] = 1.f;
    }
    fetch_wait();
    __syncthreads();
    if (p.rqk) {
        const size_t nrows = (size_t)p.B * H * p.Tp;
        for (int r = warp; r < C; r += NT / 32) {
            float sq = 0.f, sk = 0.f;
#pragma unroll
            for (int d = 2 * lane; d < DK; d += 64) {
                const float2 q = mQ.ld2(r, d), k = mK.ld2(r, d);
                sq = fmaf(q.x, q.x, fmaf(q.y, q.y, sq));
                sk = fmaf(k.x, k.x, fmaf(k.y, k.y, sk));
            }
            sq = warp_sum(sq); sk = warp_sum(sk);
            if (lane == 0) {
                const float rq = 1.f / sqrtf(sq + kNormEps), rk = 1.f / sqrtf(sk + kNormEps);
                srq[r] = rq; srk[r] = rk;
                scq[r] *= rq; sck[r] = rk;
                p.rqk[wrow0 + r] = rq; p.rqk[nrows + wrow0 + r] = rk;
            }
        }
        __syncthreads();
    }
    const int wm = (warp & 1) * 32, wn = warp >> 1;
    {
        float kk[2][2][4], qk[2][2][4];
        zero(kk); zero(qk);
        pmm<false, false>(kk, mK, mK, wm, wn * 16, DK);
        pmm<false, false>(qk, mQ, mK, wm, wn * 16, DK);
        // A = strictLower(beta_r Gamma_ri (x_r . k_i)),  P = Gamma o (Q K^T), causal including the diagonal
        each2(kk, qk, wm, wn * 16, [&](int r, int i, float k0, float k1, float q0, float q1) {
            const float e0 = i <= r ? expf(sg[r] - sg[i]) * srk[i] : 0.f, e1 = i + 1 <= r ? expf(sg[r] - sg[i + 1]) * srk[i + 1] : 0.f;
            const float f = sbeta[r], cq = scq[r], ck = sck[r], rq = srq[r];
            st2(sA + r * LDC + i, i < r ? f * e0 * fmaf(ck, k0, cq * q0) : 0.f, i + 1 < r ? f * e1 * fmaf(ck, k1, cq * q1) : 0.f);
            st2((IO*)p.P + (wrow0 + r) * C + i, rq * e0 * q0, rq * e1 * q1);
        });
    }
    __syncthreads();
    invert_unit_lower(sA, sM, sS);
    // T diag(f) into the planes
    auto put_T = [&](auto f) {
#pragma unroll
        for (int e = tid * 4; e < C * C; e += NT * 4) {
            const int r = e / C, i = e % C;
            float4 m = *reinterpret_cast<const float4*>(sM + r * LDC + i);
            m.x *= f(i); m.y *= f(i + 1); m.z *= f(i + 2); m.w *= f(i + 3);
            mT.st4(r, i, m);
        }
        __syncthreads();
    };
    if (p.save)
#pragma unroll
        for (int e = tid * 4; e < C * C; e += NT * 4)
            *reinterpret_cast<float4*>(p.M + wrow0 * C + e) = *reinterpret_cast<const float4*>(sM + (e / C) * LDC + e % C);
    if (tid < C) { const float gm = expf(sg[tid]) * sbeta[tid]; scq[tid] *= gm; sck[tid] *= gm; }
    put_T([&](int i) { return sbeta[i]; });
    {
        float u[2][DV / 32][4];
        zero(u);
        pmm<false, true>(u, mT, mV, wm, wn * (DV / 4), C);
        each(u, wm, wn * (DV / 4), [&](int r, int j, float x, float y) { st2((IO*)p.U + (wrow0 + r) * DV + j, x, y); });
    }
    __syncthreads();
    float w[2][DK / 32][4];
    zero(w);
    put_T([&](int i) { return sck[i]; });
    pmm<false, true>(w, mT, mK, wm, wn * (DK / 4), C);
    __syncthreads();
    put_T([&](int i) { return scq[i]; });
    pmm<false, true>(w, mT, mQ, wm, wn * (DK / 4), C);
    each(w, wm, wn * (DK / 4), [&](int r, int d, float x, float y) { st2((IO*)p.W + (wrow0 + r) * DK + d, x, y); });
}

// ---------------------------------------------------------------------------------------------
// K2: forward state chain.  One CTA per (sequence, DS-column slice of d_v); columns of the state evolve independently,
// the chunks of a sequence are walked in order.  The next chunk's tiles are fetched into registers while the present
// chunk is worked on: a chunk costs its two dependent products and three barriers, not its loads.
template <int DK, int DS>
__global__ void __launch_bounds__(NT) k_chain_fwd(Ptrs p, int DV) {
    typedef float IO;
    constexpr int TH = NT;
    extern __shared__ float sm[];
    constexpr int LA = DK + 4, LB = DK + 8, LS = DS + 8, TI = kTerms<IO>, NS = DS / 8;
    // the two products of a phase take half of the warps each: 64 tokens x DS columns in 16 x 8 NH, DK x DS in 16 MU x 8 NU
    constexpr int HW = TH / 64, NH = NS / (HW / 4), MU = DK / 16 > HW ? DK / 16 / HW : 1, RU = DK / 16 / MU, NU = NS / (HW / RU);
    constexpr bool EX = TI == 2;
    float *sW = sm, *sQ = sW + C * LA, *sK = sQ + C * LA, *sP = sK + C * LB, *sU = sP + C * LDC, *sD = sU + C * LS,
          *sDs = sD + C * LS, *sh = sDs + C * LS;                     // sh: the state slice [DK][DS]
    __shared__ float sgq[C], sgk[C], sgC;
    const int H = p.H, nsl = DV / DS, j0 = (blockIdx.x % nsl) * DS, bh = blockIdx.x / nsl, b = bh / H, hh = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    for (int e = tid; e < DK * DS; e += TH)
        sh[(e / DS) * LS + e % DS] = p.h0 ? p.h0[((size_t)bh * DK + e / DS) * DV + j0 + e % DS] : 0.f;
    Tile<IO, C, DK, LA, TH> tw, tq;
    Tile<IO, C, DK, LB, TH> tk;
    Tile<IO, C, C, LDC, TH> tp;
    Tile<IO, C, DS, LS, TH> tu;
    float g = 0.f, gC = 0.f, rq = 1.f, rk = 1.f;
    const size_t nrows = (size_t)p.B * H * p.Tp;
    auto fetch = [&](int n) {
        const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh, wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
        const int live = min(C, p.T - n * C);
        tw.get((const IO*)p.W + wrow0 * DK, DK, C);
        tq.get((const IO*)p.q + row0 * DK, (size_t)H * DK, live);
        tk.get((const IO*)p.k + row0 * DK, (size_t)H * DK, live);
        tp.get((const IO*)p.P + wrow0 * C, C, C);
        tu.get((const IO*)p.U + wrow0 * DV + j0, DV, C);
        if (tid < C) {
            g = p.g[wrow0 + tid]; gC = p.g[wrow0 + C - 1];
            if (p.rqk) { rq = p.rqk[wrow0 + tid]; rk = p.rqk[nrows + wrow0 + tid]; }
        }
    };
    fetch(0);
    for (int n = 0; n < p.N; ++n) {
        const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh, wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
        const int live = min(C, p.T - n * C);
        tw.put(sW); tq.put(sQ); tk.put(sK); tp.put(sP); tu.put(sU);
        if (tid < C) { sgq[tid] = expf(g) * rq; sgk[tid] = expf(gC - g) * rk; if (tid == 0) sgC = expf(gC); }
        __syncthreads();
        if (n + 1 < p.N) fetch(n + 1);
        if (p.save) {
            float* dst = p.hs + ((size_t)bh * p.N + n) * DK * DV + j0;
            for (int e = tid * 4; e < DK * DS; e += TH * 4)
                *reinterpret_cast<float4*>(dst + (size_t)(e / DS) * DV + e % DS) =
                    *reinterpret_cast<const float4*>(sh + (e / DS) * LS + e % DS);
        }
        // first half of the warps: Delta = U~ - W<- h;  second: Q h, the inter-chunk part of the output, kept in registers
        float acc[1][NH][4];
        zero(acc);
        const int m0 = (warp & 3) * 16, n0 = (warp % HW / 4) * 8 * NH;
        auto hf = [&](int i, int j) { return sh[i * LS + j]; };
        if (warp < HW) {
            wmm<1, NH, TI, 2, EX>(acc, m0, n0, DK, [&](int r, int i) { return sW[r * LA + i]; }, hf);
            each(acc, m0, n0, [&](int r, int j, float x, float y) {
                x = sU[r * LS + j] - x; y = sU[r * LS + j + 1] - y;
                st2(sD + r * LS + j, x, y);
                st2(sDs + r * LS + j, x * sgk[r], y * sgk[r]);
                if (p.save) st2((IO*)p.D + (wrow0 + r) * DV + j0 + j, x, y);
            });
        } else {
            wmm<1, NH, TI, 2, EX>(acc, m0, n0, DK, [&](int r, int i) { return sQ[r * LA + i]; }, hf);
        }
        __syncthreads();
        if (warp >= HW) {
            // + P Delta, the intra-chunk part
            const int gq = (tid & 31) >> 2;
            const float s0 = sgq[m0 + gq], s1 = sgq[m0 + 8 + gq];
#pragma unroll
            for (int j = 0; j < NH; ++j) { acc[0][j][0] *= s0; acc[0][j][1] *= s0; acc[0][j][2] *= s1; acc[0][j][3] *= s1; }
            wmm<1, NH, TI, 2, EX>(acc, m0, n0, C, [&](int r, int s) { return sP[r * LDC + s]; },
                                  [&](int s, int j) { return sD[s * LS + j]; });
            each(acc, m0, n0, [&](int r, int j, float x, float y) {
                if (r < live) st2((IO*)p.o + (row0 + (size_t)r * H) * DV + j0 + j, x, y);
            });
        } else {
            // h <- gamma_C h + K^T (diag(gamma_C/gamma) Delta)
            float ha[MU][NU][4];
            zero(ha);
            const int i0 = (warp % RU) * 16 * MU, u0 = (warp / RU) * 8 * NU;
            wmm<MU, NU, TI, 2, EX>(ha, i0, u0, C, [&](int i, int r) { return sK[r * LB + i]; },
                                   [&](int r, int j) { return sDs[r * LS + j]; });
            each(ha, i0, u0, [&](int i, int j, float x, float y) {
                float* d = sh + i * LS + j;
                st2(d, fmaf(sgC, d[0], x), fmaf(sgC, d[1], y));
            });
        }
        __syncthreads();
    }
    if (p.hT)
        for (int e = tid; e < DK * DS; e += TH)
            p.hT[((size_t)bh * DK + e / DS) * DV + j0 + e % DS] = sh[(e / DS) * LS + e % DS];
}

// ---------------------------------------------------------------------------------------------
// K3: reverse state chain.  Carries dh (gradient w.r.t. the chunk's exit state) backwards:
//   dDelta = P^T dO + K-> dh ;   dh_in = gamma_C dh + (diag(gamma) Q)^T dO - W<-^T dDelta
// and leaves per chunk: dh (exit), dDelta, and two scalar partial sums the decay gradient needs.
template <int DK, int DS>
__global__ void __launch_bounds__(NT) k_chain_bwd(Ptrs p, int DV) {
    typedef float IO;
    constexpr int TH = NT;
    extern __shared__ float sm[];
    constexpr int LA = DK + 4, LB = DK + 8, LP = C + 8, LS = DS + 8, TI = kTerms<IO>, NS = DS / 8;
    // the two products of a phase take half of the warps each: 64 tokens x DS columns in 16 x 8 NH, DK x DS in 16 MU x 8 NU
    constexpr int HW = TH / 64, NH = NS / (HW / 4), MU = DK / 16 > HW ? DK / 16 / HW : 1, RU = DK / 16 / MU, NU = NS / (HW / RU);
    constexpr bool EX = TI == 2;
    float *sK = sm, *sQ = sK + C * LA, *sW = sQ + C * LB, *sP = sW + C * LB, *sO = sP + C * LP, *sOs = sO + C * LS,
          *sD = sOs + C * LS, *sdD = sD + C * LS, *sdh = sdD + C * LS;
    __shared__ float sgq[C], sgk[C], sgC, sred[TH / 32], skd[HW / 4][C];
    const int H = p.H, nsl = DV / DS, sl = blockIdx.x % nsl, j0 = sl * DS, bh = blockIdx.x / nsl, b = bh / H, hh = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5;
    const size_t nrows = (size_t)p.B * H * p.Tp, BHN = (size_t)p.B * H * p.N;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    for (int e = tid; e < DK * DS; e += TH)
        sdh[(e / DS) * LS + e % DS] = p.dhT ? p.dhT[((size_t)bh * DK + e / DS) * DV + j0 + e % DS] : 0.f;
    Tile<IO, C, DK, LA, TH> tk;
    Tile<IO, C, DK, LB, TH> tq, tw;
    Tile<IO, C, C, LP, TH> tp;
    Tile<IO, C, DS, LS, TH> to, td;
    float g = 0.f, gC = 0.f, rq = 1.f, rk = 1.f;
    auto fetch = [&](int n) {
        const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh, wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
        const int live = min(C, p.T - n * C);
        tk.get((const IO*)p.k + row0 * DK, (size_t)H * DK, live);
        tq.get((const IO*)p.q + row0 * DK, (size_t)H * DK, live);
        tw.get((const IO*)p.W + wrow0 * DK, DK, C);
        tp.get((const IO*)p.P + wrow0 * C, C, C);
        to.get((const IO*)p.dO + row0 * DV + j0, (size_t)H * DV, live);
        td.get((const IO*)p.D + wrow0 * DV + j0, DV, C);
        if (tid < C) {
            g = p.g[wrow0 + tid]; gC = p.g[wrow0 + C - 1];
            if (p.rqk) { rq = p.rqk[wrow0 + tid]; rk = p.rqk[nrows + wrow0 + tid]; }
        }
    };
    fetch(p.N - 1);
    for (int n = p.N - 1; n >= 0; --n) {
        const size_t wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
        tk.put(sK); tq.put(sQ); tw.put(sW); tp.put(sP); to.put(sO); td.put(sD);
        if (tid < C) { sgq[tid] = expf(g) * rq; sgk[tid] = expf(gC - g) * rk; if (tid == 0) sgC = expf(gC); }
        __syncthreads();
        if (n > 0) fetch(n - 1);
        // keep dh of this chunk's exit state; partial <dh, h_entry>_F over this slice
        {
            float* dst = p.dhs + ((size_t)bh * p.N + n) * DK * DV + j0;
            const float* hsrc = p.hs + ((size_t)bh * p.N + n) * DK * DV + j0;
            float part = 0.f;
#pragma unroll 2
            for (int e = tid * 4; e < DK * DS; e += TH * 4) {
                const size_t off = (size_t)(e / DS) * DV + e % DS;
                const float4 x = *reinterpret_cast<const float4*>(sdh + (e / DS) * LS + e % DS);
                const float4 y = *reinterpret_cast<const float4*>(hsrc + off);
                *reinterpret_cast<float4*>(dst + off) = x;
                part = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, part))));
            }
            part = warp_sum(part);
            if ((tid & 31) == 0) sred[warp] = part;
            for (int e = tid; e < C * DS; e += TH) {             // diag(gamma / |q|) dO, the operand of Q^T
                const int r = e / DS, j = e % DS;
                sOs[r * LS + j] = sO[r * LS + j] * sgq[r];
            }
        }
        __syncthreads();
        if (tid == 0) {
            float tot = 0.f;
            for (int w = 0; w < TH / 32; ++w) tot += sred[w];
            p.dhh[(size_t)sl * BHN + (size_t)bh * p.N + n] = tot;
        }
        float ha[MU][NU][4];
        zero(ha);
        const int hw = warp % HW, i0 = (hw % RU) * 16 * MU, u0 = (hw / RU) * 8 * NU;
        if (warp < HW) {
            // dDelta = diag(gamma_C/gamma) K dh + P^T dO, 16 tokens per warp; row sums of the first term times Delta
            float acc[1][NH][4];
            zero(acc);
            const int m0 = (warp & 3) * 16, n0 = (warp >> 2) * 8 * NH;
            wmm<1, NH, TI, 2, EX>(acc, m0, n0, DK, [&](int s, int i) { return sK[s * LA + i]; },
                                  [&](int i, int j) { return sdh[i * LS + j]; });
            const int gq = (tid & 31) >> 2;
            const float s0 = sgk[m0 + gq], s1 = sgk[m0 + 8 + gq];
#pragma unroll
            for (int j = 0; j < NH; ++j) { acc[0][j][0] *= s0; acc[0][j][1] *= s0; acc[0][j][2] *= s1; acc[0][j][3] *= s1; }
            row_sums(acc, m0, n0, skd[warp >> 2],
                     [&](int s, int j, float x, float y) { return fmaf(x, sD[s * LS + j], y * sD[s * LS + j + 1]); });
            wmm<1, NH, TI, TI, EX>(acc, m0, n0, C, [&](int s, int r) { return sP[r * LP + s]; },
                                   [&](int r, int j) { return sO[r * LS + j]; });
            each(acc, m0, n0, [&](int s, int j, float x, float y) {
                st2(sdD + s * LS + j, -x, -y);
                st2((IO*)p.dD + (wrow0 + s) * DV + j0 + j, x, y);
            });
        } else {
            wmm<MU, NU, TI, 2, EX>(ha, i0, u0, C, [&](int i, int r) { return sQ[r * LB + i]; },
                                   [&](int r, int j) { return sOs[r * LS + j]; });
        }
        __syncthreads();
        if (warp >= HW) {
            wmm<MU, NU, TI, 2, EX>(ha, i0, u0, C, [&](int i, int r) { return sW[r * LB + i]; },
                                   [&](int r, int j) { return sdD[r * LS + j]; });
            each(ha, i0, u0, [&](int i, int j, float x, float y) {
                float* d = sdh + i * LS + j;
                st2(d, fmaf(sgC, d[0], x), fmaf(sgC, d[1], y));
            });
        } else if (tid < C) {
            float kd = skd[0][tid];
            if (HW > 4) kd += skd[HW / 4 - 1][tid];
            p.kdhd[(size_t)sl * nrows + wrow0 + tid] = kd;
        }
        __syncthreads();
    }
    if (p.dh0)
        for (int e = tid; e < DK * DS; e += TH)
            p.dh0[((size_t)bh * DK + e / DS) * DV + j0 + e % DS] = sdh[(e / DS) * LS + e % DS];
}

// The state chains for bf16 storage, on bf16 planes.  Every warp takes a 16 x 16 tile of the 64 x DS products and DK/4 x 16 of
// the state, which it keeps in fp32 in its registers (planes of it are what the others read).  A chunk is two phases and two
// barriers; the tiles of one phase arrive while the other is worked on, those of the first two phases ahead.  Slices of 32
// columns and d_k = 64 let two CTAs share an SM.  B4 T1024 H16 d_k = d_v = 64: 73 and 85 us with tf32 halves, 50 and 56 so (3 us a
// chunk, of which the tensor unit works a quarter: the rest is the latency of two dependent products and two barriers).
template <int DK, int DS>
struct ChainPlanes {
    typedef Planes<C, DK, 1> TA;
    typedef Planes<2 * C, DK, 1> TA2;      // W<- above Q
    typedef Planes<C, C, 1> TP;
    typedef Planes<C, DS, 1> TO;
    typedef Planes<C, DS, 3> TD;
    typedef Planes<DK, DS, 3> TS;
    static constexpr int kThreads = 8 * DS, kFwd = 2 * TA2::kBytes + TA::kBytes + TP::kBytes + TS::kBytes + 2 * TD::kBytes,
                         kBwd = 2 * (TA::kBytes + TP::kBytes + TO::kBytes) + 2 * TA::kBytes + TS::kBytes + 2 * TD::kBytes;
};
template <int N> __device__ __forceinline__ void fetch_wait_but() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void fetch_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// decay factors of a chunk's tokens, thread t < 64 token t: fetched a chunk ahead, written before the barrier that ends the present one
struct ChainCoef {
    float g = 0.f, gC = 0.f, rq = 1.f, rk = 1.f;
    __device__ __forceinline__ void get(const Ptrs& p, size_t wrow0, size_t nrows) {
        if (threadIdx.x >= C) return;
        g = p.g[wrow0 + threadIdx.x]; gC = p.g[wrow0 + C - 1];
        if (p.rqk) { rq = p.rqk[wrow0 + threadIdx.x]; rk = p.rqk[nrows + wrow0 + threadIdx.x]; }
    }
    __device__ __forceinline__ void put(float* gq, float* gk, float* gc) const {
        if (threadIdx.x >= C) return;
        gq[threadIdx.x] = expf(g) * rq; gk[threadIdx.x] = expf(gC - g) * rk;
        if (threadIdx.x == 0) *gc = expf(gC);
    }
};
template <int DK, int DS>
__global__ void __launch_bounds__(8 * DS) k_chain_fwd_planes(Ptrs p, int DV) {
    extern __shared__ __align__(16) unsigned char smb[];
    typedef ChainPlanes<DK, DS> L;
    typedef __nv_bfloat16 IO;
    constexpr int TH = L::kThreads, MU = DK / 64;
    typename L::TA2 mWQ(smb);
    const typename L::TA mK(smb + 2 * L::TA2::kBytes);
    const typename L::TP mP(smb + 2 * L::TA2::kBytes + L::TA::kBytes);
    const typename L::TS mS(smb + 2 * L::TA2::kBytes + L::TA::kBytes + L::TP::kBytes);
    const typename L::TD mD(smb + L::kFwd - 2 * L::TD::kBytes), mDs(smb + L::kFwd - L::TD::kBytes);
    __shared__ float sgq[2][C], sgk[2][C], sgC[2];
    const int H = p.H, nsl = DV / DS, j0 = (blockIdx.x % nsl) * DS, bh = blockIdx.x / nsl, b = bh / H, hh = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5, g = (tid & 31) >> 2, t = tid & 3;
    const int wm = (warp & 3) * 16, wn = (warp >> 2) * 16, si = (warp & 3) * 16 * MU;
    const size_t nrows = (size_t)p.B * H * p.Tp, row0 = (size_t)b * p.T * H + hh, wrow0 = (size_t)bh * p.Tp;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    auto fetch1 = [&](int n) {         // W<- and Q, read in the first phase of chunk n
        const typename L::TA w(smb + (n & 1) * L::TA2::kBytes), q(smb + (n & 1) * L::TA2::kBytes + L::TA::kBytes);
        w.template fetch<TH>((const IO*)p.W + (wrow0 + (size_t)n * C) * DK, DK, C);
        q.template fetch<TH>((const IO*)p.q + (row0 + (size_t)n * C * H) * DK, (size_t)H * DK, min(C, p.T - n * C));
    };
    auto fetch2 = [&](int n) {         // K and P, read in the second
        mK.template fetch<TH>((const IO*)p.k + (row0 + (size_t)n * C * H) * DK, (size_t)H * DK, min(C, p.T - n * C));
        mP.template fetch<TH>((const IO*)p.P + (wrow0 + (size_t)n * C) * C, C, C);
    };
    uint32_t u[2][2];                  // U~ at this thread's elements
    auto fetch_u = [&](int n) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                u[h][j] = *reinterpret_cast<const uint32_t*>((const IO*)p.U + (wrow0 + (size_t)n * C + wm + 8 * h + g) * DV + j0 + wn + 8 * j + 2 * t);
    };
    ChainCoef cf;
    fetch1(0);
    fetch_commit();
    cf.get(p, wrow0, nrows);
    fetch_u(0);
    float hst[MU][2][4];
    zero(hst);
    auto state_at = [&](float* base, int i, int j) { return reinterpret_cast<float2*>(base + (size_t)i * DV + j0 + j); };
    if (p.h0) each(hst, si, wn, [&](int i, int j, float& x, float& y) {
        const float2 v = *state_at(const_cast<float*>(p.h0) + (size_t)bh * DK * DV, i, j);
        x = v.x; y = v.y;
    });
    each(hst, si, wn, [&](int i, int j, float x, float y) {
        mS.st2(i, j, x, y);
        if (p.save) *state_at(p.hs + (size_t)bh * p.N * DK * DV, i, j) = make_float2(x, y);
    });
    cf.put(sgq[0], sgk[0], sgC);
    for (int n = 0; n < p.N; ++n) {
        const int bf = n & 1, live = min(C, p.T - n * C);
        const bool more = n + 1 < p.N;
        fetch_wait();
        __syncthreads();
        fetch2(n);
        fetch_commit();
        if (more) { fetch1(n + 1); cf.get(p, wrow0 + (size_t)(n + 1) * C, nrows); }
        fetch_commit();
        // Delta = U~ - W<- h, and Q h, the inter-chunk part of the output
        float a[2][2][4], o[1][2][4];
        zero(a); zero(o);
        mWQ.p = reinterpret_cast<IO*>(smb + bf * L::TA2::kBytes);
        pmm<false, true, 2, 2, typename L::TA2, typename L::TS, C>(a, mWQ, mS, wm, wn, DK);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int r = wm + 8 * h + g, c = wn + 8 * j + 2 * t;
                const float x = __uint_as_float(u[h][j] << 16) - a[0][j][2 * h], y = __uint_as_float(u[h][j] & 0xffff0000u) - a[0][j][2 * h + 1];
                mD.st2(r, c, x, y);
                mDs.st2(r, c, x * sgk[bf][r], y * sgk[bf][r]);
                if (p.save) st2((IO*)p.D + (wrow0 + (size_t)n * C + r) * DV + j0 + c, x, y);
            }
        if (more) fetch_u(n + 1);
        fetch_wait_but<1>();
        __syncthreads();
        // h <- gamma_C h + K^T (diag(gamma_C/gamma) Delta)
        {
            float s[MU][2][4];
            zero(s);
            pmm<true, true>(s, mK, mDs, si, wn, C);
            const float gc = sgC[bf];
            each2(hst, s, si, wn, [&](int i, int j, float& x, float& y, float dx, float dy) {
                x = fmaf(gc, x, dx); y = fmaf(gc, y, dy);
                mS.st2(i, j, x, y);
                if (p.save && more) *state_at(p.hs + ((size_t)bh * p.N + n + 1) * DK * DV, i, j) = make_float2(x, y);
            });
        }
        // o = diag(gamma) Q h + P Delta
        pmm<false, true>(o, mP, mD, wm, wn, C);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int r = wm + 8 * h + g;
                const float f = sgq[bf][r];
                if (r < live) st2((IO*)p.o + (row0 + (size_t)(n * C + r) * H) * DV + j0 + wn + 8 * j + 2 * t,
                                  fmaf(f, a[1][j][2 * h], o[0][j][2 * h]), fmaf(f, a[1][j][2 * h + 1], o[0][j][2 * h + 1]));
            }
        if (more) cf.put(sgq[bf ^ 1], sgk[bf ^ 1], sgC + (bf ^ 1));
    }
    if (p.hT) each(hst, si, wn, [&](int i, int j, float x, float y) { *state_at(p.hT + (size_t)bh * DK * DV, i, j) = make_float2(x, y); });
}

template <int DK, int DS>
__global__ void __launch_bounds__(8 * DS) k_chain_bwd_planes(Ptrs p, int DV) {
    extern __shared__ __align__(16) unsigned char smb[];
    typedef ChainPlanes<DK, DS> L;
    typedef __nv_bfloat16 IO;
    constexpr int TH = L::kThreads, MU = DK / 64, kSet = L::TA::kBytes + L::TP::kBytes + L::TO::kBytes;
    const typename L::TA mQ(smb + 2 * kSet), mW(smb + 2 * kSet + L::TA::kBytes);
    const typename L::TS mS(smb + 2 * kSet + 2 * L::TA::kBytes);
    const typename L::TD mdD(smb + L::kBwd - 2 * L::TD::kBytes), mOs(smb + L::kBwd - L::TD::kBytes);
    __shared__ float sgq[2][C], sgk[2][C], sgC[2], sred[TH / 32], skd[DS / 16][C];
    const int H = p.H, nsl = DV / DS, sl = blockIdx.x % nsl, j0 = sl * DS, bh = blockIdx.x / nsl, b = bh / H, hh = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5, g = (tid & 31) >> 2, t = tid & 3;
    const int wm = (warp & 3) * 16, wn = (warp >> 2) * 16, si = (warp & 3) * 16 * MU;
    const size_t nrows = (size_t)p.B * H * p.Tp, BHN = (size_t)p.B * H * p.N, row0 = (size_t)b * p.T * H + hh, wrow0 = (size_t)bh * p.Tp;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    auto fetch1 = [&](int n) {         // K, P and dO, read in the first phase of chunk n
        unsigned char* s = smb + (n & 1) * kSet;
        const typename L::TA k(s);
        const typename L::TP pm(s + L::TA::kBytes);
        const typename L::TO o(s + L::TA::kBytes + L::TP::kBytes);
        const int live = min(C, p.T - n * C);
        k.template fetch<TH>((const IO*)p.k + (row0 + (size_t)n * C * H) * DK, (size_t)H * DK, live);
        pm.template fetch<TH>((const IO*)p.P + (wrow0 + (size_t)n * C) * C, C, C);
        o.template fetch<TH>((const IO*)p.dO + (row0 + (size_t)n * C * H) * DV + j0, (size_t)H * DV, live);
    };
    auto fetch2 = [&](int n) {         // Q and W<-, read in the second
        mQ.template fetch<TH>((const IO*)p.q + (row0 + (size_t)n * C * H) * DK, (size_t)H * DK, min(C, p.T - n * C));
        mW.template fetch<TH>((const IO*)p.W + (wrow0 + (size_t)n * C) * DK, DK, C);
    };
    uint32_t d[2][2];                  // Delta and the entry state at this thread's elements
    float2 hin[MU][2][2];
    auto state_at = [&](float* base, int i, int j) { return reinterpret_cast<float2*>(base + (size_t)i * DV + j0 + j); };
    auto fetch_d = [&](int n) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                d[h][j] = *reinterpret_cast<const uint32_t*>((const IO*)p.D + (wrow0 + (size_t)n * C + wm + 8 * h + g) * DV + j0 + wn + 8 * j + 2 * t);
#pragma unroll
                for (int m = 0; m < MU; ++m) hin[m][h][j] = *state_at(p.hs + ((size_t)bh * p.N + n) * DK * DV, si + 16 * m + 8 * h + g, wn + 8 * j + 2 * t);
            }
    };
    ChainCoef cf;
    fetch1(p.N - 1);
    fetch_commit();
    cf.get(p, wrow0 + (size_t)(p.N - 1) * C, nrows);
    fetch_d(p.N - 1);
    float dst[MU][2][4];
    zero(dst);
    if (p.dhT) each(dst, si, wn, [&](int i, int j, float& x, float& y) {
        const float2 v = *state_at(const_cast<float*>(p.dhT) + (size_t)bh * DK * DV, i, j);
        x = v.x; y = v.y;
    });
    each(dst, si, wn, [&](int i, int j, float x, float y) { mS.st2(i, j, x, y); });
    cf.put(sgq[(p.N - 1) & 1], sgk[(p.N - 1) & 1], sgC + ((p.N - 1) & 1));
    for (int n = p.N - 1; n >= 0; --n) {
        const int bf = n & 1;
        fetch_wait();
        __syncthreads();
        fetch2(n);
        fetch_commit();
        if (n > 0) { fetch1(n - 1); cf.get(p, wrow0 + (size_t)(n - 1) * C, nrows); }
        fetch_commit();
        const typename L::TA mK(smb + bf * kSet);
        const typename L::TP mP(smb + bf * kSet + L::TA::kBytes);
        const typename L::TO mO(smb + bf * kSet + L::TA::kBytes + L::TP::kBytes);
        // dDelta = diag(gamma_C/gamma) K dh + P^T dO; row sums of the first term times Delta
        {
            float a[1][2][4], c[1][2][4];
            zero(a); zero(c);
            pmm<false, true>(a, mK, mS, wm, wn, DK);
            each(a, wm, wn, [&](int r, int, float& x, float& y) { x *= sgk[bf][r]; y *= sgk[bf][r]; });
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float s = 0.f;
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    s += fmaf(a[0][j][2 * h], __uint_as_float(d[h][j] << 16), a[0][j][2 * h + 1] * __uint_as_float(d[h][j] & 0xffff0000u));
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                if (t == 0) skd[warp >> 2][wm + 8 * h + g] = s;
            }
            pmm<true, true>(c, mP, mO, wm, wn, C);
            each2(a, c, wm, wn, [&](int s, int j, float x, float y, float u, float v) {
                x += u; y += v;
                mdD.st2(s, j, -x, -y);
                st2((IO*)p.dD + (wrow0 + (size_t)n * C + s) * DV + j0 + j, x, y);
                const float2 o = mO.ld2(s, j);                   // diag(gamma / |q|) dO, the operand of Q^T
                mOs.st2(s, j, o.x * sgq[bf][s], o.y * sgq[bf][s]);
            });
        }
        // keep dh of this chunk's exit state; partial <dh, h_entry>_F over this slice
        float part = 0.f;
#pragma unroll
        for (int m = 0; m < MU; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float2 v = make_float2(dst[m][j][2 * h], dst[m][j][2 * h + 1]);
                    *state_at(p.dhs + ((size_t)bh * p.N + n) * DK * DV, si + 16 * m + 8 * h + g, wn + 8 * j + 2 * t) = v;
                    part = fmaf(v.x, hin[m][h][j].x, fmaf(v.y, hin[m][h][j].y, part));
                }
        part = warp_sum(part);
        if ((tid & 31) == 0) sred[warp] = part;
        if (n > 0) fetch_d(n - 1);
        fetch_wait_but<1>();
        __syncthreads();
        if (tid < C) {
            float kd = 0.f;
#pragma unroll
            for (int w = 0; w < DS / 16; ++w) kd += skd[w][tid];
            p.kdhd[(size_t)sl * nrows + wrow0 + (size_t)n * C + tid] = kd;
        }
        if (tid == TH - 1) {
            float tot = 0.f;
            for (int w = 0; w < TH / 32; ++w) tot += sred[w];
            p.dhh[(size_t)sl * BHN + (size_t)bh * p.N + n] = tot;
        }
        // dh <- gamma_C dh + (diag(gamma) Q)^T dO - W<-^T dDelta
        {
            float s[MU][2][4];
            zero(s);
            pmm<true, true>(s, mQ, mOs, si, wn, C);
            pmm<true, true>(s, mW, mdD, si, wn, C);
            const float gc = sgC[bf];
            each2(dst, s, si, wn, [&](int i, int j, float& x, float& y, float dx, float dy) {
                x = fmaf(gc, x, dx); y = fmaf(gc, y, dy);
                mS.st2(i, j, x, y);
            });
        }
        if (n > 0) cf.put(sgq[bf ^ 1], sgk[bf ^ 1], sgC + (bf ^ 1));
    }
    if (p.dh0) each(dst, si, wn, [&](int i, int j, float x, float y) { *state_at(p.dh0 + (size_t)bh * DK * DV, i, j) = make_float2(x, y); });
}

// ---------------------------------------------------------------------------------------------
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

// ---------------------------------------------------------------------------------------------
// K4: chunk-parallel part of the backward: dq, dk, dv, dbeta, dlambda, dalpha.  The 64 x d_k results dX, dq and dk stay in
// registers from their first product to their store (each warp owns the same 32 x d_k/4 tile of all three); four tile
// slots of shared memory take turns holding Q, K, h, dh, dO, Delta, dDelta, dW<- and V.
template <int DK, int DV>
struct BwdSmem {
    static constexpr int LT = (DK > DV ? DK : DV) + kPad;
    static constexpr int kSlot = C * LT;
    static constexpr size_t bytes = sizeof(float) * (4 * kSlot + 5 * C * LDC);
};
template <int DK, int DV>
__global__ void __launch_bounds__(NT) k_chunk_bwd(Ptrs p) {
    typedef float IO;
    extern __shared__ float sm[];
    constexpr int LT = BwdSmem<DK, DV>::LT, LH = DV + kPad, TI = kTerms<IO>, kSlot = BwdSmem<DK, DV>::kSlot, NK = DK / 32;
    constexpr bool EX = TI == 2;
    static_assert(DK * LH <= 2 * kSlot, "a state fits two slots");
    float *s0 = sm, *s1 = s0 + kSlot, *s2 = s1 + kSlot, *s3 = s2 + kSlot;
    float* m0 = s3 + kSlot;          // X K^T          -> dA o A
    float* m1 = m0 + C * LDC;        // M
    float* m2 = m1 + C * LDC;        // dT             -> dXK
    float* m3 = m2 + C * LDC;        // dP o Gamma
    float* m4 = m3 + C * LDC;        // dP o P         -> dT diag(beta) M^T
    __shared__ float sbeta[C], slam[C], salpha[C], sg[C], sgam[C], segc[C], srq[C], srk[C], scq[C];
    __shared__ float sdg[C], skd[C], part[4][C], prow[5][4][C];   // prow: row sums by warp column: dP o P, t1, t2, d beta, d lambda
    __shared__ float pcol[4][C];
    const int H = p.H, ch = blockIdx.x, n = ch % p.N, bh = ch / p.N, b = bh / H, hh = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5;
    const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh, wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
    const size_t nrows = (size_t)p.B * H * p.Tp;
    const int live = min(C, p.T - n * C);
    const float* hs = p.hs + ((size_t)bh * p.N + n) * DK * DV;
    const float* dhs = p.dhs + ((size_t)bh * p.N + n) * DK * DV;
    const int wm = (warp & 1) * 32, wn = warp >> 1, nc = wn * 16, nk = wn * (DK / 4);

    Tile<IO, C, DK, LT> tq, tk;
    Tile<IO, C, DV, LT> tv;
    Tile<float, DK, DV, LH> th;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    // ---- coefficients, Q, K, M; dO and Delta ----------------------------------------------------
    tq.get((const IO*)p.q + row0 * DK, (size_t)H * DK, live);
    tk.get((const IO*)p.k + row0 * DK, (size_t)H * DK, live);
    if (tid < C) {
        const size_t r = row0 + (size_t)tid * H;
        const bool in = tid < live;
        const float g = p.g[wrow0 + tid], gC = p.g[wrow0 + C - 1];
        sbeta[tid] = in ? gate(ld((const IO*)p.beta, r), p.logits) : 0.f;
        const float lm = (in && p.lam) ? gate(ld((const IO*)p.lam, r), p.logits) : 0.f;
        salpha[tid] = (in && p.alpha) ? gate(ld((const IO*)p.alpha, r), p.logits) : 1.f;
        const float rq = p.rqk ? p.rqk[wrow0 + tid] : 1.f, rk = p.rqk ? p.rqk[nrows + wrow0 + tid] : 1.f;
        slam[tid] = lm; sg[tid] = g; sgam[tid] = expf(g); segc[tid] = expf(gC - g);
        srq[tid] = rq; srk[tid] = rk; scq[tid] = lm * rq;
    }
    tq.put(s0); tk.put(s1);
    load_tile<float, C, C, LDC>(m1, p.M + wrow0 * C, C, C);
    load_tile<IO, C, DV, LT>(s2, (const IO*)p.dO + row0 * DV, (size_t)H * DV, live);
    load_tile<IO, C, DV, LT>(s3, (const IO*)p.D + wrow0 * DV, DV, C);
    __syncthreads();
    auto Qf = [&](int r, int d) { return s0[r * LT + d]; };                                       // as stored
    auto Kf = [&](int r, int d) { return s1[r * LT + d]; };
    auto Xf = [&](int r, int d) { return fmaf(scq[r], s0[r * LT + d], srk[r] * s1[r * LT + d]); };
    th.get(dhs, DV, DK);
    // ---- X K^T, and dP with its uses: dP o P (row and column sums) and dP o Gamma -------------------
    {
        float a[2][2][4];
        zero(a);
        wmm<2, 2, 2, TI, EX>(a, wm, nc, DK, Xf, [&](int d, int i) { return s1[i * LT + d]; });
        each(a, wm, nc, [&](int r, int i, float x, float y) { st2(m0 + r * LDC + i, x * srk[i], y * srk[i + 1]); });
        zero(a);
        wmm<2, 2, TI, TI, EX>(a, wm, nc, DV, [&](int r, int j) { return s2[r * LT + j]; }, [&](int j, int s) { return s3[s * LT + j]; });
        each(a, wm, nc, [&](int r, int s, float& x, float& y) {
            const float2 pv = ld2((const IO*)p.P + (wrow0 + r) * C + s);
            const float d0 = s <= r ? x : 0.f, d1 = s + 1 <= r ? y : 0.f;
            st2(m3 + r * LDC + s, s <= r ? d0 * expf(sg[r] - sg[s]) : 0.f, s + 1 <= r ? d1 * expf(sg[r] - sg[s + 1]) : 0.f);
            x = d0 * pv.x; y = d1 * pv.y;
            st2(m4 + r * LDC + s, x, y);
        });
        row_sums(a, wm, nc, prow[0][wn], [&](int, int, float x, float y) { return x + y; });
    }
    __syncthreads();                                            // Q and K have been read
    // ---- dk <- diag(gamma_C/gamma) Delta dh^T,  dq <- diag(gamma) dO h^T,  dW<- = -dDelta h^T -------
    float aK[2][NK][4], aQ[2][NK][4], aX[2][NK][4];
    th.put(s0);
    th.get(hs, DV, DK);
    {
        const int col = tid & 63, q4 = tid >> 6;                // column sums of dP o P
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < 16; ++r) s += m4[(q4 * 16 + r) * LDC + col];
        pcol[q4][col] = s;
    }
    __syncthreads();
    zero(aK);
    wmm<2, NK, TI, 2, EX>(aK, wm, nk, DV, [&](int r, int j) { return s3[r * LT + j]; }, [&](int j, int i) { return s0[i * LH + j]; });
    __syncthreads();                                            // dh and Delta have been read
    th.put(s0);
    tv.get((const IO*)p.dD + wrow0 * DV, DV, C);
    tv.put(s3);
    __syncthreads();
    tv.get((const IO*)p.v + row0 * DV, (size_t)H * DV, live);
    zero(aQ); zero(aX);
    wmm<2, NK, TI, 2, EX>(aQ, wm, nk, DV, [&](int r, int j) { return s2[r * LT + j]; }, [&](int j, int i) { return s0[i * LH + j]; });
    wmm<2, NK, TI, 2, EX>(aX, wm, nk, DV, [&](int r, int j) { return s3[r * LT + j]; }, [&](int j, int i) { return s0[i * LH + j]; });
    __syncthreads();                                            // h and dO have been read
    each(aX, wm, nk, [&](int r, int i, float x, float y) { st2(s2 + r * LT + i, -x, -y); });       // dW<-
    tv.put(s0);
    each(aK, wm, nk, [&](int r, int, float& x, float& y) { x *= segc[r]; y *= segc[r]; });
    each(aQ, wm, nk, [&](int r, int, float& x, float& y) { x *= sgam[r]; y *= sgam[r]; });
    __syncthreads();
    tq.get((const IO*)p.q + row0 * DK, (size_t)H * DK, live);
    tk.get((const IO*)p.k + row0 * DK, (size_t)H * DK, live);
    // ---- dT = dDelta V^T + dW<- (gamma X)^T;  dV = T^T dDelta -------------------------------------
    float aT[2][2][4];
    zero(aT);
    wmm<2, 2, TI, TI, EX>(aT, wm, nc, DV, [&](int r, int j) { return s3[r * LT + j]; }, [&](int j, int s) { return s0[s * LT + j]; });
    {
        float a[2][DV / 32][4];
        zero(a);
        wmm<2, DV / 32, 2, TI, EX>(a, wm, wn * (DV / 4), C, [&](int s, int r) { return m1[r * LDC + s]; },
                               [&](int r, int j) { return s3[r * LT + j]; });
        each(a, wm, wn * (DV / 4), [&](int s, int j, float x, float y) {
            if (s < live) st2((IO*)p.dv_ + (row0 + (size_t)s * H) * DV + j, sbeta[s] * x, sbeta[s] * y);
        });
    }
    __syncthreads();                                            // V has been read
    tq.put(s0); tk.put(s1);
    __syncthreads();
    {
        float a[2][2][4];
        zero(a);
        wmm<2, 2, 2, 2, EX>(a, wm, nc, DK, [&](int r, int i) { return s2[r * LT + i]; }, [&](int i, int s) { return Xf(s, i); });
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int s = nc + 8 * j + 2 * (tid & 3);
                const float ga = sgam[s], gb = sgam[s + 1];
                aT[i][j][0] = fmaf(ga, a[i][j][0], aT[i][j][0]); aT[i][j][1] = fmaf(gb, a[i][j][1], aT[i][j][1]);
                aT[i][j][2] = fmaf(ga, a[i][j][2], aT[i][j][2]); aT[i][j][3] = fmaf(gb, a[i][j][3], aT[i][j][3]);
            }
        each(aT, wm, nc, [&](int r, int s, float x, float y) { st2(m2 + r * LDC + s, x, y); });
    }
    // ---- dX <- diag(gamma) T^T dW<-; the row sums t1 = <dQ1, Q>, t2 = <dXg, gamma X> -----------------
    zero(aX);
    wmm<2, NK, 2, 2, EX>(aX, wm, nk, C, [&](int s, int r) { return m1[r * LDC + s]; }, [&](int r, int i) { return s2[r * LT + i]; });
    each(aX, wm, nk, [&](int s, int, float& x, float& y) { const float f = sbeta[s] * sgam[s]; x *= f; y *= f; });
    row_sums(aX, wm, nk, prow[2][wn], [&](int r, int i, float x, float y) { return fmaf(x, Xf(r, i), y * Xf(r, i + 1)); });
    row_sums(aQ, wm, nk, prow[1][wn],
             [&](int r, int i, float x, float y) { return srq[r] * fmaf(x, Qf(r, i), y * Qf(r, i + 1)); });
    __syncthreads();                                            // dT is complete
    // ---- d beta from T;  dA = -strictLower(M^T (dT diag(beta) M^T)) --------------------------------
    {
        const int col = tid & 63, q4 = tid >> 6;
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < 16; ++r) s = fmaf(m2[(q4 * 16 + r) * LDC + col], m1[(q4 * 16 + r) * LDC + col], s);
        part[q4][col] = s;
        float a[2][2][4];
        zero(a);
        wmm<2, 2, 2, 2, EX>(a, wm, nc, C, [&](int r, int u) { return m2[r * LDC + u] * sbeta[u]; }, [&](int u, int s2_) { return m1[s2_ * LDC + u]; });
        each(a, wm, nc, [&](int r, int s_, float x, float y) { st2(m4 + r * LDC + s_, x, y); });
    }
    __syncthreads();
    {
        float a[2][2][4];
        zero(a);
        wmm<2, 2, 2, 2, EX>(a, wm, nc, C, [&](int r, int u) { return m1[u * LDC + r]; }, [&](int u, int s) { return m4[u * LDC + s]; });
        // its uses: d beta (row sums), dA o A (column sums), d(X K^T)
        each(a, wm, nc, [&](int r, int s, float& x, float& y) {
            const float e0 = s < r ? -x * expf(sg[r] - sg[s]) : 0.f, e1 = s + 1 < r ? -y * expf(sg[r] - sg[s + 1]) : 0.f;
            const float be = sbeta[r];
            float* xk = m0 + r * LDC + s;
            x = e0 * xk[0]; y = e1 * xk[1];
            st2(xk, be * x, be * y);
            st2(m2 + r * LDC + s, be * e0, be * e1);
        });
        row_sums(a, wm, nc, prow[3][wn], [&](int, int, float x, float y) { return x + y; });
    }
    __syncthreads();
    // ---- dX += dXK K;  dk += dXK^T X + dPG^T Q + dX;  dq += dPG K + lambda dX ----------------------
    wmm<2, NK, 2, 2, EX>(aX, wm, nk, C, [&](int r, int s) { return m2[r * LDC + s]; }, [&](int s, int d) { return srk[s] * Kf(s, d); });
    row_sums(aX, wm, nk, prow[4][wn],
             [&](int r, int i, float x, float y) { return srq[r] * fmaf(x, Qf(r, i), y * Qf(r, i + 1)); });
    wmm<2, NK, 2, 2, EX>(aK, wm, nk, C, [&](int i, int r) { return m2[r * LDC + i]; }, Xf);
    wmm<2, NK, 2, 2, EX>(aK, wm, nk, C, [&](int i, int r) { return m3[r * LDC + i]; }, [&](int r, int d) { return srq[r] * Qf(r, d); });
    wmm<2, NK, 2, 2, EX>(aQ, wm, nk, C, [&](int r, int s) { return m3[r * LDC + s]; }, [&](int s, int d) { return srk[s] * Kf(s, d); });
    {
        const int g = (tid & 31) >> 2;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < NK; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    aK[i][j][e] += aX[i][j][e];
                    aQ[i][j][e] = fmaf(slam[wm + 16 * i + 8 * (e >> 1) + g], aX[i][j][e], aQ[i][j][e]);
                }
    }
    float db1 = 0.f;
    if (tid < C) db1 = part[0][tid] + part[1][tid] + part[2][tid] + part[3][tid];      // column sums of dT o M
    __syncthreads();
    if (p.rqk) {
        // through the normalisation: dx = r (dx^ - x^ <x^, dx^>)
        row_sums(aQ, wm, nk, part[wn], [&](int r, int i, float x, float y) { return srq[r] * fmaf(x, Qf(r, i), y * Qf(r, i + 1)); });
        __syncthreads();
        each(aQ, wm, nk, [&](int r, int i, float& x, float& y) {
            const float c = part[0][r] + part[1][r] + part[2][r] + part[3][r], f = srq[r];
            x = f * fmaf(-c * f, Qf(r, i), x); y = f * fmaf(-c * f, Qf(r, i + 1), y);
        });
        __syncthreads();
        row_sums(aK, wm, nk, part[wn], [&](int r, int i, float x, float y) { return srk[r] * fmaf(x, Kf(r, i), y * Kf(r, i + 1)); });
        __syncthreads();
        each(aK, wm, nk, [&](int r, int i, float& x, float& y) {
            const float c = part[0][r] + part[1][r] + part[2][r] + part[3][r], f = srk[r];
            x = f * fmaf(-c * f, Kf(r, i), x); y = f * fmaf(-c * f, Kf(r, i + 1), y);
        });
    }
    each(aK, wm, nk, [&](int r, int i, float x, float y) { if (r < live) st2((IO*)p.dk_ + (row0 + (size_t)r * H) * DK + i, x, y); });
    each(aQ, wm, nk, [&](int r, int i, float x, float y) { if (r < live) st2((IO*)p.dq + (row0 + (size_t)r * H) * DK + i, x, y); });
    __syncthreads();
    {
        const int col = tid & 63, q4 = tid >> 6;
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < 16; ++r) s += m0[(q4 * 16 + r) * LDC + col];           // column sums of dA o A
        part[q4][col] = s;
    }
    __syncthreads();
    token_gradients<IO>(p, prow, pcol, part, db1, sbeta, slam, salpha, sgam, sdg, skd, row0, wrow0, bh, n, live);
}

// The same for bf16 storage, on bf16 planes.  X is never formed: a product with it is one with K and one with Q, which are
// exact in one plane, their coefficients applied to the result or to the other operand.  One slot of shared memory holds dh,
// h, dW<- and dT M^T in turn; M takes Delta's place, dT that of dO, dDelta and V.  So two CTAs fit an SM at d_k = d_v = 64: one
// computes while the other loads or waits at a barrier, and a warp's 32 x 16 tile reads 1.5 operand pieces per 16 x 16 x 16
// product, half of what 16 x 16 tiles of 16 warps would.  B4 T1024 H16 d_k = d_v = 64: 208 us with tf32 halves, 150 with 16
// warps and one CTA, 122 so.
template <int DK, int DV>
struct BwdPlanes {
    typedef Planes<C, DK, 1> TQ;
    typedef Planes<C, DV, 1> TV;
    typedef Planes<DK, DV, 3> TS;
    typedef Planes<C, DK, 3> TW;
    typedef Planes<C, C, 3> TC;
    static constexpr int kV = 2 * TQ::kBytes, kS = kV + 3 * TV::kBytes, kM = kS + (TS::kBytes > TW::kBytes ? TS::kBytes : TW::kBytes),
                         kBytes = kM + TC::kBytes;
    static_assert(TV::kBytes <= TC::kBytes && TC::kBytes <= 3 * TV::kBytes && TC::kBytes <= kM - kS && kV + 3 * TC::kBytes <= kBytes, "reused room");
    // where two CTAs fit: 32 x 16 tiles of 8 warps; one CTA: 16 warps hide more (d 128 and 64: 202 against 207 us, normalised 217, 233)
    static constexpr int kCtas = kBytes <= 100 * 1024 ? 2 : 1, kThreads = kCtas == 2 ? 256 : 512;
};
template <int DK, int DV>
__global__ void __launch_bounds__(BwdPlanes<DK, DV>::kThreads, BwdPlanes<DK, DV>::kCtas) k_chunk_bwd_planes(Ptrs p) {
    extern __shared__ __align__(16) unsigned char smb[];
    typedef BwdPlanes<DK, DV> L;
    typedef __nv_bfloat16 IO;
    constexpr int TH = L::kThreads, MT = 512 / TH, NK = DK / 32, NV = DV / 32, WR = 4 / MT;      // WR x 4 warps of 16 MT rows
    const typename L::TQ mQ(smb), mK(smb + L::TQ::kBytes);
    const typename L::TV mO(smb + L::kV), mdD(smb + L::kV + L::TV::kBytes), mV(smb + L::kV + 2 * L::TV::kBytes), mD(smb + L::kM);
    const typename L::TS mS(smb + L::kS);
    const typename L::TW mW(smb + L::kS);
    const typename L::TC mM(smb + L::kM), mT(smb + L::kV), m4(smb + L::kS);
    __shared__ float sbeta[C], slam[C], salpha[C], sg[C], sgam[C], segc[C], srq[C], srk[C], scq[C];
    __shared__ float sdg[C], skd[C], part[4][C], prow[5][4][C];   // prow: row sums by warp column: dP o P, t1, t2, d beta, d lambda
    __shared__ float pcol[3][WR][C];                              // column sums by warp row: dP o P, dT o M, dA o A
    const int H = p.H, ch = blockIdx.x, n = ch % p.N, bh = ch / p.N, b = bh / H, hh = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh, wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
    const size_t nrows = (size_t)p.B * H * p.Tp;
    const int live = min(C, p.T - n * C);
    const int wr = warp % WR, wm = wr * 16 * MT, wn = warp / WR, nc = wn * 16, nk = wn * (DK / 4), nv = wn * (DV / 4);
    // sums over this warp's rows of each of its 16 columns, to dst[column]
    auto col_sums = [&](float (&a)[MT][2][4], float* dst) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float s = 0.f;
#pragma unroll
                for (int i = 0; i < MT; ++i) s += a[i][j][e] + a[i][j][e + 2];
                s += __shfl_xor_sync(0xffffffffu, s, 4);
                s += __shfl_xor_sync(0xffffffffu, s, 8);
                s += __shfl_xor_sync(0xffffffffu, s, 16);
                if (lane < 4) dst[nc + 8 * j + 2 * lane + e] = s;
            }
    };
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    // ---- everything that the chunk reads, but the entry state, in flight together ----------------
    mQ.template fetch<TH>((const IO*)p.q + row0 * DK, (size_t)H * DK, live);
    mK.template fetch<TH>((const IO*)p.k + row0 * DK, (size_t)H * DK, live);
    mO.template fetch<TH>((const IO*)p.dO + row0 * DV, (size_t)H * DV, live);
    mD.template fetch<TH>((const IO*)p.D + wrow0 * DV, DV, C);
    mdD.template fetch<TH>((const IO*)p.dD + wrow0 * DV, DV, C);
    mV.template fetch<TH>((const IO*)p.v + row0 * DV, (size_t)H * DV, live);
    FloatTile<DK, DV, TH> th;
    FloatTile<C, C, TH> tm;
    th.get(p.dhs + ((size_t)bh * p.N + n) * DK * DV);
    {
        if (tid < C) {
            const size_t r = row0 + (size_t)tid * H;
            const bool in = tid < live;
            const float g = p.g[wrow0 + tid], gC = p.g[wrow0 + C - 1];
            sbeta[tid] = in ? gate(ld((const IO*)p.beta, r), p.logits) : 0.f;
            const float lm = (in && p.lam) ? gate(ld((const IO*)p.lam, r), p.logits) : 0.f;
            salpha[tid] = (in && p.alpha) ? gate(ld((const IO*)p.alpha, r), p.logits) : 1.f;
            const float rq = p.rqk ? p.rqk[wrow0 + tid] : 1.f, rk = p.rqk ? p.rqk[nrows + wrow0 + tid] : 1.f;
            slam[tid] = lm; sg[tid] = g; sgam[tid] = expf(g); segc[tid] = expf(gC - g);
            srq[tid] = rq; srk[tid] = rk; scq[tid] = lm * rq;
        }
    }
    th.put(mS);
    th.get(p.hs + ((size_t)bh * p.N + n) * DK * DV);
    tm.get(p.M + wrow0 * C);
    fetch_wait();
    __syncthreads();
    // ---- dP with its uses: dP o P (row and column sums), dP o Gamma;  dk <- diag(gamma_C/gamma) Delta dh^T ----
    float a3[MT][2][4], aK[MT][NK][4], aQ[MT][NK][4], aX[MT][NK][4];
    zero(a3); zero(aK); zero(aQ); zero(aX);
    pmm<false, false>(a3, mO, mD, wm, nc, DV);
    {
        float a[MT][2][4];
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int r = wm + 16 * i + 8 * h + (lane >> 2), s = nc + 8 * j + 2 * (lane & 3);
                    float *d = a3[i][j] + 2 * h, *o = a[i][j] + 2 * h;
                    const float2 pv = ld2((const IO*)p.P + (wrow0 + r) * C + s);
                    const float d0 = s <= r ? d[0] : 0.f, d1 = s + 1 <= r ? d[1] : 0.f;
                    o[0] = d0 * pv.x; o[1] = d1 * pv.y;
                    d[0] = s <= r ? d0 * expf(sg[r] - sg[s]) : 0.f;
                    d[1] = s + 1 <= r ? d1 * expf(sg[r] - sg[s + 1]) : 0.f;
                }
        col_sums(a, pcol[0][wr]);
        row_sums(a, wm, nc, prow[0][wn], [&](int, int, float x, float y) { return x + y; });
    }
    pmm<false, false>(aK, mD, mS, wm, nk, DV);
    each(aK, wm, nk, [&](int r, int, float& x, float& y) { x *= segc[r]; y *= segc[r]; });
    __syncthreads();                                            // dh and Delta have been read
    th.put(mS);
    tm.put(mM);
    __syncthreads();
    // ---- dq <- diag(gamma) dO h^T;  dW<- = -dDelta h^T;  dT = dDelta V^T + ...;  dV = T^T dDelta ------------
    float aT[MT][2][4];
    zero(aT);
    pmm<false, false>(aQ, mO, mS, wm, nk, DV);
    pmm<false, false>(aX, mdD, mS, wm, nk, DV);
    pmm<false, false>(aT, mdD, mV, wm, nc, DV);
    {
        float a[MT][NV][4];
        zero(a);
        pmm<true, true>(a, mM, mdD, wm, nv, C);
        each(a, wm, nv, [&](int s, int j, float x, float y) {
            if (s < live) st2((IO*)p.dv_ + (row0 + (size_t)s * H) * DV + j, sbeta[s] * x, sbeta[s] * y);
        });
    }
    each(aQ, wm, nk, [&](int r, int, float& x, float& y) { x *= sgam[r]; y *= sgam[r]; });
    auto qsum = [&](int r, int i, float x, float y) { const float2 q = mQ.ld2(r, i); return srq[r] * fmaf(x, q.x, y * q.y); };
    auto ksum = [&](int r, int i, float x, float y) { const float2 k = mK.ld2(r, i); return srk[r] * fmaf(x, k.x, y * k.y); };
    row_sums(aQ, wm, nk, prow[1][wn], qsum);                    // t1 = <dQ1, Q>
    __syncthreads();                                            // h, dO, dDelta and V have been read
    each(aX, wm, nk, [&](int r, int i, float x, float y) { mW.st2(r, i, -x, -y); });
    __syncthreads();
    // ---- ... + dW<- (gamma X)^T;  d beta from T;  dX <- diag(gamma) T^T dW<-;  t2 = <dXg, gamma X> ----------
    {
        float a[MT][2][4];
        zero(a);
        pmm<false, false>(a, mW, mK, wm, nc, DK);
        each2(aT, a, wm, nc, [&](int, int s, float& x, float& y, float u, float v) {
            x = fmaf(sgam[s] * srk[s], u, x); y = fmaf(sgam[s + 1] * srk[s + 1], v, y);
        });
        zero(a);
        pmm<false, false>(a, mW, mQ, wm, nc, DK);
        each2(aT, a, wm, nc, [&](int, int s, float& x, float& y, float u, float v) {
            x = fmaf(sgam[s] * scq[s], u, x); y = fmaf(sgam[s + 1] * scq[s + 1], v, y);
        });
        each(aT, wm, nc, [&](int r, int s, float& x, float& y) {
            const float2 m = mM.ld2(r, s);
            mT.st2(r, s, x * sbeta[s], y * sbeta[s + 1]);
            x *= m.x; y *= m.y;
        });
        col_sums(aT, pcol[1][wr]);
    }
    zero(aX);
    pmm<true, true>(aX, mM, mW, wm, nk, C);
    each(aX, wm, nk, [&](int s, int, float& x, float& y) { const float f = sbeta[s] * sgam[s]; x *= f; y *= f; });
    row_sums(aX, wm, nk, prow[2][wn], [&](int r, int i, float x, float y) {
        const float2 k = mK.ld2(r, i), q = mQ.ld2(r, i);
        return fmaf(x, fmaf(scq[r], q.x, srk[r] * k.x), y * fmaf(scq[r], q.y, srk[r] * k.y));
    });
    __syncthreads();                                            // dT diag(beta) is complete
    // ---- dA = -strictLower(M^T (dT diag(beta) M^T)) -------------------------------------------------
    {
        float a[MT][2][4];
        zero(a);
        pmm<false, false>(a, mT, mM, wm, nc, C);
        each(a, wm, nc, [&](int r, int s, float x, float y) { m4.st2(r, s, x, y); });
    }
    __syncthreads();
    {
        float a[MT][2][4], x[MT][2][4];
        zero(a); zero(x);
        pmm<true, true>(a, mM, m4, wm, nc, C);
        pmm<false, false>(x, mQ, mK, wm, nc, DK);               // X K^T
        each(x, wm, nc, [&](int r, int, float& u, float& v) { u *= scq[r]; v *= scq[r]; });
        {
            float y[MT][2][4];
            zero(y);
            pmm<false, false>(y, mK, mK, wm, nc, DK);
            each2(x, y, wm, nc, [&](int r, int s, float& u, float& v, float k0, float k1) {
                u = srk[s] * fmaf(srk[r], k0, u); v = srk[s + 1] * fmaf(srk[r], k1, v);
            });
        }
        __syncthreads();                                        // M and dT M^T have been read: dX K^T and dP o Gamma over them
        // the uses of dA: d beta (row sums), dA o A (column sums), d(X K^T)
        const typename L::TC e1(smb + L::kV), e2(smb + L::kV + L::TC::kBytes), e3(smb + L::kV + 2 * L::TC::kBytes);
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int r = wm + 16 * i + 8 * h + (lane >> 2), s = nc + 8 * j + 2 * (lane & 3);
                    const float be = sbeta[r], cq = scq[r], rq = srq[r];
                    float d[2], *f = a3[i][j] + 2 * h;
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float& v = a[i][j][2 * h + e];
                        float& w = x[i][j][2 * h + e];
                        const float u = s + e < r ? -v * expf(sg[r] - sg[s + e]) : 0.f;
                        v = u * w;
                        w = be * v;
                        d[e] = be * u;
                    }
                    e1.st2(r, s, d[0] * srk[s], d[1] * srk[s + 1]);
                    e2.st2(r, s, f[0] * srk[s], f[1] * srk[s + 1]);
                    e3.st2(r, s, fmaf(cq, d[0], rq * f[0]), fmaf(cq, d[1], rq * f[1]));
                }
        row_sums(a, wm, nc, prow[3][wn], [&](int, int, float u, float v) { return u + v; });
        col_sums(x, pcol[2][wr]);
        __syncthreads();
        // ---- dX += dXK K;  dk += dXK^T X + dPG^T Q + dX;  dq += dPG K + lambda dX ----------------------
        pmm<false, true>(aX, e1, mK, wm, nk, C);
        row_sums(aX, wm, nk, prow[4][wn], qsum);
        pmm<false, true>(aQ, e2, mK, wm, nk, C);
        pmm<true, true>(aK, e3, mQ, wm, nk, C);
        if (p.rqk) {                                            // dXK scaled by row instead of by column
            __syncthreads();
            each(a, wm, nc, [&](int r, int s, float, float) {
                const float2 d = e1.ld2(r, s);
                e1.st2(r, s, d.x * (srk[r] / srk[s]), d.y * (srk[r] / srk[s + 1]));
            });
            __syncthreads();
        }
        pmm<true, true>(aK, e1, mK, wm, nk, C);
    }
    each2(aQ, aX, wm, nk, [&](int r, int, float& x, float& y, float u, float v) { x = fmaf(slam[r], u, x); y = fmaf(slam[r], v, y); });
    each2(aK, aX, wm, nk, [&](int, int, float& x, float& y, float u, float v) { x += u; y += v; });
    if (p.rqk) {
        // through the normalisation: dx = r (dx^ - x^ <x^, dx^>)
        row_sums(aQ, wm, nk, part[wn], qsum);
        __syncthreads();
        each(aQ, wm, nk, [&](int r, int i, float& x, float& y) {
            const float c = part[0][r] + part[1][r] + part[2][r] + part[3][r], f = srq[r];
            const float2 q = mQ.ld2(r, i);
            x = f * fmaf(-c * f, q.x, x); y = f * fmaf(-c * f, q.y, y);
        });
        __syncthreads();
        row_sums(aK, wm, nk, part[wn], ksum);
        __syncthreads();
        each(aK, wm, nk, [&](int r, int i, float& x, float& y) {
            const float c = part[0][r] + part[1][r] + part[2][r] + part[3][r], f = srk[r];
            const float2 k = mK.ld2(r, i);
            x = f * fmaf(-c * f, k.x, x); y = f * fmaf(-c * f, k.y, y);
        });
    }
    each(aK, wm, nk, [&](int r, int i, float x, float y) { if (r < live) st2((IO*)p.dk_ + (row0 + (size_t)r * H) * DK + i, x, y); });
    each(aQ, wm, nk, [&](int r, int i, float x, float y) { if (r < live) st2((IO*)p.dq + (row0 + (size_t)r * H) * DK + i, x, y); });
    __syncthreads();
    float db1 = 0.f;
    if (tid < C) {
#pragma unroll
        for (int c = 0; c < WR; ++c) db1 += pcol[1][c][tid];
    }
    token_gradients<IO>(p, prow, pcol[0], pcol[2], db1, sbeta, slam, salpha, sgam, sdg, skd, row0, wrow0, bh, n, live);
}

Ptrs make_ptrs(const ChunkArgs& a) {
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

// Small grids, where the gap between two kernels is a tenth of the time (31 -> 28 us for two sequences of 256 tokens), are
// launched while the kernel before them drains.  Larger ones are not: CTAs that come early take the SMs that are free first
// instead of one each, which cost 15 us on 128 chunks of 128 x 128 and 40 where two chains fit an SM.
template <class K, class... Args>
cudaError_t launch(K kern, int grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaError_t e = set_max_smem_once(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
    if (grid <= 64) return launch_overlapped(kern, dim3((unsigned)grid), dim3(threads), smem, stream, args...);
    kern<<<grid, threads, smem, stream>>>(args...);
    return cudaGetLastError();
}

template <typename IO, int DK, int DV>
cudaError_t prep_for(const ChunkArgs& a, const Ptrs& p) {
    const int grid = a.s.B * a.s.H * p.N;
    if constexpr (sizeof(IO) == 2) {
        return launch(k_prep_planes<DK, DV>, grid, NT, PrepPlanes<DK, DV>::kBytes, a.stream, p);
    } else {
        constexpr size_t smem = sizeof(float) * (2 * C * (DK + kPad) + C * (DV + kPad) + 2 * C * LDC + C * LDI);
        return launch(k_prep<DK, DV>, grid, NT, smem, a.stream, p);
    }
}
template <typename IO, int DK, int DS>
cudaError_t chain_fwd_for(const ChunkArgs& a, const Ptrs& p) {
    const int grid = a.s.B * a.s.H * (a.s.dv / DS);
    if constexpr (sizeof(IO) == 2) {
        typedef ChainPlanes<DK, DS> L;
        return launch(k_chain_fwd_planes<DK, DS>, grid, L::kThreads, L::kFwd, a.stream, p, a.s.dv);
    } else {
        constexpr size_t smem = sizeof(float) * (2 * C * (DK + 4) + C * (DK + 8) + C * LDC + (3 * C + DK) * (DS + 8));
        return launch(k_chain_fwd<DK, DS>, grid, NT, smem, a.stream, p, a.s.dv);
    }
}
template <typename IO, int DK, int DS>
cudaError_t chain_bwd_for(const ChunkArgs& a, const Ptrs& p) {
    const int grid = a.s.B * a.s.H * (a.s.dv / DS);
    if constexpr (sizeof(IO) == 2) {
        typedef ChainPlanes<DK, DS> L;
        return launch(k_chain_bwd_planes<DK, DS>, grid, L::kThreads, L::kBwd, a.stream, p, a.s.dv);
    } else {
        constexpr size_t smem = sizeof(float) * (C * (DK + 4) + 2 * C * (DK + 8) + C * (C + 8) + (4 * C + DK) * (DS + 8));
        return launch(k_chain_bwd<DK, DS>, grid, NT, smem, a.stream, p, a.s.dv);
    }
}
template <typename IO, int DK, int DV>
cudaError_t chunk_bwd_for(const ChunkArgs& a, const Ptrs& p) {
    if constexpr (sizeof(IO) == 2) {
        return launch(k_chunk_bwd_planes<DK, DV>, a.s.B * a.s.H * p.N, BwdPlanes<DK, DV>::kThreads, BwdPlanes<DK, DV>::kBytes, a.stream, p);
    } else {
        return launch(k_chunk_bwd<DK, DV>, a.s.B * a.s.H * p.N, NT, BwdSmem<DK, DV>::bytes, a.stream, p);
    }
}

typedef __nv_bfloat16 bf16;

}  // namespace

// d_v columns that one CTA of the state chains owns: narrow slices while they are what it takes to put a CTA on most of
// the SMs, because a chain's time is its dependent steps; wider ones, which read W<-, Q, K and P fewer times, beyond.
int split_slice(const qd_shape& s) { return (long long)s.B * s.H * (s.dv / 32) >= 120 ? 32 : 16; }

#define QD_BY_DIMS(fn, ...)                                                                     \
    (s.dtype == QD_F32 ? (s.dk == 128 ? (s.dv == 128 ? fn<float, 128, 128>(__VA_ARGS__) : fn<float, 128, 64>(__VA_ARGS__)) \
                                      : (s.dv == 128 ? fn<float, 64, 128>(__VA_ARGS__) : fn<float, 64, 64>(__VA_ARGS__)))  \
                       : (s.dk == 128 ? fn<bf16, 128, 64>(__VA_ARGS__)   /* 128 x 128: the tcgen05 kernels */                \
                                      : (s.dv == 128 ? fn<bf16, 64, 128>(__VA_ARGS__) : fn<bf16, 64, 64>(__VA_ARGS__))))
#define QD_BY_SLICE(fn, ...)                                                                    \
    (s.dtype == QD_F32 ? (s.dk == 128 ? (a.L.slice == 32 ? fn<float, 128, 32>(__VA_ARGS__) : fn<float, 128, 16>(__VA_ARGS__)) \
                                      : (a.L.slice == 32 ? fn<float, 64, 32>(__VA_ARGS__) : fn<float, 64, 16>(__VA_ARGS__)))  \
                       : (s.dk == 128 ? (a.L.slice == 32 ? fn<bf16, 128, 32>(__VA_ARGS__) : fn<bf16, 128, 16>(__VA_ARGS__))   \
                                      : (a.L.slice == 32 ? fn<bf16, 64, 32>(__VA_ARGS__) : fn<bf16, 64, 16>(__VA_ARGS__))))

cudaError_t split_prep(const ChunkArgs& a) {
    const qd_shape& s = a.s;
    const Ptrs p = make_ptrs(a);
    return QD_BY_DIMS(prep_for, a, p);
}
cudaError_t split_chain_fwd(const ChunkArgs& a) {
    const qd_shape& s = a.s;
    const Ptrs p = make_ptrs(a);
    return QD_BY_SLICE(chain_fwd_for, a, p);
}
cudaError_t split_chain_bwd(const ChunkArgs& a) {
    const qd_shape& s = a.s;
    const Ptrs p = make_ptrs(a);
    return QD_BY_SLICE(chain_bwd_for, a, p);
}
cudaError_t split_chunk_bwd(const ChunkArgs& a) {
    const qd_shape& s = a.s;
    const Ptrs p = make_ptrs(a);
    return QD_BY_DIMS(chunk_bwd_for, a, p);
}

}  // namespace qd
