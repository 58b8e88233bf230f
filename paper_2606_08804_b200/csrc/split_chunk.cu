// Chunkwise Q-Delta forward and backward with fp32-accurate products on the warp-level tensor instructions: fp32 storage.
//
// Arithmetic.  A product of two fp32 matrices is three m16n8k8 tf32 products of their 11-bit halves, x = hi + lo, both
// halves rounded: hi hi + hi lo + lo hi, accumulated in fp32 (the dropped lo lo term is below 2^-22 of the product).
// Measured on a B200: m16n8k8 runs at 276 TFLOP/s, i.e. 92 as three products, against 68 for packed fp32 FMAs and 39 for
// scalar ones; the difference that counts more is operand traffic, 16 shared-memory loads for 24 instructions of 1024
// multiply-adds here.  Operands live in shared memory as fp32 tiles with padded rows; each kernel reads every global
// operand once.
#include "split_common.cuh"

namespace qd {

// the same path for bf16 storage, split_bf16.cu
cudaError_t split_bf16_prep(const ChunkArgs& a);
cudaError_t split_bf16_chain_fwd(const ChunkArgs& a);
cudaError_t split_bf16_chain_bwd(const ChunkArgs& a);
cudaError_t split_bf16_chunk_bwd(const ChunkArgs& a);

namespace {

constexpr int kPad = 4;            // of a d-wide tile: rows g, columns t of a fragment fall on banks 4 g + t

// ---- tiles --------------------------------------------------------------------------------------------------------
// A ROWS x W tile on its way from global memory (rows `stride` elements apart, rows >= live read as zeros) through
// registers into shared memory with leading dimension LD.  All loads of a tile are in flight together, and a
// caller may put work between get() and put().
template <int ROWS, int W, int LD>
struct Tile {
    static constexpr int kPer = 4, kChunks = W / kPer, kTotal = ROWS * kChunks;
    static constexpr int kN = (kTotal + NT - 1) / NT;
    float4 r[kN];
    __device__ __forceinline__ void get(const float* src, size_t stride, int live) {
#pragma unroll
        for (int i = 0; i < kN; ++i) {
            const int id = i * NT + threadIdx.x, row = id / kChunks, c = id % kChunks;
            r[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if ((kTotal % NT == 0 || id < kTotal) && row < live)
                r[i] = *reinterpret_cast<const float4*>(src + (size_t)row * stride + c * kPer);
        }
    }
    __device__ __forceinline__ void put(float* dst) const {
#pragma unroll
        for (int i = 0; i < kN; ++i) {
            const int id = i * NT + threadIdx.x, row = id / kChunks, c = id % kChunks;
            if (kTotal % NT != 0 && id >= kTotal) continue;
            *reinterpret_cast<float4*>(dst + row * LD + c * kPer) = r[i];
        }
    }
};
template <int ROWS, int W, int LD>
__device__ __forceinline__ void load_tile(float* dst, const float* src, size_t stride, int live) {
    Tile<ROWS, W, LD> t;
    t.get(src, stride, live);
    t.put(dst);
}

// The same asynchronously, by the threads that load (number `me` of kLoaders).
template <int ROWS, int W, int LD>
__device__ __forceinline__ void fetch_tile(float* dst, const float* src, size_t stride, int live, int me) {
    constexpr int kChunks = W / 4, kTotal = ROWS * kChunks;
#pragma unroll 8
    for (int id = me; id < kTotal; id += kLoaders) {
        const int row = id / kChunks, c = id % kChunks * 4;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sm100::smem_u32(dst + row * LD + c)),
                     "l"(src + (row < live ? (size_t)row * stride : 0) + c), "r"(row < live ? 16 : 0) : "memory");
    }
}
__device__ __forceinline__ void fetched() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---------------------------------------------------------------------------------------------
// K1: per chunk-head, state-independent part: g, P, W<-, U~ (and M for the backward).
template <int DK, int DV>
__global__ void __launch_bounds__(NT) k_prep(Ptrs p) {
    extern __shared__ __align__(16) float sm[];
    constexpr int LK = DK + kPad, LV = DV + kPad;
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
        Tile<C, DK, LK> tq, tk;
        Tile<C, DV, LV> tv;
        tq.get((const float*)p.q + row0 * DK, (size_t)H * DK, live);
        tk.get((const float*)p.k + row0 * DK, (size_t)H * DK, live);
        tv.get((const float*)p.v + row0 * DV, (size_t)H * DV, live);
        if (tid < C) {
            const size_t r = row0 + (size_t)tid * H;
            const bool in = tid < live;
            const float la = (in && p.alpha) ? log_gate(ld((const float*)p.alpha, r), p.logits) : 0.f;
            const float be = in ? gate(ld((const float*)p.beta, r), p.logits) : 0.f;
            const float lm = (in && p.lam) ? gate(ld((const float*)p.lam, r), p.logits) : 0.f;
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
    const int wm = ((warp ^ (warp >> 2)) & 1) * 32, wn = warp >> 1;      // both halves of the rows on every scheduler
    {
        float a1[2][2][4], a2[2][2][4];
        zero(a1); zero(a2);
        auto Kt = [&](int d, int i) { return sK[i * LK + d]; };
        if (wn * 16 < wm + 32) {                                // not above the diagonal
            wmm<2, 2>(a1, wm, wn * 16, DK, Xf, Kt);
            wmm<2, 2>(a2, wm, wn * 16, DK, [&](int r, int d) { return sQ[r * LK + d]; }, Kt);
        }
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
            st2((float*)p.P + (wrow0 + r) * C + i, x, y);
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
        wmm<2, DV / 32>(u, wm, wn * (DV / 4), wm + 32, Tf, [&](int i, int j) { return sV[i * LV + j]; });
        each(u, wm, wn * (DV / 4), [&](int r, int j, float x, float y) { st2((float*)p.U + (wrow0 + r) * DV + j, x, y); });
    }
    {
        float w[2][DK / 32][4];
        zero(w);
        wmm<2, DK / 32>(w, wm, wn * (DK / 4), wm + 32, Tf, Xf);
        each(w, wm, wn * (DK / 4), [&](int r, int d, float x, float y) { st2((float*)p.W + (wrow0 + r) * DK + d, x, y); });
    }
}

// ---------------------------------------------------------------------------------------------
// K2: forward state chain.  One CTA per (sequence, DS-column slice of d_v); columns of the state evolve independently,
// the chunks of a sequence are walked in order.  A chunk costs its two dependent products and two barriers, not its loads: four
// warps do nothing else than copy, K and P while Delta is made, the next W<-, Q and U~ while the state is updated.
template <int DK, int DS>
__global__ void __launch_bounds__(NT + kLoaders) k_chain_fwd(Ptrs p, int DV) {
    extern __shared__ __align__(16) float sm[];
    constexpr int LA = DK + 4, LB = DK + 8, LS = DS + 8, NS = DS / 8;
    float *sW = sm, *sQ = sW + C * LA, *sK = sQ + C * LA, *sP = sK + C * LB, *sU = sP + C * LDC, *sD = sU + C * LS,
          *sDs = sD + C * LS, *sh = sDs + C * LS;                     // sh: the state slice [DK][DS]
    __shared__ float sgq_[2][C], sgk_[2][C], sgC_[2];                 // by parity of the chunk
    const int H = p.H, nsl = DV / DS, j0 = (blockIdx.x % nsl) * DS, bh = blockIdx.x / nsl, b = bh / H, hh = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    const size_t nrows = (size_t)p.B * H * p.Tp;
    if (tid >= NT) {
        const int me = tid - NT;
        auto fetch1 = [&](int n) {     // read in the first phase of chunk n
            const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh, wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
            fetch_tile<C, DK, LA>(sW, (const float*)p.W + wrow0 * DK, DK, C, me);
            fetch_tile<C, DK, LA>(sQ, (const float*)p.q + row0 * DK, (size_t)H * DK, min(C, p.T - n * C), me);
            fetch_tile<C, DS, LS>(sU, (const float*)p.U + wrow0 * DV + j0, DV, C, me);
        };
        auto fetch2 = [&](int n) {     // read in the second
            const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh, wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
            fetch_tile<C, DK, LB>(sK, (const float*)p.k + row0 * DK, (size_t)H * DK, min(C, p.T - n * C), me);
            fetch_tile<C, C, LDC>(sP, (const float*)p.P + wrow0 * C, C, C, me);
        };
        ChainCoef cf;
        fetch1(0);
        cf.get(p, (size_t)bh * p.Tp, nrows, me);
        for (int n = 0; n < p.N; ++n) {
            cf.put(sgq_[n & 1], sgk_[n & 1], sgC_ + (n & 1), me);
            fetched();
            __syncthreads();           // W<-, Q, U~ and the factors are there; K and P have been read
            fetch2(n);
            fetched();
            __syncthreads();           // K and P are there; W<-, Q and U~ have been read
            if (n + 1 < p.N) { fetch1(n + 1); cf.get(p, (size_t)bh * p.Tp + (size_t)(n + 1) * C, nrows, me); }
        }
        return;
    }
    for (int e = tid; e < DK * DS; e += NT)
        sh[(e / DS) * LS + e % DS] = p.h0 ? p.h0[((size_t)bh * DK + e / DS) * DV + j0 + e % DS] : 0.f;
    for (int n = 0; n < p.N; ++n) {
        const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh, wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
        const int live = min(C, p.T - n * C);
        const float *sgq = sgq_[n & 1], *sgk = sgk_[n & 1];
        __syncthreads();
        const float gC = sgC_[n & 1];
        if (p.save) {
            float* dst = p.hs + ((size_t)bh * p.N + n) * DK * DV + j0;
            for (int e = tid * 4; e < DK * DS; e += NT * 4)
                *reinterpret_cast<float4*>(dst + (size_t)(e / DS) * DV + e % DS) =
                    *reinterpret_cast<const float4*>(sh + (e / DS) * LS + e % DS);
        }
        // first half of the warps: Delta = U~ - W<- h;  second: Q h, the inter-chunk part of the output, kept in registers
        float acc[1][NS][4];
        zero(acc);
        const int m0 = (warp & 3) * 16;
        auto hf = [&](int i, int j) { return sh[i * LS + j]; };
        if (warp < 4) {
            wmm<1, NS>(acc, m0, 0, DK, [&](int r, int i) { return sW[r * LA + i]; }, hf);
            each(acc, m0, 0, [&](int r, int j, float x, float y) {
                x = sU[r * LS + j] - x; y = sU[r * LS + j + 1] - y;
                st2(sD + r * LS + j, x, y);
                st2(sDs + r * LS + j, x * sgk[r], y * sgk[r]);
                if (p.save) st2((float*)p.D + (wrow0 + r) * DV + j0 + j, x, y);
            });
        } else {
            wmm<1, NS>(acc, m0, 0, DK, [&](int r, int i) { return sQ[r * LA + i]; }, hf);
        }
        __syncthreads();
        if (warp >= 4) {
            // + P Delta, the intra-chunk part
            const int gq = (tid & 31) >> 2;
            const float s0 = sgq[m0 + gq], s1 = sgq[m0 + 8 + gq];
#pragma unroll
            for (int j = 0; j < NS; ++j) { acc[0][j][0] *= s0; acc[0][j][1] *= s0; acc[0][j][2] *= s1; acc[0][j][3] *= s1; }
            wmm<1, NS>(acc, m0, 0, m0 + 16, [&](int r, int s) { return sP[r * LDC + s]; },
                                  [&](int s, int j) { return sD[s * LS + j]; });
            each(acc, m0, 0, [&](int r, int j, float x, float y) {
                if (r < live) st2((float*)p.o + (row0 + (size_t)r * H) * DV + j0 + j, x, y);
            });
        } else {
            // h <- gamma_C h + K^T (diag(gamma_C/gamma) Delta)
            float ha[DK / 64][NS][4];
            zero(ha);
            const int i0 = (warp & 3) * (DK / 4);
            wmm<DK / 64, NS>(ha, i0, 0, C, [&](int i, int r) { return sK[r * LB + i]; },
                                   [&](int r, int j) { return sDs[r * LS + j]; });
            each(ha, i0, 0, [&](int i, int j, float x, float y) {
                float* d = sh + i * LS + j;
                st2(d, fmaf(gC, d[0], x), fmaf(gC, d[1], y));
            });
        }
    }
    if (p.hT) {
        asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");    // the state is complete
        for (int e = tid; e < DK * DS; e += NT)
            p.hT[((size_t)bh * DK + e / DS) * DV + j0 + e % DS] = sh[(e / DS) * LS + e % DS];
    }
}

// ---------------------------------------------------------------------------------------------
// K3: reverse state chain.  Carries dh (gradient w.r.t. the chunk's exit state) backwards:
//   dDelta = P^T dO + K-> dh ;   dh_in = gamma_C dh + (diag(gamma) Q)^T dO - W<-^T dDelta
// and leaves per chunk: dh (exit), dDelta, and two scalar partial sums the decay gradient needs.
template <int DK, int DS>
__global__ void __launch_bounds__(NT + kLoaders) k_chain_bwd(Ptrs p, int DV) {
    extern __shared__ __align__(16) float sm[];
    constexpr int LA = DK + 4, LB = DK + 8, LP = C + 8, LS = DS + 8, NS = DS / 8;
    float *sK = sm, *sQ = sK + C * LA, *sW = sQ + C * LB, *sP = sW + C * LB, *sO = sP + C * LP, *sOs = sO + C * LS,
          *sD = sOs + C * LS, *sdD = sD + C * LS, *sdh = sdD + C * LS;
    __shared__ float sgq_[2][C], sgk_[2][C], sgC_[2], sred[NT / 32], skd[C];          // the first three by parity of the chunk
    const int H = p.H, nsl = DV / DS, sl = blockIdx.x % nsl, j0 = sl * DS, bh = blockIdx.x / nsl, b = bh / H, hh = bh % H;
    const int tid = threadIdx.x, warp = tid >> 5;
    const size_t nrows = (size_t)p.B * H * p.Tp, BHN = (size_t)p.B * H * p.N;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    if (tid >= NT) {
        const int me = tid - NT;
        auto fetch1 = [&](int n) {     // read in the first two phases of chunk n
            const size_t row0 = ((size_t)b * p.T + (size_t)n * C) * H + hh, wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
            const int live = min(C, p.T - n * C);
            fetch_tile<C, DS, LS>(sO, (const float*)p.dO + row0 * DV + j0, (size_t)H * DV, live, me);
            fetch_tile<C, DS, LS>(sD, (const float*)p.D + wrow0 * DV + j0, DV, C, me);
            fetch_tile<C, DK, LA>(sK, (const float*)p.k + row0 * DK, (size_t)H * DK, live, me);
            fetch_tile<C, DK, LB>(sQ, (const float*)p.q + row0 * DK, (size_t)H * DK, live, me);
            fetch_tile<C, C, LP>(sP, (const float*)p.P + wrow0 * C, C, C, me);
        };
        ChainCoef cf;
        fetch1(p.N - 1);
        cf.get(p, (size_t)bh * p.Tp + (size_t)(p.N - 1) * C, nrows, me);
        for (int n = p.N - 1; n >= 0; --n) {
            const size_t wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
            cf.put(sgq_[n & 1], sgk_[n & 1], sgC_ + (n & 1), me);
            fetched();
            __syncthreads();           // all but W<- is there; W<- has been read
            fetch_tile<C, DK, LB>(sW, (const float*)p.W + wrow0 * DK, DK, C, me);
            __syncthreads();
            fetched();
            __syncthreads();           // W<- is there; the others have been read
            if (n > 0) { fetch1(n - 1); cf.get(p, wrow0 - C, nrows, me); }
        }
        return;
    }
    for (int e = tid; e < DK * DS; e += NT)
        sdh[(e / DS) * LS + e % DS] = p.dhT ? p.dhT[((size_t)bh * DK + e / DS) * DV + j0 + e % DS] : 0.f;
    for (int n = p.N - 1; n >= 0; --n) {
        const size_t wrow0 = (size_t)bh * p.Tp + (size_t)n * C;
        const float *sgq = sgq_[n & 1], *sgk = sgk_[n & 1];
        __syncthreads();
        const float gC = sgC_[n & 1];
        // keep dh of this chunk's exit state; partial <dh, h_entry>_F over this slice
        {
            float* dst = p.dhs + ((size_t)bh * p.N + n) * DK * DV + j0;
            const float* hsrc = p.hs + ((size_t)bh * p.N + n) * DK * DV + j0;
            float part = 0.f;
#pragma unroll 2
            for (int e = tid * 4; e < DK * DS; e += NT * 4) {
                const size_t off = (size_t)(e / DS) * DV + e % DS;
                const float4 x = *reinterpret_cast<const float4*>(sdh + (e / DS) * LS + e % DS);
                const float4 y = *reinterpret_cast<const float4*>(hsrc + off);
                *reinterpret_cast<float4*>(dst + off) = x;
                part = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, part))));
            }
            part = warp_sum(part);
            if ((tid & 31) == 0) sred[warp] = part;
            for (int e = tid; e < C * DS; e += NT) {             // diag(gamma / |q|) dO, the operand of Q^T
                const int r = e / DS, j = e % DS;
                sOs[r * LS + j] = sO[r * LS + j] * sgq[r];
            }
        }
        __syncthreads();
        if (tid == 0) {
            float tot = 0.f;
            for (int w = 0; w < NT / 32; ++w) tot += sred[w];
            p.dhh[(size_t)sl * BHN + (size_t)bh * p.N + n] = tot;
        }
        float ha[DK / 64][NS][4];
        zero(ha);
        const int i0 = (warp & 3) * (DK / 4);
        if (warp < 4) {
            // dDelta = diag(gamma_C/gamma) K dh + P^T dO, 16 tokens per warp; row sums of the first term times Delta
            float acc[1][NS][4];
            zero(acc);
            const int m0 = (warp & 3) * 16;
            wmm<1, NS>(acc, m0, 0, DK, [&](int s, int i) { return sK[s * LA + i]; },
                                  [&](int i, int j) { return sdh[i * LS + j]; });
            const int gq = (tid & 31) >> 2;
            const float s0 = sgk[m0 + gq], s1 = sgk[m0 + 8 + gq];
#pragma unroll
            for (int j = 0; j < NS; ++j) { acc[0][j][0] *= s0; acc[0][j][1] *= s0; acc[0][j][2] *= s1; acc[0][j][3] *= s1; }
            row_sums(acc, m0, 0, skd,
                     [&](int s, int j, float x, float y) { return fmaf(x, sD[s * LS + j], y * sD[s * LS + j + 1]); });
            wmm<1, NS>(acc, m0, 0, C, [&](int s, int r) { return sP[r * LP + s]; },
                                   [&](int r, int j) { return sO[r * LS + j]; });
            each(acc, m0, 0, [&](int s, int j, float x, float y) {
                st2(sdD + s * LS + j, -x, -y);
                st2((float*)p.dD + (wrow0 + s) * DV + j0 + j, x, y);
            });
        } else {
            wmm<DK / 64, NS>(ha, i0, 0, C, [&](int i, int r) { return sQ[r * LB + i]; },
                                   [&](int r, int j) { return sOs[r * LS + j]; });
        }
        __syncthreads();
        if (warp >= 4) {
            wmm<DK / 64, NS>(ha, i0, 0, C, [&](int i, int r) { return sW[r * LB + i]; },
                                   [&](int r, int j) { return sdD[r * LS + j]; });
            each(ha, i0, 0, [&](int i, int j, float x, float y) {
                float* d = sdh + i * LS + j;
                st2(d, fmaf(gC, d[0], x), fmaf(gC, d[1], y));
            });
        } else if (tid < C) {
            p.kdhd[(size_t)sl * nrows + wrow0 + tid] = skd[tid];
        }
    }
    if (p.dh0) {
        asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");    // the gradient is complete
        for (int e = tid; e < DK * DS; e += NT)
            p.dh0[((size_t)bh * DK + e / DS) * DV + j0 + e % DS] = sdh[(e / DS) * LS + e % DS];
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
    extern __shared__ __align__(16) float sm[];
    constexpr int LT = BwdSmem<DK, DV>::LT, LH = DV + kPad, kSlot = BwdSmem<DK, DV>::kSlot, NK = DK / 32;
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
    const bool low = nc < wm + 32;                              // a 64 x 64 tile of this warp matters only if it reaches below the diagonal

    Tile<C, DK, LT> tq, tk;
    Tile<C, DV, LT> tv;
    Tile<DK, DV, LH> th;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    // ---- coefficients, Q, K, M; dO and Delta ----------------------------------------------------
    tq.get((const float*)p.q + row0 * DK, (size_t)H * DK, live);
    tk.get((const float*)p.k + row0 * DK, (size_t)H * DK, live);
    if (tid < C) {
        const size_t r = row0 + (size_t)tid * H;
        const bool in = tid < live;
        const float g = p.g[wrow0 + tid], gC = p.g[wrow0 + C - 1];
        sbeta[tid] = in ? gate(ld((const float*)p.beta, r), p.logits) : 0.f;
        const float lm = (in && p.lam) ? gate(ld((const float*)p.lam, r), p.logits) : 0.f;
        salpha[tid] = (in && p.alpha) ? gate(ld((const float*)p.alpha, r), p.logits) : 1.f;
        const float rq = p.rqk ? p.rqk[wrow0 + tid] : 1.f, rk = p.rqk ? p.rqk[nrows + wrow0 + tid] : 1.f;
        slam[tid] = lm; sg[tid] = g; sgam[tid] = expf(g); segc[tid] = expf(gC - g);
        srq[tid] = rq; srk[tid] = rk; scq[tid] = lm * rq;
    }
    tq.put(s0); tk.put(s1);
    load_tile<C, C, LDC>(m1, p.M + wrow0 * C, C, C);
    load_tile<C, DV, LT>(s2, (const float*)p.dO + row0 * DV, (size_t)H * DV, live);
    load_tile<C, DV, LT>(s3, (const float*)p.D + wrow0 * DV, DV, C);
    __syncthreads();
    auto Qf = [&](int r, int d) { return s0[r * LT + d]; };                                       // as stored
    auto Kf = [&](int r, int d) { return s1[r * LT + d]; };
    auto Xf = [&](int r, int d) { return fmaf(scq[r], s0[r * LT + d], srk[r] * s1[r * LT + d]); };
    th.get(dhs, DV, DK);
    // ---- X K^T, and dP with its uses: dP o P (row and column sums) and dP o Gamma -------------------
    {
        float a[2][2][4];
        zero(a);
        if (low) wmm<2, 2>(a, wm, nc, DK, Xf, [&](int d, int i) { return s1[i * LT + d]; });
        each(a, wm, nc, [&](int r, int i, float x, float y) { st2(m0 + r * LDC + i, x * srk[i], y * srk[i + 1]); });
        zero(a);
        if (low) wmm<2, 2>(a, wm, nc, DV, [&](int r, int j) { return s2[r * LT + j]; }, [&](int j, int s) { return s3[s * LT + j]; });
        each(a, wm, nc, [&](int r, int s, float& x, float& y) {
            const float2 pv = ld2((const float*)p.P + (wrow0 + r) * C + s);
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
    wmm<2, NK>(aK, wm, nk, DV, [&](int r, int j) { return s3[r * LT + j]; }, [&](int j, int i) { return s0[i * LH + j]; });
    __syncthreads();                                            // dh and Delta have been read
    th.put(s0);
    tv.get((const float*)p.dD + wrow0 * DV, DV, C);
    tv.put(s3);
    __syncthreads();
    tv.get((const float*)p.v + row0 * DV, (size_t)H * DV, live);
    zero(aQ); zero(aX);
    wmm<2, NK>(aQ, wm, nk, DV, [&](int r, int j) { return s2[r * LT + j]; }, [&](int j, int i) { return s0[i * LH + j]; });
    wmm<2, NK>(aX, wm, nk, DV, [&](int r, int j) { return s3[r * LT + j]; }, [&](int j, int i) { return s0[i * LH + j]; });
    __syncthreads();                                            // h and dO have been read
    each(aX, wm, nk, [&](int r, int i, float x, float y) { st2(s2 + r * LT + i, -x, -y); });       // dW<-
    tv.put(s0);
    each(aK, wm, nk, [&](int r, int, float& x, float& y) { x *= segc[r]; y *= segc[r]; });
    each(aQ, wm, nk, [&](int r, int, float& x, float& y) { x *= sgam[r]; y *= sgam[r]; });
    __syncthreads();
    tq.get((const float*)p.q + row0 * DK, (size_t)H * DK, live);
    tk.get((const float*)p.k + row0 * DK, (size_t)H * DK, live);
    // ---- dT = dDelta V^T + dW<- (gamma X)^T;  dV = T^T dDelta -------------------------------------
    float aT[2][2][4];
    zero(aT);
    if (low) wmm<2, 2>(aT, wm, nc, DV, [&](int r, int j) { return s3[r * LT + j]; }, [&](int j, int s) { return s0[s * LT + j]; });
    {
        float a[2][DV / 32][4];
        zero(a);
        wmm<2, DV / 32>(a, wm, wn * (DV / 4), C, [&](int s, int r) { return m1[r * LDC + s]; },
                               [&](int r, int j) { return s3[r * LT + j]; }, wm);
        each(a, wm, wn * (DV / 4), [&](int s, int j, float x, float y) {
            if (s < live) st2((float*)p.dv_ + (row0 + (size_t)s * H) * DV + j, sbeta[s] * x, sbeta[s] * y);
        });
    }
    __syncthreads();                                            // V has been read
    tq.put(s0); tk.put(s1);
    __syncthreads();
    {
        float a[2][2][4];
        zero(a);
        if (low) wmm<2, 2>(a, wm, nc, DK, [&](int r, int i) { return s2[r * LT + i]; }, [&](int i, int s) { return Xf(s, i); });
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
    wmm<2, NK>(aX, wm, nk, C, [&](int s, int r) { return m1[r * LDC + s]; }, [&](int r, int i) { return s2[r * LT + i]; }, wm);
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
        if (low) wmm<2, 2>(a, wm, nc, nc + 16, [&](int r, int u) { return m2[r * LDC + u] * sbeta[u]; }, [&](int u, int s2_) { return m1[s2_ * LDC + u]; });
        each(a, wm, nc, [&](int r, int s_, float x, float y) { st2(m4 + r * LDC + s_, x, y); });
    }
    __syncthreads();
    {
        float a[2][2][4];
        zero(a);
        if (low) wmm<2, 2>(a, wm, nc, C, [&](int r, int u) { return m1[u * LDC + r]; }, [&](int u, int s) { return m4[u * LDC + s]; }, wm);
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
    wmm<2, NK>(aX, wm, nk, wm + 32, [&](int r, int s) { return m2[r * LDC + s]; }, [&](int s, int d) { return srk[s] * Kf(s, d); });
    row_sums(aX, wm, nk, prow[4][wn],
             [&](int r, int i, float x, float y) { return srq[r] * fmaf(x, Qf(r, i), y * Qf(r, i + 1)); });
    wmm<2, NK>(aK, wm, nk, C, [&](int i, int r) { return m2[r * LDC + i]; }, Xf, wm);
    wmm<2, NK>(aK, wm, nk, C, [&](int i, int r) { return m3[r * LDC + i]; }, [&](int r, int d) { return srq[r] * Qf(r, d); }, wm);
    wmm<2, NK>(aQ, wm, nk, wm + 32, [&](int r, int s) { return m3[r * LDC + s]; }, [&](int s, int d) { return srk[s] * Kf(s, d); });
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
    each(aK, wm, nk, [&](int r, int i, float x, float y) { if (r < live) st2((float*)p.dk_ + (row0 + (size_t)r * H) * DK + i, x, y); });
    each(aQ, wm, nk, [&](int r, int i, float x, float y) { if (r < live) st2((float*)p.dq + (row0 + (size_t)r * H) * DK + i, x, y); });
    __syncthreads();
    {
        const int col = tid & 63, q4 = tid >> 6;
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < 16; ++r) s += m0[(q4 * 16 + r) * LDC + col];           // column sums of dA o A
        part[q4][col] = s;
    }
    __syncthreads();
    token_gradients<float>(p, prow, pcol, part, db1, sbeta, slam, salpha, sgam, sdg, skd, row0, wrow0, bh, n, live);
}

template <int DK, int DV>
cudaError_t prep_for(const ChunkArgs& a, const Ptrs& p) {
    constexpr size_t smem = sizeof(float) * (2 * C * (DK + kPad) + C * (DV + kPad) + 2 * C * LDC + C * LDI);
    return launch(k_prep<DK, DV>, a.s.B * a.s.H * p.N, NT, smem, a.stream, p);
}
template <int DK, int DS>
cudaError_t chain_fwd_for(const ChunkArgs& a, const Ptrs& p) {
    constexpr size_t smem = sizeof(float) * (2 * C * (DK + 4) + C * (DK + 8) + C * LDC + (3 * C + DK) * (DS + 8));
    return launch(k_chain_fwd<DK, DS>, a.s.B * a.s.H * (a.s.dv / DS), NT + kLoaders, smem, a.stream, p, a.s.dv);
}
template <int DK, int DS>
cudaError_t chain_bwd_for(const ChunkArgs& a, const Ptrs& p) {
    constexpr size_t smem = sizeof(float) * (C * (DK + 4) + 2 * C * (DK + 8) + C * (C + 8) + (4 * C + DK) * (DS + 8));
    return launch(k_chain_bwd<DK, DS>, a.s.B * a.s.H * (a.s.dv / DS), NT + kLoaders, smem, a.stream, p, a.s.dv);
}
template <int DK, int DV>
cudaError_t chunk_bwd_for(const ChunkArgs& a, const Ptrs& p) {
    return launch(k_chunk_bwd<DK, DV>, a.s.B * a.s.H * p.N, NT, BwdSmem<DK, DV>::bytes, a.stream, p);
}

}  // namespace

// d_v columns that one CTA of the state chains owns: 16 while each CTA then has an SM of its own, because a chain's time is its
// dependent steps; 32, which read W<-, Q, K and P half as often, beyond.  Both kernels turn there.  Training pass of 512 tokens,
// narrow against wide, on either side of 148 narrow CTAs (d_k x d_v, sequences):
//   fp32   64 x 64    37: 145 against 169 us   38: 226 against 202      bf16   64 x 64    37:  83 against  96   38: 124 against 116
//         128 x 64    37: 219 against 262      38: 354 against 318            128 x 64    37: 112 against 132   38: 193 against 163
//          64 x 128   18: 117 against 139      19: 207 against 181             64 x 128   18:  70 against  82   19: 112 against 105
//         128 x 128   18: 164 against 199      19: 310 against 272
// With 2048 tokens both sides are further apart (fp32 128 x 128 661 against 792, 1046 against 866); between 160 and 800 narrow CTAs wide
// slices stay ahead, least with fp32 at 300 to 400 of them (1.3 - 3.5 %).
int split_slice(const qd_shape& s) { return (long long)s.B * s.H * (s.dv / 16) <= kSMs ? 16 : 32; }

#define QD_BY_DIMS(fn, a, p)                                                                                  \
    ((a).s.dk == 128 ? ((a).s.dv == 128 ? fn<128, 128>(a, p) : fn<128, 64>(a, p))                                  \
                     : ((a).s.dv == 128 ? fn<64, 128>(a, p) : fn<64, 64>(a, p)))
#define QD_BY_SLICE(fn, a, p)                                                                                 \
    ((a).s.dk == 128 ? ((a).L.slice == 32 ? fn<128, 32>(a, p) : fn<128, 16>(a, p))                                 \
                     : ((a).L.slice == 32 ? fn<64, 32>(a, p) : fn<64, 16>(a, p)))

cudaError_t split_prep(const ChunkArgs& a) {
    return a.s.dtype == QD_BF16 ? split_bf16_prep(a) : QD_BY_DIMS(prep_for, a, make_ptrs(a));
}
cudaError_t split_chain_fwd(const ChunkArgs& a) {
    return a.s.dtype == QD_BF16 ? split_bf16_chain_fwd(a) : QD_BY_SLICE(chain_fwd_for, a, make_ptrs(a));
}
cudaError_t split_chain_bwd(const ChunkArgs& a) {
    return a.s.dtype == QD_BF16 ? split_bf16_chain_bwd(a) : QD_BY_SLICE(chain_bwd_for, a, make_ptrs(a));
}
cudaError_t split_chunk_bwd(const ChunkArgs& a) {
    return a.s.dtype == QD_BF16 ? split_bf16_chunk_bwd(a) : QD_BY_DIMS(chunk_bwd_for, a, make_ptrs(a));
}

}  // namespace qd
