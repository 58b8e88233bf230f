// The accurate path for bf16 storage: the head dimensions that the tcgen05 kernels do not cover (d_k or d_v = 64).  The same
// kernels as those for fp32 storage (split_chunk.cu), with fp32-accurate products of bf16 planes (planes.cuh): q, k, v, dO and
// what the kernels leave one another in bf16 are exact in one plane, states and 64 x 64 matrices take three.
#include "split_common.cuh"
#include "planes.cuh"

namespace qd {
namespace {

// ---------------------------------------------------------------------------------------------
// K1: per chunk-head, state-independent part: g, P, W<-, U~ (and M for the backward).  X is never formed, X K^T and T diag(gamma) X are each a product with K and one
// with Q, their coefficients applied to the result or to T.  One set of planes holds T, T diag(gamma / |k|) and
// T diag(lambda gamma / |q|) in turn, over what the inverse needed; at d_k = d_v = 64 three CTAs fit an SM.
// 1024 chunks of 64 x 64: 72 us with tf32 halves and two CTAs, 46 so (d_k 128, d_v 64: 119 and 60; d_k 64, d_v 128: 55; 64 x 64
// normalised 56), bound by the latency of its chain of small steps.
template <int DK, int DV>
struct PrepPlanes {
    typedef Planes<C, DK, 1> TQ;
    typedef Planes<C, DV, 1> TV;
    typedef Planes<C, C, 3> TC;
    static constexpr int kT = 2 * TQ::kBytes + TV::kBytes, kM = kT + TC::kBytes, kBytes = kM + C * LDC * 4, kCtas = kBytes <= 74 * 1024 ? 3 : 2;
    static_assert(C * (LDC + LDI) * 4 <= TC::kBytes, "A and the inverse's scratch");
};
template <int DK, int DV>
__global__ void __launch_bounds__(NT, PrepPlanes<DK, DV>::kCtas) k_prep(Ptrs p) {
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
    const int wm = ((warp ^ (warp >> 2)) & 1) * 32, wn = warp >> 1;      // both halves of the rows on every scheduler
    {
        float kk[2][2][4], qk[2][2][4];
        zero(kk); zero(qk);
        if (wn * 16 < wm + 32) {                                // not above the diagonal
            pmm<false, false>(kk, mK, mK, wm, wn * 16, DK);
            pmm<false, false>(qk, mQ, mK, wm, wn * 16, DK);
        }
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
        pmm<false, true>(u, mT, mV, wm, wn * (DV / 4), wm + 32);
        each(u, wm, wn * (DV / 4), [&](int r, int j, float x, float y) { st2((IO*)p.U + (wrow0 + r) * DV + j, x, y); });
    }
    __syncthreads();
    float w[2][DK / 32][4];
    zero(w);
    put_T([&](int i) { return sck[i]; });
    pmm<false, true>(w, mT, mK, wm, wn * (DK / 4), wm + 32);
    __syncthreads();
    put_T([&](int i) { return scq[i]; });
    pmm<false, true>(w, mT, mQ, wm, wn * (DK / 4), wm + 32);
    each(w, wm, wn * (DK / 4), [&](int r, int d, float x, float y) { st2((IO*)p.W + (wrow0 + r) * DK + d, x, y); });
}

// ---------------------------------------------------------------------------------------------
// K2, K3: the state chains.  One CTA per (sequence, DS-column slice of d_v).  Every warp takes a 16 x 16 tile of the 64 x DS
// products and DK/4 x 16 of the state, which it keeps in fp32 in its registers (planes of it are what the others read).  A
// chunk is two phases and two barriers; the tiles of one phase arrive while the other is worked on, those of the first two
// phases ahead.  Slices of 32 columns and d_k = 64 let two CTAs share an SM.  B4 T1024 H16 d_k = d_v = 64: 73 and 85 us with
// tf32 halves, 45 and 54 with everybody loading, 42 and 49 so (2.5 us a chunk, of which the tensor unit works a third: the rest is
// the latency of two dependent products and two barriers).  LOADERS: the copies have warps of their own, while a CTA has
// an SM to itself; beyond that two CTAs share one, whose registers the extra warps would not leave room for (128 sequences of 1024
// tokens, 256 CTAs: forward and backward 435 us without, 457 with).
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
template <int DK, int DS, bool LOADERS>
__global__ void __launch_bounds__(8 * DS + (LOADERS ? kLoaders : 0)) k_chain_fwd(Ptrs p, int DV) {
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
    const int wm = (warp & 4 ? 3 - (warp & 3) : warp & 3) * 16, wn = (warp >> 2) * 16, si = (warp & 3) * 16 * MU;
    const size_t nrows = (size_t)p.B * H * p.Tp, row0 = (size_t)b * p.T * H + hh, wrow0 = (size_t)bh * p.Tp;
    constexpr int NL = LOADERS ? kLoaders : TH;
    const int me = LOADERS ? tid - TH : tid;               // who loads: extra warps, or everybody; me < 0: not this one
    const bool loads = !LOADERS || tid >= TH, works = !LOADERS || tid < TH;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    auto fetch1 = [&](int n) {         // W<- and Q, read in the first phase of chunk n
        const typename L::TA w(smb + (n & 1) * L::TA2::kBytes), q(smb + (n & 1) * L::TA2::kBytes + L::TA::kBytes);
        w.template fetch<NL>((const IO*)p.W + (wrow0 + (size_t)n * C) * DK, DK, C, me);
        q.template fetch<NL>((const IO*)p.q + (row0 + (size_t)n * C * H) * DK, (size_t)H * DK, min(C, p.T - n * C), me);
    };
    auto fetch2 = [&](int n) {         // K and P, read in the second
        mK.template fetch<NL>((const IO*)p.k + (row0 + (size_t)n * C * H) * DK, (size_t)H * DK, min(C, p.T - n * C), me);
        mP.template fetch<NL>((const IO*)p.P + (wrow0 + (size_t)n * C) * C, C, C, me);
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
    if (loads) {
        fetch1(0);
        cf.get(p, wrow0, nrows, me);
    }
    fetch_commit();
    if (works) fetch_u(0);
    float hst[MU][2][4];
    zero(hst);
    auto state_at = [&](float* base, int i, int j) { return reinterpret_cast<float2*>(base + (size_t)i * DV + j0 + j); };
    if (p.h0 && works) each(hst, si, wn, [&](int i, int j, float& x, float& y) {
        const float2 v = *state_at(const_cast<float*>(p.h0) + (size_t)bh * DK * DV, i, j);
        x = v.x; y = v.y;
    });
    if (works) each(hst, si, wn, [&](int i, int j, float x, float y) {
        mS.st2(i, j, x, y);
        if (p.save) *state_at(p.hs + (size_t)bh * p.N * DK * DV, i, j) = make_float2(x, y);
    });
    if (loads) cf.put(sgq[0], sgk[0], sgC, me);
    for (int n = 0; n < p.N; ++n) {
        const int bf = n & 1, live = min(C, p.T - n * C);
        const bool more = n + 1 < p.N;
        fetch_wait();
        __syncthreads();
        if (loads) fetch2(n);
        fetch_commit();
        if (more && loads) { fetch1(n + 1); cf.get(p, wrow0 + (size_t)(n + 1) * C, nrows, me); }
        fetch_commit();
        if (LOADERS && loads) {
            fetch_wait_but<1>();
            __syncthreads();
            if (more) cf.put(sgq[bf ^ 1], sgk[bf ^ 1], sgC + (bf ^ 1), me);
            continue;
        }
        // Delta = U~ - W<- h, and Q h, the inter-chunk part of the output
        float a[2][2][4], o[1][2][4];
        zero(a); zero(o);
        mWQ.p = reinterpret_cast<IO*>(smb + bf * L::TA2::kBytes);
        pmm<false, true, 4, 2, 2, typename L::TA2, typename L::TS, C>(a, mWQ, mS, wm, wn, DK);
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
            pmm<true, true, 4>(s, mK, mDs, si, wn, C);
            const float gc = sgC[bf];
            each2(hst, s, si, wn, [&](int i, int j, float& x, float& y, float dx, float dy) {
                x = fmaf(gc, x, dx); y = fmaf(gc, y, dy);
                mS.st2(i, j, x, y);
                if (p.save && more) *state_at(p.hs + ((size_t)bh * p.N + n + 1) * DK * DV, i, j) = make_float2(x, y);
            });
        }
        // o = diag(gamma) Q h + P Delta
        pmm<false, true, 4>(o, mP, mD, wm, wn, wm + 16);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int r = wm + 8 * h + g;
                const float f = sgq[bf][r];
                if (r < live) st2((IO*)p.o + (row0 + (size_t)(n * C + r) * H) * DV + j0 + wn + 8 * j + 2 * t,
                                  fmaf(f, a[1][j][2 * h], o[0][j][2 * h]), fmaf(f, a[1][j][2 * h + 1], o[0][j][2 * h + 1]));
            }
        if (!LOADERS && more) cf.put(sgq[bf ^ 1], sgk[bf ^ 1], sgC + (bf ^ 1));
    }
    if (p.hT && works) each(hst, si, wn, [&](int i, int j, float x, float y) { *state_at(p.hT + (size_t)bh * DK * DV, i, j) = make_float2(x, y); });
}

template <int DK, int DS, bool LOADERS>
__global__ void __launch_bounds__(8 * DS + (LOADERS ? kLoaders : 0)) k_chain_bwd(Ptrs p, int DV) {
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
    const int wm = (warp & 4 ? 3 - (warp & 3) : warp & 3) * 16, wn = (warp >> 2) * 16, si = (warp & 3) * 16 * MU;
    const size_t nrows = (size_t)p.B * H * p.Tp, BHN = (size_t)p.B * H * p.N, row0 = (size_t)b * p.T * H + hh, wrow0 = (size_t)bh * p.Tp;
    constexpr int NL = LOADERS ? kLoaders : TH;
    const int me = LOADERS ? tid - TH : tid;               // who loads: extra warps, or everybody; me < 0: not this one
    const bool loads = !LOADERS || tid >= TH, works = !LOADERS || tid < TH;
    sm100::grid_dep_wait();            // launched while the kernel before it drains
    sm100::grid_dep_launch();
    auto fetch1 = [&](int n) {         // K, P and dO, read in the first phase of chunk n
        unsigned char* s = smb + (n & 1) * kSet;
        const typename L::TA k(s);
        const typename L::TP pm(s + L::TA::kBytes);
        const typename L::TO o(s + L::TA::kBytes + L::TP::kBytes);
        const int live = min(C, p.T - n * C);
        k.template fetch<NL>((const IO*)p.k + (row0 + (size_t)n * C * H) * DK, (size_t)H * DK, live, me);
        pm.template fetch<NL>((const IO*)p.P + (wrow0 + (size_t)n * C) * C, C, C, me);
        o.template fetch<NL>((const IO*)p.dO + (row0 + (size_t)n * C * H) * DV + j0, (size_t)H * DV, live, me);
    };
    auto fetch2 = [&](int n) {         // Q and W<-, read in the second
        mQ.template fetch<NL>((const IO*)p.q + (row0 + (size_t)n * C * H) * DK, (size_t)H * DK, min(C, p.T - n * C), me);
        mW.template fetch<NL>((const IO*)p.W + (wrow0 + (size_t)n * C) * DK, DK, C, me);
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
    if (loads) {
        fetch1(p.N - 1);
        cf.get(p, wrow0 + (size_t)(p.N - 1) * C, nrows, me);
    }
    fetch_commit();
    if (works) fetch_d(p.N - 1);
    float dst[MU][2][4];
    zero(dst);
    if (p.dhT && works) each(dst, si, wn, [&](int i, int j, float& x, float& y) {
        const float2 v = *state_at(const_cast<float*>(p.dhT) + (size_t)bh * DK * DV, i, j);
        x = v.x; y = v.y;
    });
    if (works) each(dst, si, wn, [&](int i, int j, float x, float y) { mS.st2(i, j, x, y); });
    if (loads) cf.put(sgq[(p.N - 1) & 1], sgk[(p.N - 1) & 1], sgC + ((p.N - 1) & 1), me);
    for (int n = p.N - 1; n >= 0; --n) {
        const int bf = n & 1;
        fetch_wait();
        __syncthreads();
        if (loads) fetch2(n);
        fetch_commit();
        if (n > 0 && loads) { fetch1(n - 1); cf.get(p, wrow0 + (size_t)(n - 1) * C, nrows, me); }
        fetch_commit();
        if (LOADERS && loads) {
            fetch_wait_but<1>();
            __syncthreads();
            if (n > 0) cf.put(sgq[bf ^ 1], sgk[bf ^ 1], sgC + (bf ^ 1), me);
            continue;
        }
        const typename L::TA mK(smb + bf * kSet);
        const typename L::TP mP(smb + bf * kSet + L::TA::kBytes);
        const typename L::TO mO(smb + bf * kSet + L::TA::kBytes + L::TP::kBytes);
        // dDelta = diag(gamma_C/gamma) K dh + P^T dO; row sums of the first term times Delta
        {
            float a[1][2][4], c[1][2][4];
            zero(a); zero(c);
            pmm<false, true, 4>(a, mK, mS, wm, wn, DK);
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
            pmm<true, true, 4>(c, mP, mO, wm, wn, C, wm);
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
            pmm<true, true, 4>(s, mQ, mOs, si, wn, C);
            pmm<true, true, 4>(s, mW, mdD, si, wn, C);
            const float gc = sgC[bf];
            each2(dst, s, si, wn, [&](int i, int j, float& x, float& y, float dx, float dy) {
                x = fmaf(gc, x, dx); y = fmaf(gc, y, dy);
                mS.st2(i, j, x, y);
            });
        }
        if (!LOADERS && n > 0) cf.put(sgq[bf ^ 1], sgk[bf ^ 1], sgC + (bf ^ 1));
    }
    if (p.dh0 && works) each(dst, si, wn, [&](int i, int j, float x, float y) { *state_at(p.dh0 + (size_t)bh * DK * DV, i, j) = make_float2(x, y); });
}

// ---------------------------------------------------------------------------------------------
// K4: chunk-parallel part of the backward: dq, dk, dv, dbeta, dlambda, dalpha.  X is never formed: a product with it is one with K and one with Q, which are
// exact in one plane, their coefficients applied to the result or to the other operand.  One slot of shared memory holds dh,
// h, dW<- and dT M^T in turn; M takes Delta's place, dT that of dO, dDelta and V.  So two CTAs fit an SM at d_k = d_v = 64: one
// computes while the other loads or waits at a barrier, and a warp's 32 x 16 tile reads 1.5 operand pieces per 16 x 16 x 16
// product, half of what 16 x 16 tiles of 16 warps would.  B4 T1024 H16 d_k = d_v = 64: 208 us with tf32 halves, 150 with 16
// warps and one CTA, 122 so, 115 with triangular operands read from or to their diagonal only.
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
    // where two CTAs fit: 32 x 16 tiles of 8 warps; one CTA: 16 warps hide more (1024 chunks of d_k 128, d_v 64: 174 us against 191
    // with 8 warps, normalised 197 against 220; d_k 64, d_v 128: 158 against 166)
    static constexpr int kCtas = kBytes <= 100 * 1024 ? 2 : 1, kThreads = kCtas == 2 ? 256 : 512;
};
template <int DK, int DV>
__global__ void __launch_bounds__(BwdPlanes<DK, DV>::kThreads, BwdPlanes<DK, DV>::kCtas) k_chunk_bwd(Ptrs p) {
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
    const int re = wm + 16 * MT;                                // a 64 x 64 tile of this warp matters only if it
    const bool low = nc < re;                                   // reaches below the diagonal
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
    if (low) pmm<false, false>(a3, mO, mD, wm, nc, DV);
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
    if (low) pmm<false, false>(aT, mdD, mV, wm, nc, DV);
    {
        float a[MT][NV][4];
        zero(a);
        pmm<true, true>(a, mM, mdD, wm, nv, C, wm);
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
        if (low) pmm<false, false>(a, mW, mK, wm, nc, DK);
        each2(aT, a, wm, nc, [&](int, int s, float& x, float& y, float u, float v) {
            x = fmaf(sgam[s] * srk[s], u, x); y = fmaf(sgam[s + 1] * srk[s + 1], v, y);
        });
        zero(a);
        if (low) pmm<false, false>(a, mW, mQ, wm, nc, DK);
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
    pmm<true, true>(aX, mM, mW, wm, nk, C, wm);
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
        if (low) pmm<false, false>(a, mT, mM, wm, nc, nc + 16);
        each(a, wm, nc, [&](int r, int s, float x, float y) { m4.st2(r, s, x, y); });
    }
    __syncthreads();
    {
        float a[MT][2][4], x[MT][2][4];
        zero(a); zero(x);
        if (low) {
            pmm<true, true>(a, mM, m4, wm, nc, C, wm);
            pmm<false, false>(x, mQ, mK, wm, nc, DK);           // X K^T
        }
        each(x, wm, nc, [&](int r, int, float& u, float& v) { u *= scq[r]; v *= scq[r]; });
        {
            float y[MT][2][4];
            zero(y);
            if (low) pmm<false, false>(y, mK, mK, wm, nc, DK);
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
        pmm<false, true>(aX, e1, mK, wm, nk, re);
        row_sums(aX, wm, nk, prow[4][wn], qsum);
        pmm<false, true>(aQ, e2, mK, wm, nk, re);
        pmm<true, true>(aK, e3, mQ, wm, nk, C, wm);
        if (p.rqk) {                                            // dXK scaled by row instead of by column
            __syncthreads();
            each(a, wm, nc, [&](int r, int s, float, float) {
                const float2 d = e1.ld2(r, s);
                e1.st2(r, s, d.x * (srk[r] / srk[s]), d.y * (srk[r] / srk[s + 1]));
            });
            __syncthreads();
        }
        pmm<true, true>(aK, e1, mK, wm, nk, C, wm);
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

template <int DK, int DV>
cudaError_t prep_for(const ChunkArgs& a, const Ptrs& p) {
    return launch(k_prep<DK, DV>, a.s.B * a.s.H * p.N, NT, PrepPlanes<DK, DV>::kBytes, a.stream, p);
}
template <int DK, int DS>
cudaError_t chain_fwd_for(const ChunkArgs& a, const Ptrs& p) {
    typedef ChainPlanes<DK, DS> L;
    const int grid = a.s.B * a.s.H * (a.s.dv / DS);
    if (grid <= kSMs) return launch(k_chain_fwd<DK, DS, true>, grid, L::kThreads + kLoaders, L::kFwd, a.stream, p, a.s.dv);
    return launch(k_chain_fwd<DK, DS, false>, grid, L::kThreads, L::kFwd, a.stream, p, a.s.dv);
}
template <int DK, int DS>
cudaError_t chain_bwd_for(const ChunkArgs& a, const Ptrs& p) {
    typedef ChainPlanes<DK, DS> L;
    const int grid = a.s.B * a.s.H * (a.s.dv / DS);
    if (grid <= kSMs) return launch(k_chain_bwd<DK, DS, true>, grid, L::kThreads + kLoaders, L::kBwd, a.stream, p, a.s.dv);
    return launch(k_chain_bwd<DK, DS, false>, grid, L::kThreads, L::kBwd, a.stream, p, a.s.dv);
}
template <int DK, int DV>
cudaError_t chunk_bwd_for(const ChunkArgs& a, const Ptrs& p) {
    typedef BwdPlanes<DK, DV> L;
    return launch(k_chunk_bwd<DK, DV>, a.s.B * a.s.H * p.N, L::kThreads, L::kBytes, a.stream, p);
}

}  // namespace

#define QD_BY_DIMS(fn, a, p)                                        \
    ((a).s.dk == 128 ? fn<128, 64>(a, p) /* 128 x 128: the tcgen05 kernels */ : (a).s.dv == 128 ? fn<64, 128>(a, p) : fn<64, 64>(a, p))
#define QD_BY_SLICE(fn, a, p)                                       \
    ((a).s.dk == 128 ? ((a).L.slice == 32 ? fn<128, 32>(a, p) : fn<128, 16>(a, p)) \
                     : ((a).L.slice == 32 ? fn<64, 32>(a, p) : fn<64, 16>(a, p)))

cudaError_t split_bf16_prep(const ChunkArgs& a) { return QD_BY_DIMS(prep_for, a, make_ptrs(a)); }
cudaError_t split_bf16_chain_fwd(const ChunkArgs& a) { return QD_BY_SLICE(chain_fwd_for, a, make_ptrs(a)); }
cudaError_t split_bf16_chain_bwd(const ChunkArgs& a) { return QD_BY_SLICE(chain_bwd_for, a, make_ptrs(a)); }
cudaError_t split_bf16_chunk_bwd(const ChunkArgs& a) { return QD_BY_DIMS(chunk_bwd_for, a, make_ptrs(a)); }

}  // namespace qd
