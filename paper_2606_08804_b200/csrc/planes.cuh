// Products of matrices kept in shared memory as bf16 planes: a bf16 matrix is one plane, an fp32 matrix the three planes
// x = hi + mid + lo of 8 significant bits each, split once, when it is written.  A 16 x 16 piece of a plane is one ldmatrix,
// plain or transposed, and a product of two matrices is the m16n8k16 products of their planes, without those (mid lo,
// lo mid, lo lo) that are below 2^-24 of it; accumulated in fp32.
// Against tf32 halves split by each warp that reads a fragment: as many or fewer tensor instructions (3 for 4 where one
// operand is stored in bf16, 1 for 2 where both are, 6 for 6 else) and a quarter of the others.
#pragma once
#include "sm100.cuh"
#include <cuda_bf16.h>

namespace qd {

template <int ROWS_, int W_, int NP_>
struct Planes {
    static constexpr int ROWS = ROWS_, W = W_, NP = NP_, LD = W + 8, PS = ROWS * LD;      // rows of 8 pieces on distinct banks
    static constexpr int kBytes = NP * PS * 2;
    __nv_bfloat16* p;
    __device__ __forceinline__ explicit Planes(void* q) : p(static_cast<__nv_bfloat16*>(q)) {}
    // the pair at (r, c), c even
    __device__ __forceinline__ void st2(int r, int c, float x, float y) const {
        __nv_bfloat16* d = p + r * LD + c;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const __nv_bfloat162 t = __floats2bfloat162_rn(x, y);
            *reinterpret_cast<__nv_bfloat162*>(d + i * PS) = t;
            x -= __bfloat162float(t.x); y -= __bfloat162float(t.y);
        }
    }
    // four neighbours at (r, c), c a multiple of four
    __device__ __forceinline__ void st4(int r, int c, float4 v) const {
        __nv_bfloat16* d = p + r * LD + c;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const __nv_bfloat162 s = __floats2bfloat162_rn(v.x, v.y), t = __floats2bfloat162_rn(v.z, v.w);
            *reinterpret_cast<uint2*>(d + i * PS) = make_uint2(*reinterpret_cast<const uint32_t*>(&s), *reinterpret_cast<const uint32_t*>(&t));
            v.x -= __bfloat162float(s.x); v.y -= __bfloat162float(s.y); v.z -= __bfloat162float(t.x); v.w -= __bfloat162float(t.y);
        }
    }
    __device__ __forceinline__ float2 ld2(int r, int c) const {
        const __nv_bfloat16* d = p + r * LD + c;
        float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(d + (NP - 1) * PS));
#pragma unroll
        for (int i = NP - 2; i >= 0; --i) {
            const float2 t = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(d + i * PS));
            v.x += t.x; v.y += t.y;
        }
        return v;
    }
    // a bf16 tile on its way from global memory (rows `stride` elements apart, rows >= live read as zeros), asynchronously, by TH
    // threads, of which this is number `me`
    template <int TH>
    __device__ __forceinline__ void fetch(const __nv_bfloat16* src, size_t stride, int live, int me = threadIdx.x) const {
        static_assert(NP == 1, "stored in bf16");
        constexpr int kChunks = W / 8, kTotal = ROWS * kChunks;
#pragma unroll
        for (int id = me; id < kTotal; id += TH) {
            const int row = id / kChunks, c = id % kChunks * 8;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sm100::smem_u32(p + row * LD + c)),
                         "l"(src + (row < live ? (size_t)row * stride : 0) + c), "r"(row < live ? 16 : 0) : "memory");
        }
    }
};
__device__ __forceinline__ void fetch_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// an fp32 tile on its way from global memory through registers into planes
template <int ROWS, int W, int TH>
struct FloatTile {
    static constexpr int kN = ROWS * W / 4 / TH;
    static_assert(ROWS * W / 4 % TH == 0, "bad tile");
    float4 r[kN];
    __device__ __forceinline__ void get(const float* src) {
#pragma unroll
        for (int i = 0; i < kN; ++i) r[i] = *reinterpret_cast<const float4*>(src + (i * TH + threadIdx.x) * 4);
    }
    __device__ __forceinline__ void put(const Planes<ROWS, W, 3>& d) const {
#pragma unroll
        for (int i = 0; i < kN; ++i) {
            const int e = (i * TH + threadIdx.x) * 4;
            d.st4(e / W, e % W, r[i]);
        }
    }
};

__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, const uint32_t* b) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// acc += A B for the (16 MT) x (8 NTL) tile of this warp at row m0 (pieces of 16 rows MS apart), column n0, contraction over [kb, k1):
// a triangular operand is read from or up to its diagonal only.  A is stored as [m][k], or
// as [k][m] with AT; B as [n][k], or as [k][n] with BT.  Fragments of acc: rows g and g + 8, columns 2t and 2t + 1.
// U: steps of 16 unrolled; 4 pays where a CTA has an SM's latency to itself (chains, 47.4 -> 45.5 and 55.7 -> 54.1 us at d = 64).
template <bool AT, bool BT, int U = 2, int MT, int NTL, class MA, class MB, int MS = 16>
__device__ __forceinline__ void pmm(float (&acc)[MT][NTL][4], const MA& A, const MB& B, int m0, int n0, int k1, int kb = 0) {
    static_assert(NTL % 2 == 0, "columns come in pairs of 8");
    constexpr int PA = MA::NP, PB = MB::NP;
    const int lane = threadIdx.x & 31;
    const __nv_bfloat16* pa = A.p + (AT ? ((lane & 7) + (lane >> 4) * 8) * MA::LD + m0 + ((lane >> 3) & 1) * 8
                                        : (m0 + (lane & 15)) * MA::LD + (lane >> 4) * 8);
    const __nv_bfloat16* pb = B.p + (BT ? (lane & 15) * MB::LD + n0 + (lane >> 4) * 8
                                        : (n0 + (lane & 7) + (lane >> 4) * 8) * MB::LD + ((lane >> 3) & 1) * 8);
#pragma unroll U
    for (int k0 = kb; k0 < k1; k0 += 16) {
        uint32_t a[MT][PA][4];
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int x = 0; x < PA; ++x)
                sm100::ldsm4<AT>(pa + x * MA::PS + (AT ? k0 * MA::LD + MS * i : MS * i * MA::LD + k0), a[i][x]);
#pragma unroll
        for (int j = 0; j < NTL; j += 2) {
            uint32_t b[PB][4];
#pragma unroll
            for (int y = 0; y < PB; ++y)
                sm100::ldsm4<BT>(pb + y * MB::PS + (BT ? k0 * MB::LD + 8 * j : 8 * j * MB::LD + k0), b[y]);
#pragma unroll
            for (int s = 2; s >= 0; --s)                          // smallest products first
#pragma unroll
                for (int x = 0; x < PA; ++x) {
                    if (s - x < 0 || s - x >= PB) continue;
#pragma unroll
                    for (int i = 0; i < MT; ++i) {
                        mma_bf16(acc[i][j], a[i][x], b[s - x]);
                        mma_bf16(acc[i][j + 1], a[i][x], b[s - x] + 2);
                    }
                }
        }
    }
}

}  // namespace qd
