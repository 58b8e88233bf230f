// Host side: tensor maps (TMA descriptors) of the bf16 tiles the tensor-core kernels copy, and the once-only
// shared-memory attribute of the kernels.
// Every map uses boxes of 64 elements (128 bytes) along the innermost dimension and the 128-byte
// swizzle, i.e. exactly the shared-memory operand layout described in sm100.cuh.
#include "internal.h"
#include "sm100.cuh"

#include <cudaTypedefs.h>

#include <mutex>

namespace qd {
namespace {

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess || !fn)
            return nullptr;
        encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }
    return encode;
}

}  // namespace

namespace {

// A tensor map is a pure function of the address and the extents it is made for, and a program that calls with the same
// buffers again and again asks for the same ones: each thread keeps the last map of every slot of a small table (a
// forward and backward pair needs 33).  Nothing in it belongs to anybody: an entry is only ever compared and overwritten.
struct MapKey {
    const void* base;
    uint64_t d0, d1, d2, s0, s1;
    uint32_t box_rows, rank;
    bool operator==(const MapKey& o) const {
        return base == o.base && d0 == o.d0 && d1 == o.d1 && d2 == o.d2 && s0 == o.s0 && s1 == o.s1 && box_rows == o.box_rows &&
               rank == o.rank;
    }
};
constexpr int kSlots = 256;
struct MapSlot { MapKey key; CUtensorMap map; };

bool encode_map(CUtensorMap* map, const MapKey& k) {
    thread_local MapSlot table[kSlots];           // zero to begin with, freed with the thread
    thread_local bool context = false;
    if (!context) {
        // the driver call below wants a current context, which a thread that has made no runtime call yet does not have
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaSetDevice(dev) != cudaSuccess) return false;
        context = true;
    }
    const uint64_t h = ((uint64_t)(uintptr_t)k.base ^ (k.d0 * 31 + k.d1) * 0x9E3779B97F4A7C15ull ^ ((uint64_t)k.box_rows << 40)) * 0xBF58476D1CE4E5B9ull;
    MapSlot& slot = table[h >> 56];
    if (!(slot.key == k)) {
        PFN_cuTensorMapEncodeTiled_v12000 encode = encoder();
        if (!encode) return false;
        cuuint64_t dims[3] = {k.d0, k.d1, k.d2};
        cuuint64_t strides[2] = {k.s0, k.s1};
        cuuint32_t box[3] = {64, k.box_rows, 1};
        cuuint32_t estr[3] = {1, 1, 1};
        slot.key.base = nullptr;
        if (encode(&slot.map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, k.rank, const_cast<void*>(k.base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
        slot.key = k;
    }
    *map = slot.map;
    return true;
}

}  // namespace

bool make_tmap_bf16_2d(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows, uint64_t pitch_bytes,
                       uint32_t box_rows) {
    return encode_map(map, MapKey{base, cols, rows, 1, pitch_bytes, 0, box_rows, 2});
}

bool make_tmap_tokens(CUtensorMap* map, const void* base, int B, int T, int H, int D, uint32_t box_rows) {
    const uint64_t cols = (uint64_t)H * D;
    return encode_map(map, MapKey{base, cols, (uint64_t)T, (uint64_t)B, cols * 2, (uint64_t)T * cols * 2, box_rows, 3});
}

cudaError_t set_max_smem_once(const void* kernel, size_t bytes) {
    // fixed table, no heap: the largest size set so far for each (kernel, device)
    struct Entry { const void* kernel; int dev; size_t bytes; };
    static std::mutex mu;
    static Entry table[128];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    Entry* slot = nullptr;
    for (Entry& t : table) {
        if (!t.kernel || (t.kernel == kernel && t.dev == dev)) { slot = &t; break; }
    }
    if (slot && slot->kernel && slot->bytes >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && slot) { slot->kernel = kernel; slot->dev = dev; slot->bytes = bytes; }
    return e;
}

}  // namespace qd
