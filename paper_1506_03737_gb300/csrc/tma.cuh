// TMA box copies of 3-D and 4-D arrays of 8-byte elements, and the barriers that count them. Every wait is bounded.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace colapm {

constexpr long long SPIN_LIMIT = 1ll << 24;    // polls of a bounded wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
// Waits for phase `parity` of a barrier; false when the poll limit was reached.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    uint32_t done = 0;
    for (long long i = 0; i < SPIN_LIMIT && !done; ++i)
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}
// One box of a 3-D array of 8-byte elements into shared memory (x: element index, even: copies start at multiples of
// 16 bytes), counted on `bar`.
__device__ __forceinline__ void box_load(uint32_t dst, const CUtensorMap& map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(&map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void box_load4(uint32_t dst, const CUtensorMap& map, int x, int y, int z, int w, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(&map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
        : "memory");
}

// The box back out of shared memory (written there by ordinary stores), as a bulk group of the calling thread.
__device__ __forceinline__ void box_store(const CUtensorMap& map, int x, int y, int z, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];\n" ::"l"(
                     reinterpret_cast<uint64_t>(&map)),
                 "r"(x), "r"(y), "r"(z), "r"(src)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void box_store4(const CUtensorMap& map, int x, int y, int z, int w, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];\n" ::"l"(
                     reinterpret_cast<uint64_t>(&map)),
                 "r"(x), "r"(y), "r"(z), "r"(w), "r"(src)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void box_stores_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void box_stores_done() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

// Tensor map of boxes of a RANK-D array of 8-byte elements: extents, byte strides of the outer dimensions, box.
template <int RANK>
inline bool encode_box(CUtensorMap* map, void* p, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult st;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &st) != cudaSuccess || !fn) {
        (void)cudaGetLastError();
        return false;
    }
    const cuuint32_t one[4] = {1, 1, 1, 1};
    return reinterpret_cast<decltype(&cuTensorMapEncodeTiled)>(fn)(
               map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, RANK, p, dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
inline bool encode_box3(CUtensorMap* map, void* p, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box) {
    return encode_box<3>(map, p, dims, strides, box);
}

}  // namespace colapm
