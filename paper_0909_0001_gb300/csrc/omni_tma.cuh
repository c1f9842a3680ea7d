#pragma once
// omni_tma.cuh -- tensor-map copies of the per-sample spectra and the bounded
// mbarrier waits behind them (the cross-spectrum kernels).
#include "omni_internal.h"

#include <cuda.h>            // CUtensorMap; the encoder is fetched from the driver at run time
#include <cudaTypedefs.h>

#include <mutex>

namespace omni {

constexpr long long kWaitCycles = 4000000000LL;   // ~2 s
constexpr long long kTestWaitCycles = 1000000LL;  // the forced-expiry test hook: ~0.5 ms

// The barrier operations are memory barriers for the compiler too: loads of a stage stay
// behind the wait for it, and stores and loads of a stage before its release.
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" :: "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, long long budget = kWaitCycles) {
    const long long t0 = clock64();
    for (;;) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}\n" : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (done) return true;
        if (clock64() - t0 > budget) return false;
    }
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Orders this thread's shared-memory accesses so far before asynchronous copies that a
// later barrier lets another thread issue (a stage that is read, then filled again).
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// One box of the 3-D tensor map into shared memory, completing on bar.
__device__ __forceinline__ void tma_load3(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4}], [%5];"
                 :: "r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z),
                    "r"(smem_u32(bar))
                 : "memory");
}

// 3-D map of the spectra [samples][tiles][2K floats]; a box (x: box_x floats of
// one tile's spectrum, y: box_y tiles, z: box_z samples) lands as [z][y][x].  Past
// the end of an axis a box reads zeros.
inline cudaError_t encode_spectra_map(const void* src, int64_t K, int64_t NT, int64_t samples, int box_x, int box_y,
                                      int box_z, CUtensorMap* map) {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    });
    if (!encode) return cudaErrorNotSupported;
    const cuuint64_t dims[3] = {(cuuint64_t)(2 * K), (cuuint64_t)NT, (cuuint64_t)samples};
    const cuuint64_t strides[2] = {(cuuint64_t)(K * 8), (cuuint64_t)(NT * K * 8)};
    const cuuint32_t box[3] = {(cuuint32_t)box_x, (cuuint32_t)box_y, (cuuint32_t)box_z};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(src), dims, strides, box,
                              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace omni
