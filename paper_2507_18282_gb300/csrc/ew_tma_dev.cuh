// ew_tma_dev.cuh -- mbarriers, tensor-memory-accelerator copies and their host
// side maps, shared by the TMA-staged kernels.
#pragma once

#include <cuda.h>  // CUtensorMap

#include "ew_internal.h"

namespace ew {

// the map of one 3D array of floats (x extent nx, y extent ny, `nvec` planes a
// stride of fstride floats apart, row pitch `pitch` floats): boxes of
// boxw x boxh x 1, zeros outside.  Kept in a bounded cache (ew_tma2d.cu).
ew_status field_map(const float* base, int64_t nx, int64_t ny, int64_t pitch, int nvec, int64_t fstride, int boxw,
                    int boxh, CUtensorMap* out);

__device__ __forceinline__ unsigned tma_smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tma_mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(tma_smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void tma_mbar_arrive(uint64_t* bar) {
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(tma_smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tma_mbar_arrive_expect(uint64_t* bar, unsigned bytes) {
    asm volatile(
        "{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(tma_smem_u32(bar)),
        "r"(bytes)
        : "memory");
}
__device__ __forceinline__ bool tma_mbar_try_wait(uint64_t* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(tma_smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait: gives up after about two seconds of SM clock (or 2^26 polls)
__device__ __forceinline__ bool tma_mbar_wait_bounded(uint64_t* bar, unsigned parity) {
    const long long t0 = clock64();
    for (int it = 0; it < (1 << 26); ++it) {
        if (tma_mbar_try_wait(bar, parity)) return true;
        if (clock64() - t0 > 4000000000ll) break;
    }
    return false;
}
__device__ __forceinline__ void tma_load_3d(float* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(tma_smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(tma_smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, int x, int y, int z, const float* src) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];\n" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(z), "r"(tma_smem_u32(src))
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

}  // namespace ew
