// lb_tma.cuh -- TMA, mbarrier and tile helpers shared by the TMA-staged step kernels.
#pragma once

#include <cuda.h>

#include "lb_internal.cuh"

namespace lbf {

// Shared memory of one CTA that steps TX x TY tiles of an FP32 lattice: the stage (nine boxes of the tile being
// loaded or pulled), the nine post-collision planes on their way out, the density tile with its
// one-node ring, and the mbarrier.
template <int TX, int TY>
struct TmaTile {
    static constexpr int XO = Elem<float>::XO;                              // 16 bytes of elements
    static constexpr int BW = TX + 2 * XO;                              // box width (elements)
    static constexpr int BH = TY + 2;                                   // box height
    static constexpr int PLANE_BYTES = BW * BH * (int)sizeof(float);
    static constexpr int PS = ((PLANE_BYTES + 127) / 128) * 128 / (int)sizeof(float);   // plane stride (elements)
    static constexpr int STAGE_BYTES = Q * PS * (int)sizeof(float);
    static constexpr uint32_t TX_BYTES = Q * PLANE_BYTES;
    static constexpr int OUT = STAGE_BYTES;                             // [plane][TY][TX]: one box of the store map
    static constexpr int OUT_BYTES = Q * TX * TY * (int)sizeof(float);
    static_assert(OUT % 128 == 0 && OUT_BYTES % 128 == 0, "boxes start on 128 bytes");
    // density tile + ring, node (lx, ly) at (ly + 1) RW + lx + 2: pairs of columns (lx even) on
    // 8-byte boundaries
    static constexpr int RW = TX + 4, RH = TY + 2;
    static constexpr int RHO = OUT + OUT_BYTES;
    static constexpr int BAR = RHO + RW * RH * 4;
    static constexpr int SMEM_BYTES = BAR + 16;
    static_assert(SMEM_BYTES % 16 == 0, "what follows is 16-byte aligned");
};

static __constant__ int kCYt[Q] = {0, 0, 1, 0, -1, 1, 1, -1, -1};

// cuTensorMapEncodeTiled of the driver, looked up once per process (thread-safe); null if
// the driver does not provide it
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn tensor_map_encoder();

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// the box of shared memory at src to a tensor (part of the calling thread's current bulk group)
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y, int z) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(z), "r"(src)
                 : "memory");
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int x, int y, int z, int w) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(z), "r"(w), "r"(src)
                 : "memory");
}

__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// the calling thread's committed stores have read their shared memory / are complete
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// orders the calling thread's accesses to shared memory with those of later TMA operations
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int w,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
        : "memory");
}

constexpr uint64_t WAIT_LIMIT_NS = 2000000000ull;   // 2 s: far beyond any healthy tile load

// Bounded wait on an mbarrier phase (false once limit_ns have passed); the decision to give
// up is made by the caller collectively (__syncthreads_or) so that no thread of the block
// is left at a barrier.
__device__ __forceinline__ bool mbar_wait_bounded_ns(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
    bool ok = mbar_try_wait(bar, parity);
    if (!ok) {
        const uint64_t t0 = global_ns();
        while (!(ok = mbar_try_wait(bar, parity)))
            if (global_ns() - t0 > limit_ns) break;
    }
    return ok;
}

__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
    return mbar_wait_bounded_ns(bar, parity, WAIT_LIMIT_NS);
}

}  // namespace lbf
