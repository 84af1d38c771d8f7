// TMA tensor tiles of X viewed as [F, H, W, C] (C innermost): the host-side descriptor and the 4-d tile copies.
#pragma once

#include <cuda.h>

#include "ttf_internal.cuh"
#include "ttf_async.cuh"

namespace ttf {

// Tile copies of the source rows (a) and of the window rows (b) of every clip of a launch.  A kernel parameter, so a
// launch over one clip has a type of its own: 256 bytes instead of 4 KB to hand over with every launch.
template <int G> struct ClipMaps { CUtensorMap a[G], b[G]; };

// Tile of (kc channels, bw cells, bh rows, bf frames) elements, zeros outside X; swizzle128: the 128-byte swizzle
// (kc * element size must be 128 bytes), else rows of the tile are stored plainly.  dtype 0 fp32, 1 bf16.
bool make_tensor_map(CUtensorMap* m, const void* X, int dtype, int F, int H, int W, int C, int kc, int bw, int bh, int bf,
                     bool swizzle128);

__device__ __forceinline__ void tma_load_4d(void* dst_smem, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(smem_u32(dst_smem)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
          "r"(smem_u32(bar))
        : "memory");
}
// the same copy with an L2 cache policy (createpolicy) on the lines it reads
__device__ __forceinline__ void tma_load_4d_hint(void* dst_smem, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                                 uint64_t* bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
        ::"r"(smem_u32(dst_smem)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
          "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void tensormap_prefetch(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

}  // namespace ttf
