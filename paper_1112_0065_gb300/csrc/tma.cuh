// Tiled bulk copies (tensor maps) and plain mbarrier arrivals.
#pragma once

#include "tc.cuh"

namespace dd {
namespace tc {

__device__ __forceinline__ void mbar_arrive(uint64_t *mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(mbar)) : "memory");
}

// One tiled copy (TMA) of the map's box at (x, y) from global memory into this
// CTA's shared memory (128-byte aligned), completing its whole size on mbar;
// elements outside the tensor arrive as 0.  x times the element size is a
// multiple of 16 bytes.
__device__ __forceinline__ void tensor_copy_g2s(void *dst, const void *map, int x, int y, uint64_t *mbar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(smem_addr(dst)),
        "l"(map), "r"(x), "r"(y), "r"(smem_addr(mbar))
        : "memory");
}

// A tensor map in global memory that the host wrote before this kernel becomes
// visible to the copies that this thread issues from here on.
__device__ __forceinline__ void fence_tensormap(const void *map) {
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(map) : "memory");
}

}  // namespace tc
}  // namespace dd
