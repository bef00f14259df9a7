// vk_tiles.cuh -- pieces shared by the kernels whose thread groups take whole-line tiles from
// a ring of slots in shared memory (sweep_tile.cu, sweep_tile16.cu, sweep_pair32.cu,
// sweep_shift32.cu, adjoint_tile.cu): 4D tensor copies and the barriers of the ring.
#pragma once

#include "vk_lines.cuh"

namespace vk {

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2,
                                            int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap *map, const void *src, int c0, int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
            reinterpret_cast<uint64_t>(map)),
        "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

// Tile k sits in slot k % S and its load completes a phase of barrier k % 2S: two barriers per
// slot, taken in turn.  A group takes every NG-th tile, so the tile before k in its slot,
// k - S, is another group's, and its load can still be in flight when the group waits for
// tile k (loads complete out of order: the group's own last tile, k - NG, can land first).
// With one barrier per slot a wait by parity then took the phase before k - S's, which has
// the parity of k's, for its own, and the group marched a slot that held no tile yet.  The
// phase before k's on its own barrier is tile k - 2S's, complete because the load of k - S was
// issued (in order, before that of k - NG) only after tile k - 2S was marched; and tile k + 2S
// cannot be loaded before tile k is marched.  (S >= NG.)
__device__ __forceinline__ uint64_t *full_bar(uint64_t *full, unsigned k, unsigned S) { return full + k % (2 * S); }
__device__ __forceinline__ bool wait_tile(uint64_t *full, unsigned k, unsigned S)
{
    return mbar_wait_bounded(full_bar(full, k, S), (k / (2 * S)) & 1u);
}

constexpr int kTileBars = 384; // bytes of barriers ahead of the velocity-column table
constexpr int kTileSlots = 12; // most slots of a ring (3 kTileSlots barriers and the groups' fit)
constexpr size_t kTileHeader = kTileBars + kMaxVel * sizeof(LineCoefT<float>);

} // namespace vk
