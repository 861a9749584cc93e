// The K steps of a group of decoding warps, and the stages of packed weights ("raw" stages, SPR steps each) that hold them: the index
// arithmetic of gemm_tmw_kernel, apart from it so that the host can walk it too (tests/test_step_walk.py).
//
// GROUPS groups take every GROUPS-th step of the steps of all tiles in a row; a tile's last raw stage may hold fewer than SPR.  A wait
// asks for a PARITY, which a barrier that is two phases behind answers as well: a group may ask whether stage r is full only when it
// knows that the slot's filling before, stage r - slots, was.  A step of its own in that stage is how it usually knows.  There are
// stages without one:
// - SPR < GROUPS (weights in bytes, two steps): every third stage.  A group first waits until the slot is empty of stage r - slots,
//   which is thereby used up.  That wait is sound, because the loads are issued in order: a group has seen one of the GROUPS stages
//   before r full, so stage r - slots was issued, hence the stage before that in the slot used up (slots > GROUPS).
// - otherwise a tile's last stage of fewer than GROUPS steps.  The warp that issues the loads waits until it is full before it issues
//   the next tile's first, one of which the group has seen when it asks for the slot again.  (The first rule for these costs the
//   decoding loop 3 % at 512 x 4096 x 11008, 44.5 -> 45.2 us, 47.9 -> 49.4 with an MXInt8 result; this one nothing.)
// Asking for the full stage alone, a group whose missed load was the slower one decoded what the slot held before, and freed it.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define MX_WALK_HD __host__ __device__ __forceinline__
#else
#define MX_WALK_HD inline
#endif

namespace mx {

template <int SPR, int GROUPS> struct StepWalk {
    int kb, tile;             // the group's step within its tile
    int tile_raw;             // the tile's first raw stage
    uint32_t step;            // the step among all steps

    // kblocks, raws: steps and raw stages of a tile; stride: from one tile of this CTA to its next
    MX_WALK_HD void settle(int kblocks, int raws, int stride)
    {
        while (kb >= kblocks) { kb -= kblocks; tile += stride; tile_raw += raws; }
    }
    MX_WALK_HD uint32_t raw() const { return (uint32_t)tile_raw + (uint32_t)kb / SPR; }      // grows by at most GROUPS per turn
    static constexpr bool ASKS_EMPTY = SPR < GROUPS;
    static MX_WALK_HD bool waits_for_last(int kblocks) { return !ASKS_EMPTY && kblocks % SPR != 0 && kblocks % SPR < GROUPS; }
};

}  // namespace mx
