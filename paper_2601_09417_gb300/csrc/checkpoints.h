// Checkpoint memory of a plan whose backward walks list segments (host only).
#pragma once

#include <algorithm>
#include <cstdint>

namespace vbm {

constexpr int64_t kCheckpointPairsPerItem = 2;
constexpr int64_t kCheckpointBytes = 1ll << 30;
constexpr int64_t kCheckpointFreeShare = 16;

// Most bytes of checkpoints.  A plan that did not ask for persistence, which may
// never run a backward, takes at most a 16th of the memory that is free when it
// is created: what fits beside the earlier plans without checkpoints still fits.
inline int64_t checkpoint_bytes(bool persistent, int64_t free_bytes)
{
    return persistent ? kCheckpointBytes : std::min(kCheckpointBytes, free_bytes / kCheckpointFreeShare);
}

// Checkpoint slots (a pixel's 16 bytes for each of a tile's tile_px pixels):
// boundary slots for about kCheckpointPairsPerItem pairs per item (the workloads
// list about two per item before fine-tuning shrinks the splats, fewer after),
// one final-state slot per tile in recompute plans; never more than the pair
// capacity can use or max_bytes hold.
inline int64_t checkpoint_slots(int64_t items, int64_t tiles, int64_t pairs, int64_t tile_px, int seg_len,
                                bool recompute, int64_t max_bytes)
{
    const int64_t want = (kCheckpointPairsPerItem * items + seg_len - 1) / seg_len + (recompute ? tiles : 0);
    const int64_t usable = (pairs + seg_len - 1) / seg_len * (recompute ? 2 : 1);
    return std::max<int64_t>(1, std::min({want, usable, max_bytes / (tile_px * 16)}));
}

}  // namespace vbm
