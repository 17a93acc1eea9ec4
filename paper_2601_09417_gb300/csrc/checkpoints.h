// Checkpoint memory of a plan whose backward walks list segments (host only).
#pragma once

#include <algorithm>
#include <cstdint>

namespace vbm {

constexpr int64_t kCheckpointPairsPerItem = 2;
constexpr int64_t kCheckpointBytes = 1ll << 30;
constexpr int64_t kCheckpointFreeShare = 16;
constexpr int64_t kFinePairs = 1 << 19, kFineSlots = 1024;

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
//
// fine: segments that the library has chosen short.  The few splats of such a
// batch are wide (20,000 on 1 x 1000^2: 3 to 4 pairs an item with 16 x 16 tiles, 7
// to 10 with 8 x 8, whose slots are a quarter), and a long list that finds no slot
// holds up the whole backward: with two pairs an item the step of 100,000 splats
// on 1 x 1000^2 took 455 us (16 x 16 tiles) and 579 (8 x 8), with up to kFinePairs
// more and kFineSlots, counted in slots of 256 pixels (38 MB at most), 335 and 356.
inline int64_t checkpoint_slots(int64_t items, int64_t tiles, int64_t pairs, int64_t tile_px, int seg_len,
                                bool recompute, int64_t max_bytes, bool fine = false)
{
    const int64_t held = kCheckpointPairsPerItem * items + (fine ? std::min(4 * items, kFinePairs) : 0);
    const int64_t boundaries = (held + seg_len - 1) / seg_len + (fine ? kFineSlots : 0);
    const int64_t want = (fine ? boundaries * std::max<int64_t>(1, 256 / tile_px) : boundaries) + (recompute ? tiles : 0);
    const int64_t usable = (pairs + seg_len - 1) / seg_len * (recompute ? 2 : 1);
    return std::max<int64_t>(1, std::min({want, usable, max_bytes / (tile_px * 16)}));
}

}  // namespace vbm
