// The segment plan's entries (host and device).
#pragma once
#include <stdint.h>

namespace moe {

// ---------------------------------------------------------------------------------------
// Segment plan.  The token rows of an activated expert (a "group") are cut into segments of
// at most SEG_TOKENS (or, for calls whose groups run to hundreds of rows, 2 * SEG_TOKENS)
// consecutive sorted rows, the N extent of one tensor-core instruction.
// The plan lists one entry per segment; every entry carries its whole group, so that any
// segment index leads to the group, its first segment and its number of segments.  The plan
// is derived from the grouping offsets on the device: the host never needs the
// data-dependent counts and no launch waits for a copy.
// ---------------------------------------------------------------------------------------
constexpr int SEG_TOKENS = 128;

// A segment with its group: everything a CTA needs to start on a (segment, tile) item in one
// 32-byte load.
struct alignas(16) Segment {
    int32_t expert;     // routed expert id of the group
    int32_t row0;       // first sorted row of the group
    int32_t n;          // rows of the group (all its segments together)
    int32_t first_seg;  // plan index of the group's first segment
    int32_t seg;        // plan index of this segment
    int32_t pad[3];
};

}  // namespace moe
