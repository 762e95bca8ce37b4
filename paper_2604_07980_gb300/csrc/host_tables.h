// host_tables.h -- where a host call's tables lie in its staging block.
//
// The host entry points copy counts, frame tables and boxes to the device in one copy, so
// they lie one behind the other, as many records as the call has: a context made for many
// frames copies no more for a small call than another.  Plain C++, unit-tested on the CPU.
#pragma once

#include <stddef.h>

namespace ctm {

constexpr size_t kHostCountsBytes = 256;  // counts of the sub-batches, ahead of the frames

struct HostTables {
    size_t frames;   // frame table of the staging images
    size_t sources;  // of the caller's images (mapped calls; else empty)
    size_t boxes;
    size_t bytes;    // all of it: the call's copy
};

constexpr HostTables host_tables(size_t n_frames, size_t n_sources, size_t n_boxes, size_t frame_bytes,
                                 size_t box_bytes)
{
    HostTables t{};
    t.frames = kHostCountsBytes;
    t.sources = t.frames + n_frames * frame_bytes;
    t.boxes = (t.sources + n_sources * frame_bytes + 15) / 16 * 16;
    t.bytes = t.boxes + n_boxes * box_bytes;
    return t;
}

}  // namespace ctm
