// Rules that cut a pass into work for the device: segment sizes, work per warp
// and grids, by sizes alone.  Plain host code, so that a test can run it anywhere.
#pragma once

#include <cstdint>

namespace crac {

constexpr uint64_t kHashWarps = 8;         // warps of a hash CTA
constexpr uint64_t kSmallIters = 2;        // 512 B - 4 KiB chunks: iterations per warp,
constexpr uint64_t kSmallItersRead = 16;   // ... at most, where the pass mostly reads

// log2 of the hash kernel's segment (at most the chunk) for n_chunks chunks of
// `bytes` tracked bytes; copy: every chunk is also written.  Not for chunks of
// 512 B - 4 KiB.
//   8 KiB; 16 KiB where the pass mostly reads and is large enough that every SM
// still gets dozens of CTAs (4 GiB, read only: 623 -> 600 us), not where it writes
// every chunk (1211 -> 1234 us).  Where a chunk holds less than 8 KiB on average
// (allocations much shorter than a chunk), up to 64 KiB, so that the segments past
// an allocation's end, whose look-up costs as much as any other's, are few (50000
// allocations below 512 B in 64 KiB chunks, hash kernel: 469 us in segments of
// 8 KiB, 49 whole).
inline uint32_t split_hash_seg(uint64_t n_chunks, uint64_t bytes, uint32_t log2_chunk, bool copy) {
    const uint32_t m = (bytes >> 13) < n_chunks ? 16 : copy || (bytes >> 14) < 32768 ? 13 : 14;
    return log2_chunk < m ? log2_chunk : m;
}

// Grid of the hash kernel, and CkptParams::slots_per_warp of that grid.
//   A warp takes one segment, or as many as hold a segment's bytes on average
// (chunks below 512 B; allocations mostly much shorter than a chunk, whose
// segments past their end are empty), as long as the grid keeps twelve CTAs per
// SM, four waves: with so little in each segment, a warp's chain of look-up and
// load is what takes the time (1200 allocations of 64 bytes in 16 MiB chunks, all
// of it in two CTAs without this bound: 23.8 ms, 12 us with it).
inline uint32_t split_hash_grid(uint64_t n_chunks, uint64_t bytes, uint32_t log2_chunk, uint32_t log2_seg, bool copy,
                                int sm_count, uint32_t *slots_per_warp) {
    uint64_t per, n = n_chunks;   // items per warp, items
    if (log2_chunk >= 9 && log2_chunk < 13) {   // iterations of 4 KiB
        n = (n << log2_chunk) / 4096 + 1;
        per = copy ? kSmallIters : n >> 15;
        per = per < kSmallIters ? kSmallIters : per < kSmallItersRead ? per : kSmallItersRead;
    } else {                                    // segments
        n <<= log2_chunk - log2_seg;
        per = n / ((bytes >> (log2_seg < 13 ? 13 : log2_seg)) + 1);
        const uint64_t most = n / (kHashWarps * 12 * (uint64_t)sm_count);
        per = per < most ? per : most;
        per = per < 1 ? 1 : per < (1u << 20) ? per : (1u << 20);
    }
    *slots_per_warp = (uint32_t)per;
    const uint64_t g = (n + per * kHashWarps - 1) / (per * kHashWarps);
    return (uint32_t)(g < 1 ? 1 : g < 0x7fffffffull ? g : 0x7fffffffull);
}

}  // namespace crac
