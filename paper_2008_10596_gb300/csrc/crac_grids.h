// Rules that cut a pass into work for the device: segment sizes, work per warp
// and grids, by sizes alone.  Plain host code, so that a test can run it anywhere.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define CRAC_HD __host__ __device__
#else
#define CRAC_HD
#endif

namespace crac {

constexpr uint64_t kHashWarps = 8;         // warps of a hash CTA
constexpr uint64_t kSmallIters = 2;        // 512 B - 4 KiB chunks: iterations per warp,
constexpr uint64_t kSmallItersRead = 16;   // ... at most, where the pass mostly reads

// log2 of the hash kernel's segment (at most the chunk) for n_chunks chunks of
// `bytes` tracked bytes; copy: every chunk is also written.  Not for chunks of
// 512 B - 4 KiB.
//   8 KiB; 16 KiB where the pass is large enough that every SM still gets dozens of
// CTAs, and mostly reads (4 GiB, read only: 623 -> 600 us; writing every chunk 1211
// -> 1234) or writes chunks of 2 MiB and more: with fewer chunks than CTAs, all of
// them add to the same few sums, one after another (4 GiB in chunks of 16 MiB: 1557
// -> 1272 us, of 4 MiB 1351 -> 1272).  Where a chunk holds less than 8 KiB on average
// (allocations much shorter than a chunk), up to 64 KiB, so that the segments past
// an allocation's end, whose look-up costs as much as any other's, are few (50000
// allocations below 512 B in 64 KiB chunks, hash kernel: 469 us in segments of
// 8 KiB, 49 whole).
inline uint32_t split_hash_seg(uint64_t n_chunks, uint64_t bytes, uint32_t log2_chunk, bool copy) {
    const bool brief = (copy && log2_chunk < 21) || (bytes >> 14) < 32768;
    const uint32_t m = (bytes >> 13) < n_chunks ? 16 : brief ? 13 : 14;
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

// Whether the dense placement takes its room once per CTA instead of once per warp
// and 4 KiB.  With a fraction f of the chunks dirty at random, 4 KiB of n chunks hold
// a dirty one with probability p = 1 - (1 - f)^n, and the one counter takes about
// 400 million additions a second once they queue up: from some p on they set the
// pace, while the CTA's two barriers cost 7 - 10%.  A delta's device time, per warp and
// per CTA: 512 B chunks 4.5% dirty (p = 0.31) 2 GiB 430 and 469 us, 8 GiB 2190 and 1801,
// 10% 2 GiB 840 and 485; 1 KiB 10% (0.34) 398 and 439, 13% 682 and 446; 2 KiB 20% (0.36)
// 401 - 619 and 427.  4 KiB chunks, whose passes are the shortest, from p = 0.22 (24.5%:
// 2 GiB 402 and 430, 8 GiB 1723 and 1628).
inline bool dense_by_cta(float f, uint32_t log2_chunk) {
    float clean = 1.f;
    for (uint32_t i = 0; i < (4096u >> log2_chunk); ++i) clean *= 1.f - f;
    return clean < (log2_chunk < 12 ? 0.70f : 0.78f);
}

// log2 of the items of each of n chunks (2^log2_parts parts of 2^log2_part bytes)
// that hold `bytes` bytes together; item s takes parts s, s + items, ... of what its
// chunk holds.
//   An item per part; where nearly all parts lie past the end of an allocation, as many
// (at least 8, or as take four parts each) as `lanes` lanes look up in one round: empty
// items cost as much of a look-up as others, while a chunk's parts in one item are
// copied or coded one after another.  20000 allocations below 4 KiB, all dirty,
// a delta: 481 -> 134 us in chunks of 1 MiB, 1448 -> 135 in chunks of 4 MiB; coded
// 2267 -> 276 in the latter.
CRAC_HD inline uint32_t chunk_items(uint64_t n, uint64_t bytes, uint32_t log2_part, uint32_t log2_parts,
                                    uint64_t lanes) {
    if ((n << log2_parts) <= 32 * (bytes >> log2_part) + 3 * n) return log2_parts;
    uint32_t s = log2_parts < 5 ? (log2_parts < 2 ? 0 : log2_parts - 2) : 3;
    while (s < log2_parts && (n << (s + 1)) <= lanes) ++s;
    return s;
}

// How a restore's scatter is cut: parts of 1 << log2_part bytes of the target's
// chunks (a short chunk whole), and the grid that takes them.
//   A plain chunk is cut into parts of 8 KiB, and a warp takes about 8 KiB of
// short chunks.  Coded chunks are cut into parts of 32 KiB, and at most
// sixteen, as every part checks the whole stream's headers (also in host
// images, where the parts share them in L2: 16 MiB of bf16 in chunks of
// 1 MiB 992 -> 107 us against a warp per chunk).  Where a chunk holds less than
// 8 KiB on average (allocations much shorter than a chunk), both are up to 64 KiB.
//   Parts past an allocation's end cost a look-up, a chain of dependent loads, and
// no more, so where they are many a warp takes as many parts as hold a part's
// bytes on average and looks up 32 at a time (at least 32 warps per SM; coded:
// `lanes`, where chunks are short or allocations much shorter than they are and so most
// parts empty: a part's decoding takes long, and of parts looked up together a warp
// decodes one after another; 1200 ragged allocations of 80 KB on average, 4 MiB chunks:
// 234 us without, 268 with).  Whole restores, device
// time: 1200 allocations of 64 bytes in 16 MiB chunks 775 us with a warp per part
// of 8 KiB, 25 so; 20000 below 4 KiB in 1 MiB chunks 1205 and 74; 64 of 8 MiB and
// 20000 below 512 B in 64 KiB chunks 371 and 242.
//   An odd grid, where chunks have more parts than a CTA warps, so that the parts
// with bytes, the first of a chunk, fall to all CTAs.
struct RestoreCut {
    uint32_t log2_part, ctas;
    bool lanes;
};
inline RestoreCut restore_cut(uint64_t n_chunks, uint64_t bytes, uint32_t log2_chunk, bool coded, int sm_count,
                              uint64_t max_ctas) {
    const uint32_t l = log2_chunk, few = (bytes >> 13) < n_chunks ? 16 : coded ? 15 : 13;
    uint32_t part = l < few ? l : few;
    if (coded && part + 4 < l) part = l - 4;
    const uint64_t items = n_chunks << (l - part), least = 32ull * (uint64_t)sm_count;
    const bool lanes = coded && (l < 13 || ((bytes >> 13) < n_chunks && items > 2 * ((bytes >> part) + 1)));
    uint64_t warps = items;
    if (l < 13) {
        const uint64_t some = n_chunks < least ? n_chunks : least;
        warps = ((n_chunks - 1) >> (13 - (l < 8 ? 8 : l))) + 1;
        warps = warps > some ? warps : some;
    } else if (!coded || lanes) {
        const uint64_t full = (bytes >> part) + (n_chunks >> 3);
        warps = full > least ? full : least;
        warps = warps < items ? warps : items;
    }
    uint64_t ctas = (warps + 7) / 8;
    ctas = ctas < max_ctas ? ctas : max_ctas;
    ctas = ctas < 0x7fffffffull ? ctas : 0x7fffffffull;
    if (ctas * 8 < items && l - part > 3 && ctas > 1 && ctas % 2 == 0) --ctas;
    return {part, (uint32_t)ctas, lanes};
}

}  // namespace crac
