// The split pass (hash -> finalize + compaction -> gather, one graph) and its
// sparse variant.
#include "crac_codec.cuh"
#include "crac_grids.h"

namespace crac {

namespace {

// ---------------------------------------------------------------------------
// Split pass: H (hash) -> F (finalize + dirty test + compaction) -> G (gather).
//
// H streams the tracked bytes with no inter-CTA dependency: every warp takes
// one segment (8 or 16 KiB, or several short chunks; crac_grids.h), in rounds of eight
// 128-bit loads per lane, sums the per-word terms, and adds the warp's sum into
// the chunk's accumulator with one 64-bit atomicAdd.  The CRAC-FP64 sum is
// taken mod 2^64, so the order of these additions does not change a bit.  The
// grid covers the segments once with ordinary CTAs: HBM serves the SMs unevenly,
// and the hardware hands CTAs to whichever SM is free, where equal shares for
// one wave of resident CTAs wait for the slowest (4 GiB in 64 KiB chunks, one
// wave of two CTAs per SM with sixteen loads per lane -> this grid with three
// CTAs per SM: 1350 -> 1207 us with every chunk written, 640 -> 591 us read only;
// of the measured copy rate 0.94 -> 1.05).  F turns each accumulator into the
// fingerprint, tests it against the baseline, and compacts the dirty chunks
// (ballot + block scan per 1024-chunk tile, decoupled look-back across
// tiles).  G copies the listed chunks into staging.  HBM traffic: B + 2D plus
// small tables, against B + D for the fused kernels, in exchange for three
// dependency-free streaming phases.
// ---------------------------------------------------------------------------
constexpr int kHashNT = 256;
static_assert(kHashNT / 32 == kHashWarps, "the grid's rule");
constexpr int kFinNT = 1024;
constexpr int kGatherNT = 256;

// A chunk of len bytes predicted at staging offset po is written there by the
// hash kernels (and then found in place by the gather) when it fits the staging
// buffer.
__device__ __forceinline__ bool spec_ok(const CkptParams &P, uint64_t po, uint64_t len) {
    return po != ~0ull && po <= P.staging_cap && len <= P.staging_cap - po;
}

// Stores of the hash kernels to an address m bytes (1 .. 15) past a 16-byte
// boundary: source vector v's bytes end up in the aligned destination vectors
// v (its first 16 - m bytes) and v + 1.  A lane builds destination vector v
// from its own source vector and the one before, which the lane before it
// holds (prev); the first 16 - m bytes and the last ones, which share their
// destination vectors with the neighbouring segments, go byte by byte.  A FULL
// pass over allocations of any byte size so reads each byte once (1 GiB in 200
// allocations, 64 KiB chunks: hash 175 us + gather 331 us -> hash 310 us).
__device__ __forceinline__ uint4 shfl_vec(uint4 v, int from) {
    return make_uint4(__shfl_sync(kFull, v.x, from), __shfl_sync(kFull, v.y, from), __shfl_sync(kFull, v.z, from),
                      __shfl_sync(kFull, v.w, from));
}
__device__ __forceinline__ void store_shifted(uint8_t *dst, uint32_t m, uint32_t v, uint32_t nv, uint4 prev, uint4 cur) {
    if (v >= 1 && v < nv) __stcs(reinterpret_cast<uint4 *>(dst - m) + v, bytes_from(prev, cur, 16u - m));
}
// The bytes that store_shifted leaves, by `n` lanes (lane l): before the first
// destination vector and after the last.  Also right for m == 0 (the tail).
__device__ __forceinline__ void store_ends(uint8_t *dst, const uint8_t *src, uint32_t m, uint32_t nv, uint32_t len,
                                           uint32_t l, uint32_t n) {
    const uint32_t front = m ? min(16u - m, len) : 0u;
    for (uint32_t b = l; b < front; b += n) dst[b] = src[b];
    for (uint32_t b = (nv ? 16u * nv - m : front) + l; b < len; b += n) dst[b] = src[b];
}

// Whether the hash kernel writes every chunk at its uncompacted offset.
__device__ __forceinline__ bool copies_all(const CkptParams &P) {
    return P.full_copy && (P.full_flag == nullptr || *P.full_flag);
}

// CRZ1 header words of the first n (at most 8) blocks of q (block u: q[u]
// across the warp) to hdr[0 .. n).  Lane u keeps block u's ranges, so that the
// header words are put together once for the eight, and stored together
// (a FULL pass that makes them and writes staging, 2 GiB: 739 -> 662 us, against
// 600 without headers; one that only makes them 535, against 312.  Reducing
// several blocks' extremes together by shuffles, without reduction
// instructions, gave 520 there and lost as much on deltas to its registers).
__device__ __forceinline__ void block_headers(const uint4 q[8], uint32_t n, int lane, uint64_t *__restrict__ hdr) {
    uint32_t mins = 0, maxs = 0;
#pragma unroll
    for (uint32_t u = 0; u < 8; ++u) {
        if (u < n) {   // warp-uniform
            const uint32_t r[4] = {crz_rot(q[u].x), crz_rot(q[u].y), crz_rot(q[u].z), crz_rot(q[u].w)};
            uint32_t m, M;
            crz_block_range(r, &m, &M);
            if (lane == (int)u) mins = m, maxs = M;
        }
    }
    if (lane < 8 && (uint32_t)lane < n) hdr[lane] = crz_header(mins, maxs);
}

// Partial CRAC-FP64 sum of a segment (<= 64 KiB) whose first word is word j0
// of its chunk, over the lanes of one warp.  dest(), asked for once the first
// loads are on their way, says where the segment's bytes are also stored (null:
// nowhere); then (kHdr) the CRZ1 header word of each whole 512-byte block of
// the segment goes to hdr[block] (lane l holds bytes 16l .. 16l+15 of block u
// in q[u], the encoder's layout of a block).  Only chunks written to staging
// get headers, so their cost follows the dirty bytes.  kAny: the destination may
// have any alignment (else a multiple of 16, and the segment's length too).  U:
// vectors per lane and round.
template <bool kHdr, bool kAny, int U, class Dest>
__device__ __forceinline__ uint64_t hash_seg(const uint8_t *__restrict__ src, uint32_t len, uint32_t j0, int lane,
                                             Dest &&dest, uint64_t *__restrict__ hdr, bool store) {
    const uint4 *p = reinterpret_cast<const uint4 *>(src);
    const uint32_t nv = len >> 4;
    uint64_t acc = 0;
    uint64_t key = (uint64_t)(j0 + 2u * lane + 1u) * kK1;
    constexpr uint64_t kStep = 64ull * kK1;
    uint8_t *copy_to = nullptr;
    uint32_t m = 0;               // kAny: copy_to's bytes past a 16-byte boundary
    uint4 last = make_uint4(0u, 0u, 0u, 0u);   // kAny: the previous round's last vector of this lane
#pragma unroll 1
    for (uint32_t v0 = 0; v0 < nv || v0 == 0; v0 += 32 * U) {   // warp-uniform
        uint4 q[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (v0 + 32u * u + lane < nv) q[u] = __ldg(p + v0 + 32u * u + lane);
        if (v0 == 0) {
            copy_to = dest();
            if (kAny && store) m = (uint32_t)(uintptr_t)copy_to & 15u;
        }
        if (kAny && m) {   // warp-uniform
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint4 prev = shfl_vec(lane == 31 ? (u ? q[u - 1] : last) : q[u], (lane + 31) & 31);
                store_shifted(copy_to, m, v0 + 32u * u + lane, nv, prev, q[u]);
            }
            last = q[U - 1];
        } else if (copy_to && store) {   // the vectors also go straight to staging
            uint4 *to = reinterpret_cast<uint4 *>(copy_to) + v0 + lane;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (v0 + 32u * u + lane < nv) __stcs(to + 32u * u, q[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (v0 + 32u * u + lane < nv) {
                acc += mixw(((uint64_t)q[u].y << 32) | q[u].x, key);
                acc += mixw(((uint64_t)q[u].w << 32) | q[u].z, key + kK1);
            }
            key += kStep;
        }
        if (kHdr && copy_to) {
            block_headers(q, (len >> 9) - (v0 >> 5), lane, hdr + (v0 >> 5));
        }
    }
    const uint32_t rem = len & 15u;
    if (rem && lane == (int)(nv & 31u)) {
        const uint8_t *t = src + 16ull * nv;
        uint64_t w0 = 0, w1 = 0;
        for (uint32_t b = 0; b < rem; ++b) {
            const uint64_t byte = t[b];
            if (b < 8) w0 |= byte << (8 * b);
            else w1 |= byte << (8 * (b - 8));
        }
        const uint64_t kt = (uint64_t)(j0 + 2u * nv + 1u) * kK1;
        acc += mixw(w0, kt);
        if (rem > 8) acc += mixw(w1, kt + kK1);
    }
    if (kAny && copy_to && store && (m | rem)) store_ends(copy_to, src, m, nv, len, lane, 32);
    return acc;
}

// One warp copies a chunk of len bytes from src (16-byte aligned) to dst and
// stores the CRZ1 header word of each whole 512-byte block b at hdr[b], in the
// encoder's layout (lane l holds bytes 16l .. 16l+15 of the block).  A dst off
// the 16-byte grid is copied by copy_group, which re-reads the (cached) source.
// (!store: headers only).
template <bool kAligned>
__device__ __forceinline__ void copy_with_headers(uint8_t *__restrict__ dst, const uint8_t *__restrict__ src,
                                                  uint64_t len, int lane, uint64_t *__restrict__ hdr, bool store) {
    const uint64_t nb = len >> 9;
    const uint4 *s = reinterpret_cast<const uint4 *>(src);
    uint4 *d = reinterpret_cast<uint4 *>(dst);
    const bool vec = kAligned || ((uintptr_t)dst & 15u) == 0;
    constexpr int U = 8;
    for (uint64_t b = 0; b < nb; b += U) {   // warp-uniform
        uint4 q[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (b + u < nb) q[u] = __ldg(s + 32 * (b + u) + lane);
        if (vec && store) {
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (b + u < nb) __stcs(d + 32 * (b + u) + lane, q[u]);
        }
        block_headers(q, (uint32_t)(nb - b), lane, hdr + b);
    }
    if (!store) return;
    if (vec) copy_group<32, true>(dst + (nb << 9), src + (nb << 9), len - (nb << 9), lane);
    else copy_group<32>(dst, src, len, lane);
}

// U = 1: chunks below 512 B, a warp each (bound by the issue slots of the other seven
// vectors when they had the eight of longer ones: 1 GiB in chunks of 256 B, a clean
// pass 1790 -> 1190 us, FULL 1723 -> 1157).
template <bool kHdr, bool kAny, int U>
__global__ void __launch_bounds__(kHashNT, U > 1 ? 3 : 4)
split_hash_kernel(const CkptParams P, unsigned long long *__restrict__ acc, uint32_t log2Seg) {
    constexpr uint32_t kWarps = kHashNT / 32;
    wait_for_producer();   // the descriptors and zeroed accumulators
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t log2S = P.log2_chunk;
    const uint32_t spc = U > 1 ? log2S - log2Seg : 0;   // log2 of segments per chunk
    // The CTA's segments in rows of one per warp, so that it streams through them.
    // Which warp starts a row turns with the chunk (with the row, where a row
    // holds whole chunks), so that allocations much shorter than a chunk, which
    // fill only its first segments, keep all warps busy.
    const uint32_t rsh = spc > 3 ? spc - 3 : 0;   // log2 of rows per chunk
    uint32_t a = 0;
    uint64_t a_next = 0;   // first chunk after allocation a
    CkptDesc d{0, 1, ~0ull, 0};
    uint32_t writes = 0;   // chunks this warp wrote speculatively
#pragma unroll 1
    for (uint32_t r = 0; r < P.slots_per_warp; ++r) {
        const uint64_t row = (uint64_t)blockIdx.x * P.slots_per_warp + r;
        const uint64_t q = row * kWarps + (U > 1 ? (warp + (uint32_t)(row >> rsh)) & (kWarps - 1) : warp);
        const uint64_t c = P.c_begin + (q >> spc);
        if (c >= P.c_end) break;
        // past allocation a's chunks (kHdr: without a register for their end)
        if (kHdr ? c - d.first_chunk > (d.bytes - 1) >> log2S : c >= a_next) {
            a = r ? find_alloc_near(P.desc, P.n_allocs, a, c, lane) : find_alloc_warp(P.desc, P.n_allocs, c, lane);
            d = P.desc[a];
            a_next = d.first_chunk + ((d.bytes - 1) >> log2S) + 1;
        }
        const uint64_t local = c - d.first_chunk;
        const uint32_t clen = (uint32_t)umin64(d.bytes - (local << log2S), 1ull << log2S);
        const uint32_t off = (uint32_t)(q & ((1ull << spc) - 1)) << log2Seg;
        if (U > 1 && off >= clen) {   // beyond the end of a short last chunk (warp-uniform): to the next chunk's rows
            const uint32_t last = (1u << rsh) - 1;
            r += last - ((uint32_t)row & last);
            continue;
        }
        const uint32_t len = min(1u << log2Seg, clen - off);
        // Direct mode (the chunk is one segment, so the warp sees all of it): the baseline
        // fingerprint is loaded before the chunk so that both latencies overlap.
        uint64_t fo = 0;
        const bool has = d.base_first != kNoBase && P.fp_old;
        if (spc == 0 && lane == 0 && has) fo = __ldg(P.fp_old + d.base_first + local);
        auto dest = [&]() -> uint8_t * {
            if (copies_all(P)) {   // FULL checkpoint: the segment's final staging offset is known
                const uint64_t o = P.alloc_prefix[a] + (local << log2S) + off - P.seg_base;
                if (o + len <= P.staging_cap) return P.staging + o;
                if (lane == 0) atomicOr(&P.ctrl->err, kErrBounds);
            } else if (P.ppos) {   // predicted dirty: written to the offset it had last time
                const uint64_t po = __ldg(P.ppos + (c - P.c_begin));
                if (spec_ok(P, po, clen)) {
                    writes += off == 0 ? 1u : 0u;
                    return P.staging + po + off;
                }
            }
            return nullptr;
        };
        const uint8_t *src = reinterpret_cast<const uint8_t *>(d.ptr) + (local << log2S) + off;
        uint64_t sum = hash_seg<kHdr, kAny, U>(src, len, off >> 3, lane, dest,
                                               kHdr ? P.crz_hdr + (c << (log2S - 9)) + (off >> 9) : nullptr,
                                               !kHdr || !P.hdr_only);
        sum = warp_sum(sum);
        if (lane == 0) {
            if (spc == 0) {
                // The warp has seen the whole chunk: finalize here and leave only
                // the length and the dirty bit for the compaction kernel.
                const uint64_t fp = fp_finalize(sum, len);
                P.fp_new[c] = fp;
                if (acc) acc[c - P.c_begin] = len | ((!has || fo != fp) ? kAccDirty : 0ull);
            } else {
                atomicAdd(acc + (c - P.c_begin), (unsigned long long)sum);
            }
        }
    }
    if (lane == 0 && writes) atomicAdd(&P.ctrl->spec_writes, (unsigned long long)writes);
}

// Hash kernel for chunks of 512 B..4 KiB: one warp iteration covers 4 KiB,
// i.e. 4096/S whole chunks, one group of LPC = S/128 lanes per chunk (8
// vectors per lane), so a warp keeps 4 KiB in flight whatever the chunk size, in
// the grid of split_hash_kernel.  A warp makes two iterations where the pass
// writes every chunk (8 GiB in 4 KiB chunks: 2741 -> 2407 us against one wave of
// resident CTAs; one iteration gives 2397, four 2453).  Where it mostly reads,
// the look-up that a warp starts with weighs more: up to sixteen, as long as
// 4096 CTAs remain (32 GiB, clean: 5502 us in one wave, 5805 with two iterations,
// 5349 with sixteen; 1 GiB 206, 212, 204 with eight).
// Every chunk is finalized in place (direct mode: acc receives the dirty
// length, and finalize only compacts).
constexpr int kSmallVecs = 8;     // vectors per lane of one iteration

template <int LPC, bool kAny>
__device__ __forceinline__ void hash_small_iter(const CkptParams &P, unsigned long long *__restrict__ acc,
                                                uint64_t c, const CkptDesc &d_warp, uint32_t a_warp,
                                                uint64_t a_next, int li, uint32_t &writes) {
    const uint32_t log2S = P.log2_chunk;
    uint64_t sum = 0, fo = 0;
    uint32_t len = 0, nv = 0;
    bool has = false;
    CkptDesc d = d_warp;
    uint32_t a = a_warp;
    uint64_t local = 0;
    uint4 q[kSmallVecs];
    const uint8_t *src = nullptr;
    uint8_t *copy_to = nullptr;
    // Sparse delta pass: the group holds its whole chunk in q until the
    // fingerprint is known and stores it only if it is dirty (B + D of HBM
    // traffic instead of B + B); clean chunks' bytes are never referenced.
    bool hold = false;
    if (c < P.c_end) {
        if (c >= a_next) {   // the segment crosses an allocation end
            a = find_alloc(P.desc, P.n_allocs, c);
            d = P.desc[a];
        }
        local = c - d.first_chunk;
        const uint64_t rest = d.bytes - (local << log2S);
        len = (uint32_t)umin64(rest, 1ull << log2S);
        has = d.base_first != kNoBase && P.fp_old;
        hold = P.sparse && has;
        if (li == 0 && has) fo = __ldg(P.fp_old + d.base_first + local);
        src = reinterpret_cast<const uint8_t *>(d.ptr) + (local << log2S);
        const uint4 *p = reinterpret_cast<const uint4 *>(src);
        nv = len >> 4;
#pragma unroll
        for (int u = 0; u < kSmallVecs; ++u) {
            const uint32_t v = li + LPC * u;
            if (v < nv) q[u] = __ldg(p + v);
        }
        uint64_t key = (2ull * (uint64_t)li + 1ull) * kK1;
        constexpr uint64_t kStep = 2ull * LPC * kK1;
#pragma unroll
        for (int u = 0; u < kSmallVecs; ++u) {
            const uint32_t v = li + LPC * u;
            if (v < nv) {
                sum += mixw(((uint64_t)q[u].y << 32) | q[u].x, key);
                sum += mixw(((uint64_t)q[u].w << 32) | q[u].z, key + kK1);
            }
            key += kStep;
        }
        if (!hold && copies_all(P)) {   // FULL checkpoint: the chunk goes straight to its staging offset
            const uint64_t o = P.alloc_prefix[a] + (local << log2S) - P.seg_base;
            if (o + len <= P.staging_cap) copy_to = P.staging + o;
            else if (li == 0) atomicOr(&P.ctrl->err, kErrBounds);
        } else if (P.ppos) {   // predicted dirty: written to the offset it had last time
            const uint64_t po = __ldg(P.ppos + (c - P.c_begin));
            if (spec_ok(P, po, len)) {
                writes += li == 0 ? 1u : 0u;
                copy_to = P.staging + po;
            }
        }
        if (copy_to && (!kAny || ((uintptr_t)copy_to & 15u) == 0)) {
#pragma unroll
            for (int u = 0; u < kSmallVecs; ++u) {
                const uint32_t v = li + LPC * u;
                if (v < nv) __stcs(reinterpret_cast<uint4 *>(copy_to) + v, q[u]);
            }
        }
        const uint32_t rem = len & 15u;
        if (rem && (uint32_t)li == (nv % LPC)) {
            const uint8_t *t = reinterpret_cast<const uint8_t *>(p + nv);
            uint64_t w0 = 0, w1 = 0;
            for (uint32_t b = 0; b < rem; ++b) {
                const uint64_t byte = t[b];
                if (b < 8) w0 |= byte << (8 * b);
                else w1 |= byte << (8 * (b - 8));
            }
            const uint64_t kt = (2ull * nv + 1ull) * kK1;
            sum += mixw(w0, kt);
            if (rem > 8) sum += mixw(w1, kt + kK1);
        }
    }
    if (kAny) {
        const uint32_t m = (uint32_t)(uintptr_t)copy_to & 15u;
        if (__any_sync(kFull, m != 0)) {   // some group's chunk lies off the 16-byte grid
            const int before = (int)(threadIdx.x & 31u) - li + (li + LPC - 1) % LPC;   // the lane before, in its group
#pragma unroll
            for (int u = 0; u < kSmallVecs; ++u) {
                const uint4 prev = shfl_vec(li == LPC - 1 && u ? q[u - 1] : q[u], before);
                if (m) store_shifted(copy_to, m, li + LPC * u, nv, prev, q[u]);
            }
        }
        if (copy_to && (m | (len & 15u))) store_ends(copy_to, src, m, nv, len, li, LPC);
    }
    // butterfly: every lane of the group ends with the group's sum
#pragma unroll
    for (int o = LPC / 2; o; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
    const uint64_t fp = fp_finalize(sum, len);
    // the group leader's baseline fingerprint, for every lane of the group
    fo = __shfl_sync(kFull, fo, (int)(threadIdx.x & 31u) - li);
    const bool dirty = !has || fo != fp;
    if (li == 0 && c < P.c_end) {
        P.fp_new[c] = fp;
        if (acc) acc[c - P.c_begin] = len | (dirty ? kAccDirty : 0ull);
    }
    if (hold && dirty) {   // sparse delta pass: sizes are multiples of 16 (no tail bytes)
        const uint64_t o = P.alloc_prefix[a] + (local << log2S) - P.seg_base;
        if (o + len <= P.staging_cap) {
            uint4 *dst = reinterpret_cast<uint4 *>(P.staging + o);
#pragma unroll
            for (int u = 0; u < kSmallVecs; ++u) {
                const uint32_t v = li + LPC * u;
                if (v < nv) __stcs(dst + v, q[u]);
            }
        } else if (li == 0) {
            atomicOr(&P.ctrl->err, kErrBounds);
        }
    }
}

template <int LPC, bool kAny>
__global__ void __launch_bounds__(kHashNT, 3)
split_hash_small_kernel(const CkptParams P, unsigned long long *__restrict__ acc, uint32_t) {
    constexpr int CPS = 32 / LPC;   // chunks per iteration
    wait_for_producer();   // the descriptors and zeroed accumulators
    const int lane = threadIdx.x & 31;
    const uint64_t warp_g = ((uint64_t)blockIdx.x * kHashNT + threadIdx.x) >> 5;
    const uint64_t n_slots = (P.c_end - P.c_begin + CPS - 1) / CPS;
    uint64_t q = warp_g * P.slots_per_warp;
    const uint64_t q_end = umin64(q + P.slots_per_warp, n_slots);
    CkptDesc d{};
    uint64_t a_next = 0;
    uint32_t a = 0;
    uint32_t writes = 0;   // chunks this lane's groups wrote speculatively (group leaders)
    for (; q < q_end; ++q) {
        const uint64_t c0 = P.c_begin + q * CPS;
        if (c0 >= a_next) {
            a = find_alloc_warp(P.desc, P.n_allocs, c0, lane);
            d = P.desc[a];
            a_next = d.first_chunk + ((d.bytes - 1) >> P.log2_chunk) + 1;
        }
        hash_small_iter<LPC, kAny>(P, acc, c0 + lane / LPC, d, a, a_next, lane % LPC, writes);
    }
    writes = __reduce_add_sync(kFull, writes);
    if (lane == 0 && writes) atomicAdd(&P.ctrl->spec_writes, (unsigned long long)writes);
}

// ---------------------------------------------------------------------------
// Sparse pass on 512 B - 4 KiB chunks with dense placement (P.sparse == 2).
// A warp hashes 4 KiB of whole chunks as split_hash_small_kernel does, holding
// them in registers, takes the room of its dirty chunks in the image from a
// running byte counter (P.ctrl->pad[0], one atomicAdd where any is dirty) and
// stores them there, back to back; the SM's other warps cover the atomic's
// round trip.  The image's span is then exactly its dirty bytes, and the group
// leaders record each chunk's offset in its accumulator word.  Sizes are
// multiples of 16 (a sparse pass requires it), so every offset is 16-byte
// aligned.  8 GiB in 4 KiB chunks, 10% dirty: 1400 -> 1330 us against a form
// that staged the dirty chunks in shared memory in one wave of resident CTAs.
// kCta: one atomicAdd for the CTA's eight warps, with two barriers for it, where
// a warp's 4 KiB likely hold a dirty chunk (dense_by_cta).
// ---------------------------------------------------------------------------
constexpr uint64_t kAccLenMask = (1ull << 24) - 1;   // accumulator word: length in bits 0-23,
constexpr int kAccPosShift = 24;                     // the chunk's offset in bits 24-62 (dense
constexpr uint64_t kAccPosMask = (1ull << 39) - 1;   // sparse placement), kAccDirty in bit 63

template <int LPC, bool kCta>
__global__ void __launch_bounds__(kHashNT, 4)
split_hash_small_dense_kernel(const CkptParams P, unsigned long long *__restrict__ acc, uint32_t) {
    constexpr int CPS = 32 / LPC;   // chunks per iteration
    wait_for_producer();   // the descriptors and zeroed accumulators
    const int lane = threadIdx.x & 31;
    const int li = lane % LPC;
    const uint32_t log2S = P.log2_chunk;
    const uint64_t warp_g = ((uint64_t)blockIdx.x * kHashNT + threadIdx.x) >> 5;
    __shared__ uint32_t s_total[2][kHashNT / 32];   // kCta: by turns
    __shared__ uint64_t s_base[2];
    uint32_t a = 0;
    uint64_t a_next = 0;
    CkptDesc dw{};
#pragma unroll 1
    for (uint32_t it = 0; it < P.slots_per_warp; ++it) {
        const uint64_t c0 = P.c_begin + (warp_g * P.slots_per_warp + it) * CPS;
        // kCta: all warps stay as long as the first, whose chunks come first, has any
        const uint64_t c_go = kCta ? c0 - (uint64_t)(threadIdx.x >> 5) * P.slots_per_warp * CPS : c0;
        if (c_go >= P.c_end) break;   // uniform over the warp (kCta: the CTA)
        if (c0 >= a_next && (!kCta || c0 < P.c_end)) {
            a = find_alloc_warp(P.desc, P.n_allocs, c0, lane);
            dw = P.desc[a];
            a_next = dw.first_chunk + ((dw.bytes - 1) >> log2S) + 1;
        }
        const uint64_t c = c0 + lane / LPC;
        uint64_t sum = 0, fo = 0;
        uint32_t len = 0, nv = 0;
        bool has = false;
        uint4 q[kSmallVecs];
        if (c < P.c_end) {
            CkptDesc d = dw;
            if (c >= a_next) d = P.desc[find_alloc(P.desc, P.n_allocs, c)];   // the iteration crosses an allocation end
            const uint64_t local = c - d.first_chunk;
            len = (uint32_t)umin64(d.bytes - (local << log2S), 1ull << log2S);
            has = d.base_first != kNoBase;
            const uint4 *p = reinterpret_cast<const uint4 *>(reinterpret_cast<const uint8_t *>(d.ptr) + (local << log2S));
            nv = len >> 4;
#pragma unroll
            for (int u = 0; u < kSmallVecs; ++u)
                if ((uint32_t)(li + LPC * u) < nv) q[u] = __ldg(p + li + LPC * u);
            if (li == 0 && has) fo = __ldg(P.fp_old + d.base_first + local);
            uint64_t key = (2ull * (uint64_t)li + 1ull) * kK1;
            constexpr uint64_t kStep = 2ull * LPC * kK1;
#pragma unroll
            for (int u = 0; u < kSmallVecs; ++u) {
                if ((uint32_t)(li + LPC * u) < nv) {
                    sum += mixw(((uint64_t)q[u].y << 32) | q[u].x, key);
                    sum += mixw(((uint64_t)q[u].w << 32) | q[u].z, key + kK1);
                }
                key += kStep;
            }
        }
#pragma unroll
        for (int o = LPC / 2; o; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
        const uint64_t fp = fp_finalize(sum, len);
        fo = __shfl_sync(kFull, fo, lane - li);
        const bool dirty = c < P.c_end && (!has || fo != fp);
        if (li == 0 && c < P.c_end) {
            P.fp_new[c] = fp;
            if (!dirty) acc[c - P.c_begin] = len;
        }
        if (!kCta && !__any_sync(kFull, dirty)) continue;
        const uint32_t mine = (li == 0 && dirty) ? len : 0u;
        uint32_t incl = mine;
        if (LPC < 32) {
#pragma unroll
            for (int o = LPC; o < 32; o <<= 1) {   // only the leaders hold a length
                const uint32_t t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
        }
        const uint32_t total = __shfl_sync(kFull, incl, 32 - LPC);   // the last leader
        const uint32_t loc = __shfl_sync(kFull, incl - mine, lane - li);
        uint64_t base = 0;
        if (kCta) {
            const int warp = threadIdx.x >> 5, turn = it & 1;
            if (lane == 0) s_total[turn][warp] = total;
            __syncthreads();
            uint32_t before = 0, all = 0;
#pragma unroll
            for (int w = 0; w < kHashNT / 32; ++w) {
                const uint32_t t = s_total[turn][w];
                if (w < warp) before += t;
                all += t;
            }
            if (threadIdx.x == 0 && all) s_base[turn] = atomicAdd(&P.ctrl->pad[0], (unsigned long long)all);
            __syncthreads();
            base = all ? s_base[turn] + before : 0;
        } else {
            if (lane == 0) base = atomicAdd(&P.ctrl->pad[0], (unsigned long long)total);
            base = __shfl_sync(kFull, base, 0);
        }
        const bool fits = base + total <= P.staging_cap;
        if (!fits && lane == 0) atomicOr(&P.ctrl->err, kErrBounds);
        if (dirty) {
            if (li == 0) acc[c - P.c_begin] = len | kAccDirty | ((fits ? base + loc : 0ull) << kAccPosShift);
            if (fits) {
                uint4 *dst = reinterpret_cast<uint4 *>(P.staging + base + loc);
#pragma unroll
                for (int u = 0; u < kSmallVecs; ++u)
                    if ((uint32_t)(li + LPC * u) < nv) __stcs(dst + li + LPC * u, q[u]);
            }
        }
    }
}

constexpr uint32_t kFinCachedAllocs = 4096;   // first_chunk columns the finalize keeps on chip

// Tiles of kItems * 1024 chunks, handed out by ticket: a thread takes kItems
// consecutive chunks, the tile's place in the list comes from a decoupled
// look-back.  A tile is a chain of round trips (ticket, accumulators, look-back,
// four barriers), so long lists use larger tiles: 2 M chunks of 4 KiB take 91 us
// in tiles of 1024, 31 in tiles of 4096, 24 in tiles of 8192 (41 where every
// chunk is listed).
template <int kItems>
__global__ void __launch_bounds__(kFinNT)
split_finalize_kernel(const CkptParams P, unsigned long long *__restrict__ acc, uint32_t log2Seg) {
    // Whole: the hash kernel saw whole chunks and has finalized them; direct: it
    // also left each one's length and dirty bit in acc (the allocation-free
    // pass has no room for that).
    const bool whole = log2Seg == P.log2_chunk, direct = whole && acc;
    // Other chunks need their allocation: searched in an on-chip copy of
    // the first_chunk column when it fits (a search in global memory is a
    // chain of dependent loads per chunk).
    __shared__ uint64_t s_first[kFinCachedAllocs];
    const bool cached = !direct && P.n_allocs <= kFinCachedAllocs;
    wait_for_producer();   // the hash kernel's accumulators
    if (cached)
        for (uint32_t a = threadIdx.x; a < P.n_allocs; a += kFinNT) s_first[a] = P.desc[a].first_chunk;
    __shared__ uint32_t s_wcnt[32];
    __shared__ uint64_t s_wbytes[32];
    __shared__ uint64_t s_wdirty[32];
    __shared__ uint64_t s_k0, s_d0;
    __shared__ uint32_t s_tile;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t log2S = P.log2_chunk;
    const uint64_t S = 1ull << log2S;
    for (;;) {
        if (threadIdx.x == 0) {
            uint32_t t = atomicAdd(&P.ctrl->ticket, 1u);
            if (P.skip_first_ticket && t == 0) t = atomicAdd(&P.ctrl->ticket, 1u);
            s_tile = t;
        }
        __syncthreads();
        const uint32_t tile = s_tile;
        if (tile >= P.n_tiles) break;
        const uint64_t c0 = P.c_begin + ((uint64_t)tile * kFinNT + threadIdx.x) * kItems;
        uint32_t dl[kItems], len[kItems];
        uint64_t dpos[kItems];   // dense sparse placement: the chunk's offset in the span
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const uint64_t c = c0 + i;
            dl[i] = len[i] = 0;
            dpos[i] = 0;
            if (c < P.c_end && direct) {
                const uint64_t v = acc[c - P.c_begin];
                len[i] = (uint32_t)(v & kAccLenMask);
                dl[i] = (v & kAccDirty) ? len[i] : 0u;
                dpos[i] = (v >> kAccPosShift) & kAccPosMask;
            } else if (c < P.c_end) {
                uint32_t a;
                if (cached) {
                    uint32_t lo = 0, hi = P.n_allocs;
                    while (hi - lo > 1) {
                        const uint32_t mid = (lo + hi) >> 1;
                        if (s_first[mid] <= c) lo = mid;
                        else hi = mid;
                    }
                    a = lo;
                } else {
                    a = find_alloc(P.desc, P.n_allocs, c);
                }
                const CkptDesc d = P.desc[a];
                const uint64_t local = c - d.first_chunk;
                len[i] = (uint32_t)min(S, d.bytes - (local << log2S));
                uint64_t fp;
                if (whole) {
                    fp = P.fp_new[c];
                } else {
                    fp = fp_finalize(acc[c - P.c_begin], len[i]);
                    P.fp_new[c] = fp;
                }
                const bool dirty = d.base_first == kNoBase || !P.fp_old || P.fp_old[d.base_first + local] != fp;
                dl[i] = dirty ? len[i] : 0u;
            }
            if (P.ppos_next && c < P.c_end) P.ppos_next[c - P.c_begin] = ~0ull;   // the gather sets the dirty ones
        }
        // Bytes that advance the staging offset: the dirty ones, or in the
        // sparse pass every chunk's (each sits at its uncompacted offset);
        // under dense placement the dirty ones, whose offsets the hash kernel
        // recorded.
        uint32_t n = 0;           // this thread's dirty chunks
        uint64_t sv = 0, td = 0;  // ... bytes that advance the offset, dirty bytes
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            n += dl[i] != 0;
            td += dl[i];
            sv += P.sparse == 1u ? len[i] : dl[i];
        }
        uint32_t incl_n = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl_n, o);
            if (lane >= o) incl_n += t;
        }
        const uint64_t incl = warp_incl_scan(sv, lane);
        if (P.sparse) {
            const uint64_t wd = warp_sum(td);
            if (lane == 0) s_wdirty[warp] = wd;
        }
        if (lane == 31) {
            s_wcnt[warp] = incl_n;
            s_wbytes[warp] = incl;
        }
        __syncthreads();
        if (P.sparse && warp == 1) {   // the tile's dirty bytes, one atomic per tile
            const uint64_t all = warp_sum(s_wdirty[lane]);
            if (lane == 0 && all) atomicAdd(&P.ctrl->payload, (unsigned long long)all);
        }
        if (warp == 0) {
            const uint32_t wc = s_wcnt[lane];
            const uint64_t wb = s_wbytes[lane];
            uint32_t ic = wc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, ic, o);
                if (lane >= o) ic += t;
            }
            const uint64_t ib = warp_incl_scan(wb, lane);
            const uint32_t cnt = __shfl_sync(kFull, ic, 31);
            const uint64_t bytes = __shfl_sync(kFull, ib, 31);
            s_wcnt[lane] = ic - wc;
            s_wbytes[lane] = ib - wb;
            uint64_t k0 = 0, d0 = 0;
            if (tile == 0) {
                if (lane == 0) {
                    st_status(P.tile_cnt, kFlagInc | cnt);
                    st_status(P.tile_bytes, kFlagInc | bytes);
                }
            } else {
                if (lane == 0) {
                    st_status(P.tile_cnt + tile, kFlagAgg | cnt);
                    st_status(P.tile_bytes + tile, kFlagAgg | bytes);
                }
                lookback(P, tile, lane, &k0, &d0);
                if (lane == 0) {
                    st_status(P.tile_cnt + tile, kFlagInc | ((k0 + cnt) & kValMask));
                    st_status(P.tile_bytes + tile, kFlagInc | ((d0 + bytes) & kValMask));
                }
            }
            if (lane == 0) {
                s_k0 = k0;
                s_d0 = d0;
                if (tile == P.n_tiles - 1) {
                    P.ctrl->k = k0 + cnt;
                    P.ctrl->D = d0 + bytes;
                    if (k0 + cnt <= P.idx_cap) P.off_out[k0 + cnt] = d0 + bytes;
                    else atomicOr(&P.ctrl->err, kErrBounds);
                }
            }
        }
        __syncthreads();
        uint64_t j = s_k0 + s_wcnt[warp] + incl_n - n, o = s_d0 + s_wbytes[warp] + incl - sv;
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            if (dl[i]) {
                if (j < P.idx_cap) {
                    P.idx_out[j] = c0 + i;
                    P.off_out[j] = P.sparse == 2u ? dpos[i] : o;
                } else {
                    atomicOr(&P.ctrl->err, kErrBounds);
                }
                ++j;
            }
            o += P.sparse == 1u ? len[i] : dl[i];
        }
        __syncthreads();
    }
}

// kHdr: P.crz_hdr is set, and each copied chunk's block headers are written
// too (a separate instance, so that the plain gather keeps its registers low).
// kAligned: every allocation's size, so every payload offset, is a multiple of
// 16 bytes.
// kMulti: an item takes several parts of its entry (chunk_items).
template <bool kHdr, bool kAligned, bool kMulti>
__global__ void __launch_bounds__(kGatherNT, kHdr ? 2 : 4)
split_gather_kernel(const CkptParams P, unsigned long long *, uint32_t) {
    wait_for_producer();         // the finalize kernel's list and counts
    if (copies_all(P)) return;   // the hash kernel has already written every chunk
    const int lane = threadIdx.x & 31;
    const uint64_t kd = (uint64_t)P.ctrl->k;
    const uint64_t k = kd < P.idx_cap ? kd : P.idx_cap;
    const uint32_t log2S = P.log2_chunk;
    const uint64_t S = 1ull << log2S;
    const uint64_t nw = ((uint64_t)gridDim.x * kGatherNT) >> 5;
    // The next pass predicts this pass's offsets, if few enough chunks are dirty.
    uint64_t *next = (P.ppos_next && 2 * kd <= P.c_end - P.c_begin) ? P.ppos_next : nullptr;
    // Every entry ends by the segment's dirty bytes, which must fit staging.
    if (blockIdx.x == 0 && threadIdx.x == 0 && P.ctrl->D > P.staging_cap) atomicOr(&P.ctrl->err, kErrBounds);
    __shared__ unsigned int s_hits;
    if (threadIdx.x == 0) s_hits = 0;
    __syncthreads();
    uint32_t hits = 0;
    // An item is an entry's 8 KiB part (a short chunk whole), a warp each, so
    // that a small payload still spreads over the chip; a warp strides over the
    // items, 32 at a time, a lane looking up each (a chain of dependent loads).
    // 96 MiB in 1200 ragged allocations, 64 KiB chunks: all of them 545 -> 36 us.
    const uint32_t log2P = log2S < 13 ? log2S : 13;
    const uint32_t parts = log2S - log2P;   // log2 of the parts of an entry, and of its items:
    const uint32_t items = kMulti ? chunk_items(k, P.ctrl->D, log2P, parts, 32 * nw) : parts;
    const uint64_t n_items = k << items;
    for (uint64_t i0 = ((uint64_t)blockIdx.x * kGatherNT + threadIdx.x) >> 5; i0 < n_items; i0 += 32 * nw) {
        const uint64_t it = i0 + lane * nw;
        uint64_t dst = 0, src = 0, blk = 0;
        uint32_t len = 0;   // bytes to copy (kMulti: of the chunk, from the item's first part on)
        if (it < n_items) {
            const uint64_t j = it >> items;
            const uint64_t po = (it & ((1ull << items) - 1)) << log2P;   // the item's offset in its entry
            const uint64_t c = P.idx_out[j];
            const uint64_t o = P.off_out[j];
            if (next && po == 0) next[c - P.c_begin] = o;
            // Written there by the hash kernel already: a predicted offset equal
            // to the entry's (the chunk fits, it ends by D).
            const uint64_t pp = P.ppos ? P.ppos[c - P.c_begin] : ~0ull;
            if (pp == o) {
                hits += po == 0 ? 1u : 0u;
            } else {
                const CkptDesc d = P.desc[find_alloc(P.desc, P.n_allocs, c)];
                const uint64_t at = (c - d.first_chunk) << log2S;
                const uint64_t clen = umin64(S, d.bytes - at);
                if (o + clen > P.staging_cap) {
                    atomicOr(&P.ctrl->err, kErrBounds);
                } else if (po < clen) {   // a short last chunk has fewer items
                    dst = o + po;
                    src = d.ptr + at + po;
                    len = (uint32_t)(kMulti ? clen - po : umin64(1ull << log2P, clen - po));
                    if (kHdr) blk = (c << (log2S - 9)) + (po >> 9);
                }
            }
        }
        unsigned todo = __ballot_sync(kFull, len != 0);
        while (todo) {   // warp-uniform
            const int i = __ffs(todo) - 1;
            todo &= todo - 1;
            uint8_t *to = P.staging + __shfl_sync(kFull, dst, i);
            const uint8_t *from = reinterpret_cast<const uint8_t *>(__shfl_sync(kFull, src, i));
            const uint32_t n = __shfl_sync(kFull, len, i);
            uint64_t *hdr = kHdr ? P.crz_hdr + __shfl_sync(kFull, blk, i) : nullptr;
            for (uint32_t at = 0; at < n; at += 1u << (log2P + items)) {
                const uint32_t part = kMulti ? min(1u << log2P, n - at) : n;
                if (kHdr) copy_with_headers<kAligned>(to + at, from + at, part, lane, hdr + (at >> 9), !P.hdr_only);
                else copy_group<32, kAligned>(to + at, from + at, part, lane);
                if (!kMulti) break;
            }
        }
    }
    hits = __reduce_add_sync(kFull, hits);
    if (lane == 0 && hits) atomicAdd(&s_hits, hits);
    __syncthreads();
    if (threadIdx.x == 0 && s_hits) atomicAdd(&P.ctrl->spec_hits, (unsigned long long)s_hits);
}

}  // namespace

const void *split_hash_fn(bool crz_headers, bool aligned, uint32_t log2S) {
    if (crz_headers)   // chunks of 8 KiB and more
        return aligned ? reinterpret_cast<const void *>(&split_hash_kernel<true, false, 8>)
                       : reinterpret_cast<const void *>(&split_hash_kernel<true, true, 8>);
    if (log2S < 9)
        return aligned ? reinterpret_cast<const void *>(&split_hash_kernel<false, false, 1>)
                       : reinterpret_cast<const void *>(&split_hash_kernel<false, true, 1>);
    return aligned ? reinterpret_cast<const void *>(&split_hash_kernel<false, false, 8>)
                   : reinterpret_cast<const void *>(&split_hash_kernel<false, true, 8>);
}
template <bool kAny>
static const void *hash_small_fn(int lanes_per_chunk) {
    switch (lanes_per_chunk) {
    case 4: return reinterpret_cast<const void *>(&split_hash_small_kernel<4, kAny>);
    case 8: return reinterpret_cast<const void *>(&split_hash_small_kernel<8, kAny>);
    case 16: return reinterpret_cast<const void *>(&split_hash_small_kernel<16, kAny>);
    case 32: return reinterpret_cast<const void *>(&split_hash_small_kernel<32, kAny>);
    default: return nullptr;
    }
}
const void *split_hash_small_fn(int lanes_per_chunk, bool aligned) {
    return aligned ? hash_small_fn<false>(lanes_per_chunk) : hash_small_fn<true>(lanes_per_chunk);
}
// Tiles of 8192 chunks once there are more tiles of 1024 than two per SM.
uint32_t split_finalize_tile(uint64_t n_chunks, int sm_count) {
    return n_chunks > 2ull * sm_count * kFinNT ? 8 * kFinNT : kFinNT;
}
const void *split_finalize_fn(uint32_t tile) {
    return tile == kFinNT ? reinterpret_cast<const void *>(&split_finalize_kernel<1>)
                          : reinterpret_cast<const void *>(&split_finalize_kernel<8>);
}
template <bool kHdr>
static const void *gather_fn(bool aligned, bool multi) {
    if (multi) return reinterpret_cast<const void *>(&split_gather_kernel<kHdr, false, true>);
    return aligned ? reinterpret_cast<const void *>(&split_gather_kernel<kHdr, true, false>)
                   : reinterpret_cast<const void *>(&split_gather_kernel<kHdr, false, false>);
}
const void *split_gather_fn(bool crz_headers, bool aligned, uint64_t n_chunks, uint64_t bytes, uint32_t log2S) {
    const uint32_t parts = log2S > 13 ? log2S - 13 : 0;
    const bool multi = chunk_items(n_chunks, bytes, 13, parts, 0) != parts;
    return crz_headers ? gather_fn<true>(aligned, multi) : gather_fn<false>(aligned, multi);
}
int split_hash_threads() { return kHashNT; }
int split_finalize_threads() { return kFinNT; }
int split_gather_threads() { return kGatherNT; }
template <bool kCta>
static const void *hash_small_dense_fn(int lanes_per_chunk) {
    switch (lanes_per_chunk) {
    case 4: return reinterpret_cast<const void *>(&split_hash_small_dense_kernel<4, kCta>);
    case 8: return reinterpret_cast<const void *>(&split_hash_small_dense_kernel<8, kCta>);
    case 16: return reinterpret_cast<const void *>(&split_hash_small_dense_kernel<16, kCta>);
    case 32: return reinterpret_cast<const void *>(&split_hash_small_dense_kernel<32, kCta>);
    default: return nullptr;
    }
}
const void *split_hash_small_dense_fn(int lanes_per_chunk, bool by_cta) {
    return by_cta ? hash_small_dense_fn<true>(lanes_per_chunk) : hash_small_dense_fn<false>(lanes_per_chunk);
}

}  // namespace crac
