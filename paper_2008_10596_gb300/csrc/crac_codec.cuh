// CRZ1, the chunk codec of coded images: device helpers shared by the
// encoder (crac_codec.cu) and the restore kernels (crac_restore.cu).
//
// The paper times its checkpoints with DMTCP's gzip turned off (Sec. 4.4.1,
// "Checkpoint overhead"), so it has no codec; CRZ1 is this project's.  One
// chunk of L bytes is cut into nb = L / 512 blocks and a tail of L % 512
// bytes.  A block is 128 little-endian u32 words; every byte of every word
// is rotated left by one bit (a float's sign moves to the byte's bottom), and
// byte p of the 128 rotated words forms plane p.  Each plane is stored as
// its minimum m_p and the offsets from it in W_p = bitlength(max - m_p) bits:
// header word h = sum m_p << 8p + sum W_p << (32 + 4p), then, for p = 0..3
// and j < W_p, a 16-byte unit of four words q = 0..3 whose bit l is bit j
// of plane value 4l + q.  A stream is the nb header words (zero-padded to 16
// bytes), the blocks' units in order, then the tail; a chunk whose stream
// would not be shorter than L is stored as itself.
//
// Warp layout: lane 8q + t holds words 32g + 4t + q, g = 0 .. 3, of a block
// (four 4-byte accesses, each covering one 128-byte line across the warp).
// Gathering byte p of its four words gives the lane's plane-p word: byte g =
// value 4(8g + t) + q.  Swapping the lane bits t with the bit positions j inside
// each byte (an 8x8 bit transpose per byte, three shuffles) leaves lane 8q + j
// with word q of the plane's unit j.  (From 16-byte loads, lane l holding words
// 4l .. 4l+3, the same step is a 32x32 transpose of five shuffles.)
#pragma once

#include "crac_device.cuh"

namespace crac {
namespace {

constexpr uint32_t kCrzBlock = 512;
constexpr int kCrzDecodeGroup = 4;                           // blocks decoded per step
constexpr int kCrzDecodeSlots = 2;                           // steps whose units are on their way or in use
constexpr int kCrzDecodeScratch = 512 * kCrzDecodeGroup * kCrzDecodeSlots;   // shared bytes per decoding warp

// (a & ~mask) | (b & mask), one three-input logic operation.
__device__ __forceinline__ uint32_t crz_select(uint32_t a, uint32_t b, uint32_t mask) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xD8;" : "=r"(d) : "r"(a), "r"(b), "r"(mask));
    return d;
}

__device__ __forceinline__ uint32_t crz_rot(uint32_t w) { return crz_select(w << 1, w >> 7, 0x01010101u); }

__device__ __forceinline__ uint32_t crz_unrot(uint32_t r) { return crz_select(r >> 1, r << 7, 0x80808080u); }

__device__ __forceinline__ uint32_t crz_width(uint64_t h, int p) {
    return (uint32_t)(h >> (32 + 4 * p)) & 15u;
}

__device__ __forceinline__ uint32_t crz_width_sum(uint64_t h) {
    return crz_width(h, 0) + crz_width(h, 1) + crz_width(h, 2) + crz_width(h, 3);
}

// Running sums of a block's widths: byte p = W_0 + .. + W_p, the end of plane
// p's units (widths of at most 8: every sum fits its byte).
__device__ __forceinline__ uint32_t crz_ends(uint64_t h) {
    const uint32_t w = (uint32_t)(h >> 32);
    return ((w & 15u) | (w & 0xF0u) << 4 | (w & 0xF00u) << 8 | (w & 0xF000u) << 12) * 0x01010101u;
}

// Header words of nb blocks, zero-padded to 16 bytes.
__device__ __forceinline__ uint64_t crz_head_bytes(uint64_t nb) { return 16ull * ((nb + 1) >> 1); }

// The calling lane's four words of the block at p (any address; the raw
// payload is byte-aligned after a chunk whose length is not a multiple of 4,
// and up to 3 bytes past the block are then read: the staging slack).
__device__ __forceinline__ void crz_load_words(const uint8_t *p, int lane, uint32_t w[4]) {
    const uint32_t m = (uint32_t)(uintptr_t)p & 3u;   // warp-uniform
    const uint32_t *s = reinterpret_cast<const uint32_t *>(p - m) + 4 * (lane & 7) + (lane >> 3);
    if (m == 0) {
#pragma unroll
        for (int g = 0; g < 4; ++g) w[g] = s[32 * g];
    } else {
#pragma unroll
        for (int g = 0; g < 4; ++g) w[g] = __funnelshift_r(s[32 * g], s[32 * g + 1], 8 * m);
    }
}

// 4x4 byte transpose: byte g of out[p] = byte p of in[g].  Turns a lane's
// four rotated words into its four plane words, and back.
__device__ __forceinline__ void crz_bytes_transpose(const uint32_t in[4], uint32_t out[4]) {
    const uint32_t t01 = __byte_perm(in[0], in[1], 0x5140), t23 = __byte_perm(in[2], in[3], 0x5140);
    const uint32_t u01 = __byte_perm(in[0], in[1], 0x7362), u23 = __byte_perm(in[2], in[3], 0x7362);
    out[0] = __byte_perm(t01, t23, 0x5410);
    out[1] = __byte_perm(t01, t23, 0x7632);
    out[2] = __byte_perm(u01, u23, 0x5410);
    out[3] = __byte_perm(u01, u23, 0x7632);
}

// Per-lane constants of the bit transpose: for each butterfly stage (distance
// s = 4, 2, 1) the rotation that brings the partner's bit groups into place
// and the mask of the groups this lane keeps.
struct CrzLane {
    uint32_t amt[3], keep[3];
};

__device__ __forceinline__ CrzLane crz_lane(int lane) {
    constexpr uint32_t kMask[3] = {0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
    CrzLane L;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const uint32_t s = 4u >> i;
        const bool hi = (lane & s) != 0;
        L.amt[i] = hi ? 32u - s : s;   // rotate left by s, or right by s
        L.keep[i] = hi ? ~kMask[i] : kMask[i];
    }
    return L;
}

// Lane bits t swapped with the bit positions j of each byte: on entry lane
// 8q + t holds byte g, bit j at 8g + j; on return lane 8q + j holds it at bit
// 8g + t.  Three butterfly stages, each swapping the off-diagonal halves of
// every 2s x 2s block: the partner's word rotated by s towards this lane's
// half, merged under the keep mask (a shuffle, a funnel shift and one
// three-input logic operation per stage).
__device__ __forceinline__ uint32_t crz_transpose_stage(uint32_t v, const CrzLane &L, int i) {
    const uint32_t x = __shfl_xor_sync(kFull, v, 4 >> i);
    const uint32_t r = __funnelshift_l(x, x, L.amt[i]);
    return (v & L.keep[i]) | (r & ~L.keep[i]);
}
__device__ __forceinline__ uint32_t crz_transpose(uint32_t v, const CrzLane &L) {
#pragma unroll
    for (int i = 0; i < 3; ++i) v = crz_transpose_stage(v, L, i);
    return v;
}

__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// Minima (byte p of *mins) and maxima of the planes of the block whose rotated
// words are spread over the warp, four a lane in any order.  Planes 0 and 2
// (the even bytes) and 1 and 3 (the odd bytes) are reduced in pairs as 16-bit
// halves, then across the warp: the pair as it is gives the upper half's
// extreme, its lower half alone the other's.  Whole warp.
__device__ __forceinline__ void crz_block_range(const uint32_t r[4], uint32_t *mins, uint32_t *maxs) {
    uint32_t e[4], o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        e[q] = r[q] & 0x00FF00FFu;                   // bytes 0, 2 -> 16-bit halves
        o[q] = __byte_perm(r[q], 0u, 0x4341);        // bytes 1, 3 -> 16-bit halves
    }
    const uint32_t emin = min_u16x2(min_u16x2(e[0], e[1]), min_u16x2(e[2], e[3]));
    const uint32_t emax = max_u16x2(max_u16x2(e[0], e[1]), max_u16x2(e[2], e[3]));
    const uint32_t omin = min_u16x2(min_u16x2(o[0], o[1]), min_u16x2(o[2], o[3]));
    const uint32_t omax = max_u16x2(max_u16x2(o[0], o[1]), max_u16x2(o[2], o[3]));
    const uint32_t m0 = __reduce_min_sync(kFull, emin & 0xFFFFu), m2 = __reduce_min_sync(kFull, emin);
    const uint32_t m1 = __reduce_min_sync(kFull, omin & 0xFFFFu), m3 = __reduce_min_sync(kFull, omin);
    const uint32_t M0 = __reduce_max_sync(kFull, emax & 0xFFFFu), M2 = __reduce_max_sync(kFull, emax);
    const uint32_t M1 = __reduce_max_sync(kFull, omax & 0xFFFFu), M3 = __reduce_max_sync(kFull, omax);
    // byte 0 of the first two, byte 2 of the others
    *mins = __byte_perm(__byte_perm(m0, m1, 0x0040), __byte_perm(m2, m3, 0x0062), 0x5410);
    *maxs = __byte_perm(__byte_perm(M0, M1, 0x0040), __byte_perm(M2, M3, 0x0062), 0x5410);
}

// Header word of a block with these plane minima and maxima.
__device__ __forceinline__ uint64_t crz_header(uint32_t mins, uint32_t maxs) {
    const uint32_t range = maxs - mins;   // no plane's maximum is below its minimum: no borrow
    uint32_t widths = 0;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const uint32_t d = (range >> (8 * p)) & 255u;
        widths |= (32u - (uint32_t)__clz(d)) << (4 * p);   // bit length; 0 when they are equal
    }
    return ((uint64_t)widths << 32) | mins;
}

// Units of one block from the calling lane's four words, the planes' minima and
// the ends of their units (crz_ends), both warp-uniform:
// every plane word minus the plane minimum (every byte is at least the minimum,
// so the subtraction borrows across no byte), transposed, is word q of unit j,
// which goes to out + 16 (u_p + j) + 4q when j < W_p (out 16-byte aligned).
// kScratch: through the warp's 512 bytes of shared scratch, so that lanes
// 0 .. sum(W)-1 store one 16-byte unit each -- one coalesced store per block,
// which matters when out is mapped host memory.  Whole warp.
template <bool kScratch>
__device__ __forceinline__ void crz_block_units(uint32_t mins, uint32_t ends, const uint32_t w[4], uint8_t *out,
                                                int lane, const CrzLane &L, uint8_t *scratch) {
    if (ends == 0) return;   // every plane constant: no units
    const uint32_t j = (uint32_t)lane & 7u, q = (uint32_t)lane >> 3;
    const uint32_t r[4] = {crz_rot(w[0]), crz_rot(w[1]), crz_rot(w[2]), crz_rot(w[3])};
    uint32_t P[4], col[4];
    crz_bytes_transpose(r, P);
    // All four transposes run unconditionally (a plane of width 0 stores
    // nothing), so their dependency chains interleave.
#pragma unroll
    for (int p = 0; p < 4; ++p) col[p] = crz_transpose(P[p] - __byte_perm(mins, 0u, 0x1111u * p), L);
    uint8_t *to = (kScratch ? scratch : out) + 4u * q;
    uint32_t u = 0;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const uint32_t end = __byte_perm(ends, 0u, 0x4440u + p);
        if (j + u < end) *reinterpret_cast<uint32_t *>(to + 16u * (j + u)) = col[p];
        u = end;
    }
    if (kScratch) {
        __syncwarp();
        if ((uint32_t)lane < u)
            *reinterpret_cast<uint4 *>(out + 16u * lane) = *reinterpret_cast<const uint4 *>(scratch + 16u * lane);
        __syncwarp();   // the scratch is rewritten by the next block
    }
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Decode blocks [b_begin, b_end) (and with the last one the tail) of the z-byte
// stream at src (16-byte aligned) into the len bytes at dst (4-byte aligned).
// Whole warp; scratch is the warp's kCrzDecodeScratch bytes of shared memory
// (16-byte aligned).  Every read stays inside [src, src+z) and every write
// inside [dst, dst+len).  Returns false for a stream that no chunk of len
// bytes encodes to: nothing is written when its lengths or headers are
// inconsistent (every caller checks the whole stream's), and the chunk may be
// partly written when a plane value overflows a byte.  Bound by issue slots and
// the latency of the shuffles, hence four blocks at a time: 2 GiB of fp32 in
// device images 1264 -> 760 us (one block at a time 997, two 876 us).  dst is
// 16-byte aligned.
// kHost: the stream is in mapped host memory, where asynchronous copies into
// shared memory reach 120 GB/s, ordinary loads the link's rate (190-200): the
// units then come through registers, one step ahead of their use.
template <bool kHost>
__device__ __forceinline__ bool crz_decode_warp(uint8_t *dst, const uint8_t *src, uint64_t len, uint64_t z,
                                                uint32_t b_begin, uint32_t b_end, int lane, uint8_t *scratch) {
    const uint32_t nb = (uint32_t)(len >> 9), tl = (uint32_t)len & 511u;   // chunks are at most 2^24 bytes
    const uint64_t head = crz_head_bytes(nb);
    if (nb == 0 || z >= len || z < head || ((uintptr_t)src & 15u)) return false;
    const uint64_t *H = reinterpret_cast<const uint64_t *>(src);
    uint32_t tot = 0, before = 0;   // units of all blocks, of those before b_begin
    bool bad = false;
    for (uint32_t b = lane; b < nb; b += 32) {
        const uint64_t h = H[b];
        bad |= (h >> 48) != 0;
#pragma unroll
        for (int p = 0; p < 4; ++p) bad |= crz_width(h, p) > 8u;
        const uint32_t w = crz_width_sum(h);
        tot += w;
        if (b < b_begin) before += w;
    }
    bad = __any_sync(kFull, bad);
    tot = __reduce_add_sync(kFull, tot);   // <= 32 per block, nb <= 2^15
    before = __reduce_add_sync(kFull, before);
    if (bad || head + 16ull * tot + tl != z) return false;
    const uint8_t *units = src + head;
    const uint32_t j = (uint32_t)lane & 7u, q = (uint32_t)lane >> 3;
    const CrzLane LT = crz_lane(lane);
    constexpr int kG = kCrzDecodeGroup, kN = kCrzDecodeSlots;
    bool over = false;
    if (b_end > nb) b_end = nb;
    for (uint32_t b0 = b_begin; b0 < b_end; b0 += 32) {
        // Lane l: block b0 + l's header, and its units' place in the stream.
        const uint64_t h = b0 + lane < b_end ? H[b0 + lane] : 0ull;
        const uint32_t ends = crz_ends(h), ws = ends >> 24;
        uint32_t incl = ws;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t first = before + incl - ws;
        before += __shfl_sync(kFull, incl, 31);
        // Blocks with a plane whose largest offset could pass 255 on its minimum.
        bool tight = false;
#pragma unroll
        for (int p = 0; p < 4; ++p)
            tight |= ((uint32_t)(h >> (8 * p)) & 255u) + (1u << crz_width(h, p)) - 1u > 255u;
        const unsigned checked = __ballot_sync(kFull, tight);
        const int nblk = (int)min(32u, b_end - b0);
        if (!__any_sync(kFull, ws != 0)) {   // constant planes only (zeros, say): a word repeated per block
            for (int i = 0; i < nblk; ++i) {
                const uint32_t w = crz_unrot(__shfl_sync(kFull, (uint32_t)h, i));
                __stcs(reinterpret_cast<uint4 *>(dst + 512ull * (b0 + i)) + lane, make_uint4(w, w, w, w));
            }
            continue;
        }
        // The units arrive in shared memory ahead of their use: one 16-byte
        // copy (kHost: load) per lane and block, lane k unit k.
        uint4 raw[kHost ? kG : 1];
        auto fetch = [&](int i) {
#pragma unroll
            for (int g = 0; g < kG; ++g) {
                const uint32_t n = __shfl_sync(kFull, ws, (i + g) & 31), u = __shfl_sync(kFull, first, (i + g) & 31);
                if (i + g < nblk && (uint32_t)lane < n) {
                    const uint8_t *from = units + 16ull * (u + lane);
                    if (kHost) raw[kHost ? g : 0] = *reinterpret_cast<const uint4 *>(from);
                    else cp_async16(scratch + 512 * ((i + g) % (kG * kN)) + 16 * lane, from);
                }
            }
            if (!kHost) cp_async_commit();
        };
#pragma unroll
        for (int i = 0; i < (kHost ? kG : kG * (kN - 1)); i += kG) fetch(i);
#pragma unroll 1
        for (int i = 0; i < nblk; i += kG) {
            if (kHost) {
#pragma unroll
                for (int g = 0; g < kG; ++g)   // whatever lies past a block's units is not read
                    *reinterpret_cast<uint4 *>(scratch + 512 * ((i + g) % (kG * kN)) + 16 * lane) = raw[kHost ? g : 0];
                fetch(i + kG);
            } else {
                fetch(i + kG * (kN - 1));   // (an empty group past the end)
                cp_async_wait<kN - 1>();    // this step's units have landed
            }
            __syncwarp();
            // The group's blocks step by step together, so that their chains of
            // shuffles overlap (past the end: a block of width 0, not stored).
            uint32_t mins[kG], v[kG][4];
#pragma unroll
            for (int g = 0; g < kG; ++g) {
                mins[g] = __shfl_sync(kFull, (uint32_t)h, (i + g) & 31);
                const uint32_t be = __shfl_sync(kFull, ends, (i + g) & 31);
                // lane 8q + j: word q of the plane's unit j
                const uint8_t *from = scratch + 512 * ((i + g) % (kG * kN)) + 4u * q;
                uint32_t u = 0;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const uint32_t end = __byte_perm(be, 0u, 0x4440u + p);
                    v[g][p] = j + u < end ? *reinterpret_cast<const uint32_t *>(from + 16u * (j + u)) : 0u;
                    u = end;
                }
            }
            // each lane's values' offsets from the minimum, plus the minimum
#pragma unroll
            for (int s = 0; s < 3; ++s)
#pragma unroll
                for (int g = 0; g < kG; ++g)
#pragma unroll
                    for (int p = 0; p < 4; ++p) v[g][p] = crz_transpose_stage(v[g][p], LT, s);
#pragma unroll
            for (int g = 0; g < kG; ++g) {
                uint32_t P[4], r[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) P[p] = v[g][p] + __byte_perm(mins[g], 0u, 0x1111u * p);
                if (checked && (checked >> ((i + g) & 31) & 1u)) {   // warp-uniform
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        // bytewise sum without carries between bytes, and the
                        // bytes whose sum passes 255
                        const uint32_t d = v[g][p], m4 = __byte_perm(mins[g], 0u, 0x1111u * p);
                        const uint32_t s7 = (d & 0x7F7F7F7Fu) + (m4 & 0x7F7F7F7Fu);
                        const uint32_t sum = s7 ^ ((d ^ m4) & 0x80808080u);
                        over |= (((d & m4) | ((d | m4) & ~sum)) & 0x80808080u) != 0;
                        P[p] = sum;
                    }
                }
                crz_bytes_transpose(P, r);
                if (i + g < nblk) {
                    uint32_t *to = reinterpret_cast<uint32_t *>(dst + 512ull * (b0 + i + g)) + 4u * j + q;
#pragma unroll
                    for (int k = 0; k < 4; ++k) __stcs(to + 32 * k, crz_unrot(r[k]));
                }
            }
            __syncwarp();   // the slot is refilled by the next fetch
        }
    }
    if (b_end == nb && b_begin < nb)
        for (uint32_t i = lane; i < tl; i += 32) dst[512ull * nb + i] = units[16ull * tot + i];
    return !__any_sync(kFull, over);
}

}  // namespace
}  // namespace crac
