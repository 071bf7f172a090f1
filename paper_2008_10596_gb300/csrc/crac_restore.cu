// Restart kernels: owner marks, coverage check and scatter over every piece of
// a chain (device path), and the windowed scatter of the staged path.
#include "crac_codec.cuh"
#include "crac_grids.h"

namespace crac {

namespace {

// ---------------------------------------------------------------------------
// K4 restore scatter: payload chunks -> allocations, filtered by the owner map
// so that each target chunk is written once, by the newest image holding it.
// ---------------------------------------------------------------------------
constexpr int kScatterNT = 256;
constexpr uint32_t kScatterWarps = kScatterNT / 32;

__global__ void __launch_bounds__(kScatterNT, 4) scatter_kernel(const ScatterParams P) {
    constexpr int GT = 32;
    // A resolution or bounds error found earlier on this stream (chain not
    // covering the target, index out of range) leaves memory untouched.
    if (*(volatile unsigned int *)P.err) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t S = 1ull << P.log2_chunk;
    const uint64_t n = P.j1 - P.j0;
    for (uint64_t e = (uint64_t)blockIdx.x * (kScatterNT / 32) + warp; e < n;
         e += (uint64_t)gridDim.x * (kScatterNT / 32)) {
        const uint64_t c = P.full ? P.j0 + e : P.idx[e];
        const ScatterDesc d = P.desc[find_scatter(P.desc, P.n_desc, c)];
        const uint64_t local = c - d.img_first;
        if (d.dst == 0) continue;
        const uint64_t tc = d.tgt_first + local;
        if (tc >= P.n_owner) {
            if (lane == 0) atomicOr(P.err, kErrBounds);
            continue;
        }
        if (P.owner[tc] != P.image_index) continue;
        const uint64_t len = min(S, d.bytes - (local << P.log2_chunk));
        const uint64_t o = P.full ? d.payload_base + (local << P.log2_chunk) : P.off[e];
        if (o < P.origin || o - P.origin + len > P.window) {
            if (lane == 0) atomicOr(P.err, kErrBounds);
            continue;
        }
        copy_group<GT>(reinterpret_cast<uint8_t *>(d.dst) + (local << P.log2_chunk),
                       P.payload + (o - P.origin), len, lane);
    }
}


// ---------------------------------------------------------------------------
// Chain resolution and restore on the device (R3 + R2 for device-resident
// chains), over every piece of every image of the chain in one launch each.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t find_piece(const RestorePiece *__restrict__ p, uint32_t n, uint64_t e) {
    uint32_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (p[mid].entry_base <= e) lo = mid;
        else hi = mid;
    }
    return lo;
}

// An owner word: the newest image holding a target chunk, as chain position + 1
// (bits 40 and up), and the entry that holds it (bits 0-39); 0: none, or
// nothing to restore.  atomicMax over the entries that mark a chunk leaves the
// newest image's, whatever the order of execution.
constexpr int kOwnerShift = 40;
constexpr uint64_t kOwnerEntry = (1ull << kOwnerShift) - 1;

__global__ void __launch_bounds__(256) restore_mark_kernel(const RestoreParams P) {
    wait_for_producer();
    for (uint64_t e = (uint64_t)blockIdx.x * 256 + threadIdx.x; e < P.n_entries; e += (uint64_t)gridDim.x * 256) {
        const RestorePiece pc = P.pieces[find_piece(P.pieces, P.n_pieces, e)];
        const uint64_t c = reinterpret_cast<const uint64_t *>(pc.idx)[e - pc.entry_base];
        const ScatterDesc *dd = P.desc + pc.desc_off;
        const ScatterDesc d = dd[find_scatter(dd, pc.n_desc, c)];
        if (d.dst == 0) continue;   // its allocation is not restored
        const uint64_t tc = d.tgt_first + (c - d.img_first);
        if (tc < P.n_owner) atomicMax(P.owner + tc, ((unsigned long long)(pc.image_index + 1u) << kOwnerShift) | e);
        else atomicOr(P.err, kErrBounds);
    }
}

// Every target chunk needs an owner; the target's fingerprints go to the
// context's spare table on the way (adopted only if the restore succeeds).
__global__ void __launch_bounds__(256) restore_check_kernel(const RestoreParams P) {
    wait_for_producer();
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < P.n_owner; i += (uint64_t)gridDim.x * 256) {
        P.fp_out[i] = P.fp_img[i];
        if (P.owner[i] == 0) atomicOr(P.err, kErrUncovered);
    }
}

// Incremental restore: a target chunk that already holds the image's bytes
// (same fingerprint) keeps them; clearing its owner makes the scatter skip it.
__global__ void __launch_bounds__(256) restore_unmark_kernel(const RestoreParams P) {
    wait_for_producer();
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < P.n_owner; i += (uint64_t)gridDim.x * 256)
        if (P.fp_now[i] == P.fp_img[i]) P.owner[i] = 0;
}

// The scatter: every target chunk's bytes from the entry that owns it, so each
// byte is read once and written once, in the order of the target's memory.  An
// item is 1 << P.log2_part bytes of a target chunk (or a whole short chunk), a
// warp each.  The grid covers the items once with ordinary CTAs, so that the
// hardware hands them to whichever SM is free: HBM serves the SMs unevenly, and
// a copy cut into equal shares for one wave of resident CTAs waits for the
// slowest (4 GiB in 64 KiB chunks: 1.32 ms in one wave of 5 CTAs per SM, 1.22 ms
// with a CTA for every 64 KiB).  With a smaller grid (host images, whose link
// one CTA per SM already paces; incremental restores, where most items are
// skipped; allocations much shorter than a chunk) a warp strides over the items,
// 32 at a time, a lane looking up each, and its place in the CTA turns with each
// step, so that the first parts of chunks, at times the only ones, keep all warps
// busy.
struct RestoreItem {
    uint64_t dst, src;   // raw: the item's bytes; coded: the whole chunk, its stream
    uint32_t len;        // bytes to write (0: nothing)
    uint32_t z;          // coded: the stream's length (0: stored raw)
    uint32_t po, clen;   // the item's offset in its chunk, the chunk's length
};

template <bool kCoded>
__device__ __forceinline__ RestoreItem restore_item(const RestoreParams &P, uint64_t it) {
    RestoreItem r{};
    const uint32_t parts = P.log2_chunk - P.log2_part;   // log2 of the items per chunk
    const uint64_t tc = it >> parts;
    const uint64_t po = (it & ((1ull << parts) - 1)) << P.log2_part;   // the item's offset in its chunk
    const uint64_t own = P.owner[tc];
    const ScatterDesc *d = P.tgt + find_scatter(P.tgt, P.n_tgt, tc);
    const uint64_t at = (tc - d->img_first) << P.log2_chunk;
    const uint64_t clen = umin64(1ull << P.log2_chunk, d->bytes - at);
    if (!own || po >= clen) return r;   // a short last chunk has fewer items
    const uint64_t e = own & kOwnerEntry;
    const RestorePiece *pc = P.pieces + find_piece(P.pieces, P.n_pieces, e);
    const uint64_t o = reinterpret_cast<const uint64_t *>(pc->off)[e - pc->entry_base];
    // Coded image: the entry's stream length (equal to clen when stored raw).
    const uint64_t ez = (kCoded && pc->zlen) ? reinterpret_cast<const uint64_t *>(pc->zlen)[e - pc->entry_base] : clen;
    if (o > pc->bytes || ez > pc->bytes - o) {
        atomicOr(P.err, kErrBounds);
        return r;
    }
    const bool stream = kCoded && ez != clen;
    r.dst = d->dst + at + (stream ? 0 : po);
    r.src = pc->payload + o + (stream ? 0 : po);
    r.len = (uint32_t)umin64(1ull << P.log2_part, clen - po);
    if (kCoded) {
        r.z = stream ? (uint32_t)ez : 0u;
        r.po = (uint32_t)po;
        r.clen = (uint32_t)clen;
    }
    return r;
}

// A warp's item in step j of nw warps.
__device__ __forceinline__ uint64_t restore_step(uint64_t j, uint64_t nw, int warp) {
    return j * nw + (uint64_t)blockIdx.x * kScatterWarps + ((warp + (uint32_t)j) & (kScatterWarps - 1));
}

// kAligned: every allocation's size is a multiple of 16 bytes.
template <bool kAligned>
__device__ __forceinline__ void restore_scatter_body(const RestoreParams &P) {
    wait_for_producer();
    if (*(volatile unsigned int *)P.err) return;   // uncovered or out of range: memory untouched
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t n_items = P.n_owner << (P.log2_chunk - P.log2_part);
    const uint64_t nw = (uint64_t)gridDim.x * kScatterWarps;
    for (uint64_t j = lane; (j - lane) * nw < n_items; j += 32) {   // warp-uniform
        RestoreItem r{};
        const uint64_t it = restore_step(j, nw, warp);
        if (it < n_items) r = restore_item<false>(P, it);
        unsigned todo = __ballot_sync(kFull, r.len != 0);
        while (todo) {   // warp-uniform
            const int i = __ffs(todo) - 1;
            todo &= todo - 1;
            copy_group<32, kAligned>(reinterpret_cast<uint8_t *>(__shfl_sync(kFull, r.dst, i)),
                                     reinterpret_cast<const uint8_t *>(__shfl_sync(kFull, r.src, i)),
                                     __shfl_sync(kFull, r.len, i), lane);
        }
    }
}

__global__ void __launch_bounds__(kScatterNT, 4) restore_scatter_kernel(const RestoreParams P) {
    restore_scatter_body<true>(P);
}

__global__ void __launch_bounds__(kScatterNT, 4) restore_scatter_ragged_kernel(const RestoreParams P) {
    restore_scatter_body<false>(P);
}

// Chains with a coded image: the decoder needs registers that the plain copy
// does not (hence kernels of their own).  An item of 16 KiB or more is looked up
// by the whole warp, its decoding takes far longer; kLanes: short chunks, or mostly
// empty items, 32 at a time, a lane each.
template <bool kHost, bool kLanes>
__global__ void __launch_bounds__(kScatterNT, 3) restore_scatter_coded_kernel(const RestoreParams P) {
    extern __shared__ __align__(16) uint8_t scratch[];   // kCrzDecodeScratch per warp
    wait_for_producer();
    if (*(volatile unsigned int *)P.err) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t n_items = P.n_owner << (P.log2_chunk - P.log2_part);
    const uint64_t nw = (uint64_t)gridDim.x * kScatterWarps;
    for (uint64_t j = kLanes ? lane : 0; (kLanes ? j - lane : j) * nw < n_items; j += kLanes ? 32 : 1) {   // warp-uniform
        RestoreItem mine{};
        const uint64_t it = restore_step(j, nw, warp);
        if (it < n_items) mine = restore_item<true>(P, it);
        unsigned todo = kLanes ? __ballot_sync(kFull, mine.len != 0) : mine.len != 0;
        while (todo) {   // warp-uniform
            RestoreItem r = mine;
            if (kLanes) {
                const int i = __ffs(todo) - 1;
                r.dst = __shfl_sync(kFull, mine.dst, i);
                r.src = __shfl_sync(kFull, mine.src, i);
                r.len = __shfl_sync(kFull, mine.len, i);
                r.z = __shfl_sync(kFull, mine.z, i);
                r.po = __shfl_sync(kFull, mine.po, i);
                r.clen = __shfl_sync(kFull, mine.clen, i);
            }
            todo &= todo - 1;
            uint8_t *dst = reinterpret_cast<uint8_t *>(r.dst);
            const uint8_t *src = reinterpret_cast<const uint8_t *>(r.src);
            if (!r.z) {
                copy_group<32>(dst, src, r.len, lane);
                continue;
            }
            const uint32_t b0 = r.po >> 9, b1 = (r.po + (1u << P.log2_part)) >> 9;   // the item's blocks of its chunk
            if (!crz_decode_warp<kHost>(dst, src, r.clen, r.z, b0, b1, lane, scratch + kCrzDecodeScratch * warp) &&
                lane == 0)
                atomicOr(P.err, kErrCodec);
        }
    }
}

}  // namespace

// The restore kernels are chained: each is launched while the one before it
// drains (mark -> check -> scatter by ordinary launches left 2-3 us between them).
template <class K>
static cudaError_t chain(K *kernel, const RestoreParams &p, uint64_t grid, uint32_t threads, cudaStream_t s) {
    RestoreParams q = p;
    void *args[] = {&q};
    return launch_chained(reinterpret_cast<const void *>(kernel), (uint32_t)grid, threads, args, s);
}

cudaError_t launch_restore_mark(const RestoreParams &p, int grid, cudaStream_t s) {
    return p.n_entries ? chain(restore_mark_kernel, p, grid, 256, s) : cudaSuccess;
}

cudaError_t launch_restore_check(const RestoreParams &p, int grid, cudaStream_t s) {
    return p.n_owner ? chain(restore_check_kernel, p, grid, 256, s) : cudaSuccess;
}

cudaError_t launch_restore_unmark(const RestoreParams &p, int grid, cudaStream_t s) {
    return p.n_owner ? chain(restore_unmark_kernel, p, grid, 256, s) : cudaSuccess;
}

cudaError_t launch_restore_scatter(const RestoreParams &p, uint64_t bytes, int sm_count, uint64_t max_grid,
                                   cudaStream_t s) {
    if (p.n_entries == 0 || p.n_owner == 0) return cudaSuccess;
    RestoreParams q = p;
    const RestoreCut cut = restore_cut(p.n_owner, bytes, p.log2_chunk, p.coded != 0, sm_count, max_grid);
    q.log2_part = cut.log2_part;
    if (p.coded) {
        static const void *const kFns[2][2] = {
            {reinterpret_cast<const void *>(&restore_scatter_coded_kernel<false, false>),
             reinterpret_cast<const void *>(&restore_scatter_coded_kernel<false, true>)},
            {reinterpret_cast<const void *>(&restore_scatter_coded_kernel<true, false>),
             reinterpret_cast<const void *>(&restore_scatter_coded_kernel<true, true>)}};
        void *args[] = {&q};
        return launch_chained(kFns[p.host ? 1 : 0][cut.lanes ? 1 : 0], cut.ctas, kScatterNT, args, s,
                              kCrzDecodeScratch * kScatterWarps);
    }
    return chain(p.ragged ? restore_scatter_ragged_kernel : restore_scatter_kernel, q, cut.ctas, kScatterNT, s);
}

cudaError_t launch_scatter(const ScatterParams &p, int grid, cudaStream_t s) {
    if (p.j1 <= p.j0) return cudaSuccess;
    scatter_kernel<<<grid, kScatterNT, 0, s>>>(p);
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) count_launches(1);
    return e;
}

}  // namespace crac
