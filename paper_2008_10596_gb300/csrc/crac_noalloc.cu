#include "crac_device.cuh"
#include "crac_grids.h"

// ---------------------------------------------------------------------------
// Allocation-free checkpoint pass (crac_pass_noalloc).
//
// For callers that must not allocate (an interposed cudaMalloc/cudaFree
// wrapper, an allocator hook, a preemption-time checkpoint, a process out of
// memory): the kernels of the split pass (hash, finalize, gather), with their
// scratch -- the control block, the look-back status words and the regions'
// payload offsets -- in a fixed array of this library's device memory instead
// of a buffer obtained from cudaMalloc, and the caller's fingerprint table as
// the chunks' accumulators.  One kernel prepares all of that, and each later one
// is launched as the one before it drains (six launches and memsets in a row
// took 21 us more than the fused kernel's one on 22 MiB).
// ---------------------------------------------------------------------------

namespace {

constexpr size_t kNoAllocScratchBytes =
    sizeof(crac::CkptCtrl) + 2 * sizeof(uint64_t) * (size_t)CRAC_NOALLOC_MAX_TILES;   // 512 KiB + 64 B

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_addr[kNoAllocMaxDevices];     // device address of the scratch, per device
int g_noalloc_sms[kNoAllocMaxDevices];

constexpr int kPrepareNT = 1024;

// Before the pass: zeroed scratch and accumulators (na and nb words), and, where
// there is no baseline (prefix), the payload bytes before each region, and by the
// CTA of the last ones the flag that the hash kernel may write every chunk there as
// it reads it (there is room for them all).  A CTA takes 1024 regions, a thread
// each, and sums up those before them itself: bound by one SM's reads of the table
// (75669 chunks of 256 bytes in 50000 regions, the whole pass: 170 us, 79 of them
// here, with one CTA and a run of regions per thread; 122 with one CTA and
// neighbouring regions on neighbouring lanes; 103 this way).
__global__ void __launch_bounds__(kPrepareNT)
noalloc_prepare_kernel(uint64_t *__restrict__ zero_a, uint32_t na, uint64_t *__restrict__ zero_b, uint32_t nb,
                       const crac::CkptDesc *__restrict__ d, uint32_t n, uint64_t cap, uint64_t *__restrict__ prefix,
                       uint32_t *__restrict__ flag) {
    using namespace crac;
    __shared__ uint64_t s_before[kPrepareNT / 32], s_sum[kPrepareNT / 32];
    for (uint32_t i = blockIdx.x * kPrepareNT + threadIdx.x; i < na + nb; i += gridDim.x * kPrepareNT) {
        if (i < na) zero_a[i] = 0;
        else zero_b[i - na] = 0;
    }
    const uint32_t i0 = blockIdx.x * kPrepareNT, i = i0 + threadIdx.x;
    if (!prefix || i0 >= n) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t mine = i < n ? d[i].bytes : 0;
    if (i0) {
        uint64_t sum = 0;
#pragma unroll 8
        for (uint32_t j = threadIdx.x; j < i0; j += kPrepareNT) sum += d[j].bytes;
        sum = warp_sum(sum);
        if (lane == 0) s_before[warp] = sum;
    }
    const uint64_t incl = warp_incl_scan(mine, lane);
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    uint64_t at = 0, total = 0;
    for (int w = 0; w < kPrepareNT / 32; ++w) {
        if (w < warp) at += s_sum[w];
        total += s_sum[w];
    }
    if (i0) {
        uint64_t before = 0;
        for (int w = 0; w < kPrepareNT / 32; ++w) before += s_before[w];
        at += before;
        total += before;
    }
    if (i < n) prefix[i] = at + incl - mine;
    if (threadIdx.x == 0 && n - i0 <= kPrepareNT) *flag = total <= cap ? 1u : 0u;
}

// The pass's results (a crac_pass_totals_t at any address) from its control
// block.  `reserved` keeps the value that earlier versions left in that word
// (tiles, and CTAs at five per SM, of a ticket-driven pass).
__global__ void noalloc_totals_kernel(const crac::CkptCtrl *ctrl, uint8_t *out, uint32_t reserved) {
    const uint32_t t = threadIdx.x;
    crac::wait_for_producer();
    if (t >= sizeof(crac_pass_totals_t)) return;
    const uint64_t w = t < 8 ? (uint64_t)ctrl->err << 32 | reserved : t < 16 ? ctrl->k : ctrl->D;
    out[t] = (uint8_t)(w >> (8 * (t & 7u)));
}

// Tile of the pass's limit (CRAC_NOALLOC_MAX_TILES), in chunks.
uint32_t noalloc_split(uint32_t chunk_bytes, int *wpc) {
    *wpc = chunk_bytes >= 16384u ? 8 : 1;
    uint32_t cpt = (128u << 10) / chunk_bytes;
    if (cpt < 1) cpt = 1;
    const uint32_t groups = 8u / (uint32_t)*wpc;
    if (cpt < groups) cpt = groups;
    if (cpt > 256) cpt = 256;
    return cpt;
}

// Loads every kernel that a call of any form may launch.  A kernel is loaded at its
// first use, which may allocate device memory and synchronize: with only the
// first call's own kernels loaded, the first one of another form took 400 us of
// host time instead of 23.
cudaError_t load_kernels() {
    using namespace crac;
    const void *fns[] = {reinterpret_cast<const void *>(&noalloc_prepare_kernel),
                         reinterpret_cast<const void *>(&noalloc_totals_kernel),
                         ckpt_fused_fn(256, 1, false),
                         ckpt_fused_fn(256, 8, false),
                         split_hash_fn(false, false, 0),
                         split_hash_fn(false, false, 13),
                         split_hash_small_fn(4, false),
                         split_hash_small_fn(8, false),
                         split_hash_small_fn(16, false),
                         split_hash_small_fn(32, false),
                         split_finalize_fn(split_finalize_tile(1, 1)),
                         split_finalize_fn(split_finalize_tile(UINT64_MAX, 1)),
                         split_gather_fn(false, false, 1, 1, 0)};
    cudaError_t e = cudaSuccess;
    cudaFuncAttributes a;
    for (const void *f : fns)
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, f);
    return e;
}

}  // namespace

// Every call of crac_pass_noalloc shares this array (it keeps the last call's
// contents; each call zeroes the part it uses before its pass).
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

extern "C" crac_status_t crac_pass_noalloc(const crac_region_t *regions_dev, uint32_t n_regions,
                                           uint64_t n_chunks, uint32_t chunk_bytes,
                                           const uint64_t *fp_old_dev, uint64_t *fp_new_dev,
                                           uint64_t *idx_dev, uint64_t *off_dev, uint64_t idx_cap,
                                           uint8_t *staging_dev, uint64_t staging_cap,
                                           crac_pass_totals_t *totals_dev, crac_stream_t stream) {
    using namespace crac;
    static_assert(sizeof(crac_region_t) == sizeof(CkptDesc), "region layout");
    static_assert(sizeof(crac_pass_totals_t) == 24, "totals layout");
    if (chunk_bytes < 16 || chunk_bytes > (1u << 24) || (chunk_bytes & (chunk_bytes - 1)))
        return CRAC_ERR_INVALID_ARG;
    if (!totals_dev || (n_chunks && (!regions_dev || !n_regions || !fp_new_dev || !idx_dev || !off_dev)))
        return CRAC_ERR_INVALID_ARG;
    int wpc;
    const uint32_t cpt = noalloc_split(chunk_bytes, &wpc);
    const uint64_t n_tiles = (n_chunks + cpt - 1) / cpt;
    if (n_tiles > CRAC_NOALLOC_MAX_TILES) return CRAC_ERR_INVALID_ARG;   // beyond the fixed scratch
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev >= kNoAllocMaxDevices) {
        note_cuda_error(e == cudaSuccess ? (int)cudaErrorInvalidDevice : (int)e);
        return CRAC_ERR_CUDA;
    }
    void *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!g_noalloc_addr[dev]) {
            // One-time set-up on this device (it is current): the host-side name
            // g_noalloc_scratch is only a stand-in, the kernel needs the device address.
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess) {
                note_cuda_error((int)e);
                return CRAC_ERR_CUDA;
            }
            int sms = 0;
            e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = load_kernels();
            if (e != cudaSuccess) {
                note_cuda_error((int)e);
                return CRAC_ERR_CUDA;
            }
            g_noalloc_sms[dev] = sms;
            g_noalloc_addr[dev] = p;
        }
        scratch = g_noalloc_addr[dev];
    }
    const uint32_t fin_tile = split_finalize_tile(n_chunks, g_noalloc_sms[dev]);
    const uint32_t fin_tiles = (uint32_t)((n_chunks + fin_tile - 1) / fin_tile);
    unsigned char *sc = static_cast<unsigned char *>(scratch);
    const size_t used = sizeof(CkptCtrl) + 16 * (size_t)(fin_tiles > 32 ? fin_tiles : 32);   // at most 16.1 KiB
    CkptCtrl *ctrl = reinterpret_cast<CkptCtrl *>(sc);
    uint32_t reserved = 0;
    if (n_tiles == 0) {
        noalloc_prepare_kernel<<<1, kPrepareNT, 0, s>>>(reinterpret_cast<uint64_t *>(sc), (uint32_t)(used / 8), nullptr, 0,
                                                        nullptr, 0, 0, nullptr, nullptr);
        e = cudaGetLastError();
        if (e == cudaSuccess) count_launches(1);
    } else {
        CkptParams P{};
        // A list that one CTA takes in a few rounds, too short for a chain of
        // kernels: the fused one (4 chunks of 4 KiB: 19 us to the call's end, the
        // chain 24; 512 chunks of 512 B 53 and 26).
        const bool fused = n_chunks <= 32 && n_chunks * chunk_bytes <= (256u << 10);
        P.desc = reinterpret_cast<const CkptDesc *>(regions_dev);
        P.n_allocs = n_regions;
        uint32_t l = 0;
        while ((1u << l) < chunk_bytes) ++l;
        P.log2_chunk = l;
        P.c_begin = 0;
        P.c_end = n_chunks;
        P.cpt = fused ? cpt : fin_tile;
        P.n_tiles = fused ? (uint32_t)n_tiles : fin_tiles;
        P.fp_old = fp_old_dev;
        P.fp_new = fp_new_dev;
        P.idx_out = idx_dev;
        P.off_out = off_dev;
        P.idx_cap = idx_cap;
        P.staging = staging_dev;
        P.staging_cap = staging_dev ? staging_cap : 0;
        P.ctrl = ctrl;
        P.tile_cnt = reinterpret_cast<uint64_t *>(sc + sizeof(CkptCtrl));
        P.tile_bytes = P.tile_cnt + P.n_tiles;
        P.timeout_ns = 2000000000ull;
        // Without a baseline every chunk is dirty and its payload offset known
        // beforehand: the hash kernel writes it there as it reads it, if they
        // all fit (1 GiB in 64 KiB chunks, the whole call: 513 us with the fused
        // kernel, which reads every chunk twice, 330 us this way; with a baseline
        // and 10% dirty 283 and 215 us).
        const size_t at = (used + 255) / 256 * 256;
        uint64_t *prefix = nullptr;
        if (!fused && !fp_old_dev && staging_dev && n_regions <= (kNoAllocScratchBytes - at) / 8 - 1) {
            prefix = reinterpret_cast<uint64_t *>(sc + at);
            P.full_copy = 1;
            P.full_flag = reinterpret_cast<const uint32_t *>(prefix + n_regions);
            P.alloc_prefix = prefix;
        }
        const bool small = l >= 9 && l < 13;
        // The regions' bytes are in device memory only: taken as full chunks, but
        // with chunks above 64 KiB, which regions often do not fill, as what 32
        // CTAs per SM of 64 KiB each hold, so that a warp takes several segments
        // (full chunks keep the same bytes per warp either way, empty segments
        // are skipped; 1200 regions of 4 KiB in chunks of 1 MiB: 80 -> 49 us, of 64
        // bytes in chunks of 16 MiB 772 -> 45).
        const uint64_t full = n_chunks << l;
        const uint64_t most = l > 16 ? umin64(full, (uint64_t)g_noalloc_sms[dev] << 21) : full;
        uint32_t log2Seg = small ? l : split_hash_seg(n_chunks, full, l, P.full_copy != 0);
        const uint32_t grid = split_hash_grid(n_chunks, most, l, log2Seg, P.full_copy != 0, g_noalloc_sms[dev],
                                              &P.slots_per_warp);
        // Segmented chunks are summed up in the caller's table, in place.
        unsigned long long *acc = !fused && log2Seg < l ? reinterpret_cast<unsigned long long *>(fp_new_dev) : nullptr;
        const uint32_t sms = (uint32_t)g_noalloc_sms[dev], na = (uint32_t)(used / 8), nb = acc ? (uint32_t)n_chunks : 0u;
        const uint32_t want = (na + nb + kPrepareNT - 1) / kPrepareNT, sums = prefix ? (n_regions - 1) / kPrepareNT + 1 : 1;
        const uint32_t ctas = want < sms ? want : sms;
        noalloc_prepare_kernel<<<ctas > sums ? ctas : sums, kPrepareNT, 0, s>>>(
            reinterpret_cast<uint64_t *>(sc), na, fp_new_dev, nb, P.desc, n_regions, P.staging_cap, prefix,
            prefix ? reinterpret_cast<uint32_t *>(prefix + n_regions) : nullptr);
        e = cudaGetLastError();
        if (e == cudaSuccess) count_launches(1);
        void *args[] = {&P, &acc, &log2Seg};
        if (e == cudaSuccess && fused) {
            e = cudaLaunchKernel(ckpt_fused_fn(256, wpc, false), dim3((uint32_t)n_tiles), dim3(256), args, 0, s);
            if (e == cudaSuccess) count_launches(1);
        }
        if (e == cudaSuccess && !fused)
            e = launch_chained(small ? split_hash_small_fn(1 << (l - 7), false) : split_hash_fn(false, false, l), grid,
                               split_hash_threads(), args, s);
        if (e == cudaSuccess && !fused)
            e = launch_chained(split_finalize_fn(fin_tile), fin_tiles < 2u * sms ? fin_tiles : 2u * sms,
                               split_finalize_threads(), args, s);
        if (e == cudaSuccess && !fused)
            e = launch_chained(split_gather_fn(false, false, n_chunks, full, l), 8 * sms, split_gather_threads(), args, s);
        const uint64_t g = 5ull * sms;
        reserved = (uint32_t)(n_tiles + (n_tiles < g ? n_tiles : g));
    }
    if (e == cudaSuccess) {
        uint8_t *out = reinterpret_cast<uint8_t *>(totals_dev);
        void *args[] = {&ctrl, &out, &reserved};
        e = launch_chained(reinterpret_cast<const void *>(&noalloc_totals_kernel), 1, 32, args, s);
    }
    if (e != cudaSuccess) {
        note_cuda_error((int)e);
        return CRAC_ERR_CUDA;
    }
    return CRAC_OK;
}
