// ppf_binned.cu -- the binned likelihood path: Sec. 6.3's input-space
// decomposition on one GPU.  When a step's particles are spread over the
// frame (the prior draw, a weak signal), the direct path's patch reads touch
// a separate cache line per lane and the step becomes bound by L2 traffic.
// The binned path instead:
//   1. propagates every slot, writes its bin and counts the bin sizes (the
//      step kernel's bin_propagate; a bin is an image tile of T x T patch
//      anchors, plus one bin for particles that need no patch sum);
//   2. scatters each particle's record (x, y, I0) into its bin: each block
//      turns the bin sizes into bin starts, takes chunks of slots, ranks them
//      by bin in shared memory and reserves one range per bin with one
//      atomic, so a bin's records from one chunk are written contiguously;
//      the slot keeps its record's place;
//   3. runs the likelihood over work items of one bin: the tile's window
//      (the tile plus the patch halo) and the item's records are copied into
//      shared memory by the tensor-memory accelerator (cp.async.bulk,
//      completion on an mbarrier), the next item's while this one is summed,
//      every patch read comes from shared memory, and l is written in bin
//      order;
//   4. sums in the direct path's slot order (the step kernel's phase 1),
//      fetching each slot's l from its record's place.
// A particle's likelihood has the same bits on both paths (the same PSF
// samples and the same patch_rows arithmetic), and the sums are taken in
// the same order, so the two paths give the same results bit for bit, and
// the order of the records inside a bin does not matter.  The step's
// finaliser picks the path of the next step from the spread of its warps.
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstring>

#include "ppf_device.cuh"
#include "ppf_internal.h"
#include "ppf_kernels.cuh"

namespace ppf {

// records per likelihood work item and threads of its block (see bin_loglik_kernel); WIDE: tiles of more than 32 anchors
template <bool WIDE>
struct BinShape {
    static constexpr int THREADS = WIDE ? 512 : 256, ITEM = WIDE ? 2560 : 1536, BLOCKS = WIDE ? 1 : 2;
};
constexpr int BIN_MAX_BOX = 128;      // window edge T + 2R (a tensor copy box is at most 256 floats wide)

// ---------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(1) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// a 2D tile of the prepared frame into shared memory; completion is counted
// on the mbarrier in bytes (x is the float column, a multiple of 4 here)
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// bytes (a multiple of 16, both addresses 16-byte aligned) into shared memory, counted on the same barrier
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Waits for the phase of the given parity to complete.  Bounded: gives up
// after about a second of clock cycles (or 2^26 polls) and returns false.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    const long long t0 = clock64();
    for (uint32_t it = 0; it < (1u << 26); ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok)
            return true;
        if (clock64() - t0 > (1ll << 31))
            break;
    }
    return false;
}

// ---------------------------------------------------------- the scatter
// Each block first turns the bin sizes into their exclusive prefix (each
// bin's first record).  It then takes chunks of BIN_CHUNK consecutive slots.
// A chunk is ranked by bin in shared memory and staged there in bin order; one
// global atomic per nonempty bin reserves the chunk's range inside the bin
// (its cursor), and the staged records are then copied out so that consecutive
// threads write consecutive records of a run.  Each slot's key entry receives
// its record's place (read by the sums of phase 1).
//
// A chain of latencies bounds it: keys, shared atomics, a prefix, the
// reservations, staging, each behind a barrier.  So a chunk's keys and states
// are loaded together at its start, four consecutive slots a lane (coalesced
// 16-byte vectors), and two blocks of 512 threads share an SM, one grid of
// resident blocks.  4,000,000 slots, 290 bins: 58.8 us with 16 consecutive
// slots a thread loaded where they were staged, 33.9 us now (144 MB, 21 us at
// the copy rate).  Half the chunk doubles the reservations and the runs: 82 us
// in the first form.
constexpr int BIN_PER_THREAD = 8;
constexpr int BIN_QUADS = BIN_PER_THREAD / 4;
constexpr int BIN_THREADS = 512;
constexpr int BIN_QSTEP = 4 * BIN_THREADS;
constexpr int BIN_CHUNK = BIN_THREADS * BIN_PER_THREAD;

__global__ void __launch_bounds__(BIN_THREADS, 2) bin_scatter_kernel(const float *__restrict__ st, int64_t N, int nbins,
                                                          uint32_t *__restrict__ key,
                                                          const uint32_t *__restrict__ size,
                                                          uint32_t *__restrict__ cursor, float4 *__restrict__ rec, DevSummary *sum)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    if (__ldcg(&sum->bin_this) == 0)
        return;
    int32_t *flags = &sum->flags;
    // [BIN_CHUNK] staged records, [BIN_CHUNK] their bins, then per bin: count,
    // local start, global start, bin start
    extern __shared__ float4 stage[];
    uint16_t *sbin = reinterpret_cast<uint16_t *>(stage + BIN_CHUNK);
    uint32_t *cnt = reinterpret_cast<uint32_t *>(sbin + BIN_CHUNK);
    uint32_t *lstart = cnt + nbins, *gstart = lstart + nbins, *bstart = gstart + nbins;
    __shared__ uint64_t red[33];
    {   // bin starts: exclusive prefix of the sizes
        const int per = (nbins + blockDim.x - 1) / blockDim.x, t0 = threadIdx.x * per;
        uint64_t sm = 0;
        for (int t = t0; t < t0 + per && t < nbins; ++t)
            sm += __ldcg(size + t);
        uint64_t tot;
        uint64_t run = block_excl_scan_u64(sm, red, &tot);
        for (int t = t0; t < t0 + per && t < nbins; ++t) {
            bstart[t] = (uint32_t)run;
            run += __ldcg(size + t);
        }
        __syncthreads();
    }
    const uint32_t n = (uint32_t)N;
    const bool vec_ok = (N & 3) == 0;  // 16-byte vectors need 16-byte aligned planes
    for (uint32_t lo = blockIdx.x * (uint32_t)BIN_CHUNK; lo < n; lo += gridDim.x * (uint32_t)BIN_CHUNK) {
        for (int t = threadIdx.x; t < nbins; t += blockDim.x)
            cnt[t] = 0u;
        // quarter q of a thread's slots: four from lo + 4 (q threads + thread)
        uint32_t k[BIN_PER_THREAD], r[BIN_PER_THREAD];
        float4 xx[BIN_QUADS], yy[BIN_QUADS], zz[BIN_QUADS];
        const uint32_t i0 = lo + 4u * threadIdx.x;
        const bool full = vec_ok && n - lo >= (uint32_t)BIN_CHUNK;
        if (full) {
#pragma unroll
            for (int q = 0; q < BIN_QUADS; ++q) {
                const uint4 kk = __ldcg(reinterpret_cast<const uint4 *>(key + i0 + q * BIN_QSTEP));
                k[4 * q] = kk.x; k[4 * q + 1] = kk.y; k[4 * q + 2] = kk.z; k[4 * q + 3] = kk.w;
            }
#pragma unroll
            for (int q = 0; q < BIN_QUADS; ++q) {
                xx[q] = __ldcg(reinterpret_cast<const float4 *>(st + i0 + q * BIN_QSTEP));
                yy[q] = __ldcg(reinterpret_cast<const float4 *>(st + N + i0 + q * BIN_QSTEP));
                zz[q] = __ldcg(reinterpret_cast<const float4 *>(st + 4 * N + i0 + q * BIN_QSTEP));
            }
        } else {
#pragma unroll
            for (int q = 0; q < BIN_QUADS; ++q) {
                const uint32_t i = i0 + q * BIN_QSTEP;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    k[4 * q + e] = i + e < n ? __ldcg(key + i + e) : 0u;
                auto at = [&](const float *p, int e) { return i + e < n ? __ldcg(p + i + e) : 0.0f; };
                xx[q] = make_float4(at(st, 0), at(st, 1), at(st, 2), at(st, 3));
                yy[q] = make_float4(at(st + N, 0), at(st + N, 1), at(st + N, 2), at(st + N, 3));
                zz[q] = make_float4(at(st + 4 * N, 0), at(st + 4 * N, 1), at(st + 4 * N, 2), at(st + 4 * N, 3));
            }
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < BIN_PER_THREAD; ++e)
            r[e] = (i0 + (e / 4) * BIN_QSTEP + e % 4 < n) ? atomicAdd(&cnt[k[e]], 1u) : 0u;
        __syncthreads();
        {   // local starts (exclusive prefix of the counts) and the global reservations
            const int per = (nbins + blockDim.x - 1) / blockDim.x, t0 = threadIdx.x * per;
            uint64_t sm = 0;
            for (int t = t0; t < t0 + per && t < nbins; ++t)
                sm += cnt[t];
            uint64_t tot;
            uint64_t run = block_excl_scan_u64(sm, red, &tot);
            for (int t = t0; t < t0 + per && t < nbins; ++t) {
                const uint32_t c = cnt[t];
                lstart[t] = (uint32_t)run;
                gstart[t] = c ? bstart[t] + atomicAdd(cursor + t, c) : 0u;
                run += c;
            }
        }
        __syncthreads();
        // stage the records in bin order
#pragma unroll
        for (int q = 0; q < BIN_QUADS; ++q) {
            const float xs[4] = {xx[q].x, xx[q].y, xx[q].z, xx[q].w}, ys[4] = {yy[q].x, yy[q].y, yy[q].z, yy[q].w};
            const float zs[4] = {zz[q].x, zz[q].y, zz[q].z, zz[q].w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int e = 4 * q + c;
                if (i0 + q * BIN_QSTEP + c < n) {
                    const uint32_t j = lstart[k[e]] + r[e];
                    stage[j] = make_float4(xs[c], ys[c], zs[c], 0.0f);
                    sbin[j] = (uint16_t)k[e];
                    k[e] = gstart[k[e]] + r[e];  // the record's place, for the slot's key entry
                }
            }
        }
        if (full) {
#pragma unroll
            for (int q = 0; q < BIN_QUADS; ++q)
                *reinterpret_cast<uint4 *>(key + i0 + q * BIN_QSTEP) =
                    make_uint4(k[4 * q], k[4 * q + 1], k[4 * q + 2], k[4 * q + 3]);
        } else {
#pragma unroll
            for (int e = 0; e < BIN_PER_THREAD; ++e) {
                const uint32_t i = i0 + (e / 4) * BIN_QSTEP + e % 4;
                if (i < n)
                    key[i] = k[e];
            }
        }
        __syncthreads();
        // copy out: consecutive threads, consecutive records of a bin's run
        const uint32_t m = (n - lo < (uint32_t)BIN_CHUNK) ? n - lo : (uint32_t)BIN_CHUNK;
        for (uint32_t j = threadIdx.x; j < m; j += blockDim.x) {
            const uint32_t t = sbin[j];
            const uint32_t pos = gstart[t] + (j - lstart[t]);
            if (PPF_DCHECK(pos < n, flags, FLAG_INTERNAL))
                rec[pos] = stage[j];
        }
        __syncthreads();
    }
}

// ------------------------------------------------------- the likelihood
// Bound by the shared-memory pipe: a patch at R = 5 takes 66 eight-byte window
// reads, two wavefronts a warp each, so 4,000,000 records need 56 us of it.
// What kept the kernel from that was each item's start (its records read from
// L2 twice around three barriers) and uneven work.  Now the next item's
// records are copied with its window (one bulk copy each on one barrier)
// while this item is summed, only the 16-bit order is sorted, a window row is
// a multiple of 16 pairs (the anchor after the last of a row then stands in
// the following bank; 254 us instead of 265 for the step), and each block
// finds its items from the bin sizes, without a list made by the scatter's
// last block.  Items of 1536 records leave two blocks an SM and deal evenly:
// the whole binned step takes 246 us for 4,000,000 particles (243 with 1280,
// 254 with 2048; 286 with items of 4096 and none of this), 1168 for 24,000,000
// (1188, 1280), 86 for 1,000,000 (91, 86), 49 for 250,000 (49, 51; 66).
//
// Tiles of 64 anchors (frames of more than 3072 tiles of 32): an item's window
// of up to 51 KB and its 4096 anchor counts leave room for one block an SM and
// cost every item more, so the block has 512 threads and items of 2560
// records, the most that fits at R = 8.  Particles set over the whole frame
// and stepped, with this, with 256 threads and 1536, and as it was before the
// records were copied ahead (256, 4096): 8,000,000 on 3500 x 3000 at R = 8
// 1237, 1417, 1271 us; on 2200 x 2200 at R = 5 758, 874, 862 us; 4,000,000
// there 453, 515, 491 us; 50,000 108, 121, 150 us.  (512 threads and 2048: 1361,
// 752, 426, 105; 256 and 2560: 1308, 809, 488, 122.)
struct BinLikArgs {
    int64_t N;
    int W, H, T, nx, nbins;
    int box, pitch;                // rows of a window (T + 2R) and pairs in one of its rows (win_pitch)
    int win_stride;                // bytes between the two windows (a multiple of 128)
    float inv2s2, inv_sxi2;
    float Kc[MAX_RADIUS];
    const float4 *__restrict__ rec;
    const uint32_t *__restrict__ size;  // the bin sizes
    float *__restrict__ l;         // l of every record, in bin order
    DevSummary *sum;
};

template <int R, bool WIDE>
__global__ void __launch_bounds__(BinShape<WIDE>::THREADS, BinShape<WIDE>::BLOCKS)
    bin_loglik_kernel(const __grid_constant__ CUtensorMap tmap, BinLikArgs a)
{
    constexpr int BIN_ITEM = BinShape<WIDE>::ITEM, BIN_SORT_PER_THREAD = BIN_ITEM / BinShape<WIDE>::THREADS;
    if (!pdl_wait())
        return;
    pdl_trigger();
    DevSummary *sum = a.sum;
    if (__ldcg(&sum->bin_this) == 0)
        return;
    extern __shared__ __align__(16) unsigned char bsm[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ int failed;
    __shared__ uint64_t red[33];
    // the windows start on a 128-byte boundary (the launch adds 128 bytes of
    // slack); then two items' records, the current item's order by anchor,
    // the anchor counts, and the bins' first records and items
    const uint32_t base = smem_u32(bsm), pad = ((base + 127u) & ~127u) - base;
    unsigned char *wbase = bsm + pad;
    float4 *raw = reinterpret_cast<float4 *>(wbase + 2 * a.win_stride);
    uint16_t *srt = reinterpret_cast<uint16_t *>(raw + 2 * BIN_ITEM);
    uint32_t *hist = reinterpret_cast<uint32_t *>(srt + BIN_ITEM);
    uint32_t *bs = hist + a.T * a.T, *is = bs + a.nbins + 1;
    const uint32_t bar0 = smem_u32(&bars[0]), bar1 = smem_u32(&bars[1]);
    const uint32_t win0 = base + pad, win1 = win0 + (uint32_t)a.win_stride, raw0 = smem_u32(raw);
    const uint32_t box_bytes = (uint32_t)(a.box * a.pitch * 8);
    if (threadIdx.x == 0) {
        mbar_init(bar0);
        mbar_init(bar1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        failed = 0;
    }
    int n_items;
    {   // first item and first record of every bin
        const int per = (a.nbins + blockDim.x - 1) / blockDim.x, t0 = threadIdx.x * per;
        uint64_t sm = 0;
        for (int t = t0; t < t0 + per && t < a.nbins; ++t) {
            const uint32_t z = __ldcg(a.size + t);
            sm += ((uint64_t)((z + BIN_ITEM - 1) / BIN_ITEM) << 32) + z;
        }
        uint64_t all;
        uint64_t run = block_excl_scan_u64(sm, red, &all);
        for (int t = t0; t < t0 + per && t < a.nbins; ++t) {
            const uint32_t z = __ldcg(a.size + t);
            bs[t] = (uint32_t)run;
            is[t] = (uint32_t)(run >> 32);
            run += ((uint64_t)((z + BIN_ITEM - 1) / BIN_ITEM) << 32) + z;
        }
        n_items = (int)(all >> 32);
        if (threadIdx.x == 0) {
            bs[a.nbins] = (uint32_t)all;
            is[a.nbins] = (uint32_t)n_items;
        }
    }
    __syncthreads();
    struct Item {
        int t;
        uint32_t s0, cnt;
    };
    auto item_at = [&](int j) -> Item {  // j < n_items
        int lo = 0, up = a.nbins;        // is[lo] <= j < is[up]
        while (up - lo > 1) {
            const int mid = (lo + up) >> 1;
            if (is[mid] <= (uint32_t)j)
                lo = mid;
            else
                up = mid;
        }
        const uint32_t s0 = bs[lo] + ((uint32_t)j - is[lo]) * (uint32_t)BIN_ITEM;
        return Item{lo, s0, min(bs[lo + 1] - s0, (uint32_t)BIN_ITEM)};
    };
    const int special = a.nbins - 1;
    auto issue = [&](const Item &it, int buf) {  // thread 0: the item's window and records into buffer buf
        if (it.t == special)
            return;
        const int tx = it.t % a.nx, ty = it.t / a.nx;
        const uint32_t bar = buf ? bar1 : bar0;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar, box_bytes + 16u * it.cnt);
        tma_load_2d(buf ? win1 : win0, &tmap, 2 * tx * a.T, ty * a.T, bar);
        bulk_load(raw0 + (buf ? 16u * (uint32_t)BIN_ITEM : 0u), a.rec + it.s0, 16u * it.cnt, bar);
    };
    const PatchGeom geom{nullptr, a.W, a.H, 0, 0, a.inv2s2, a.inv_sxi2, a.Kc, 0, &sum->flags};
    const float4 *__restrict__ rec = a.rec;
    // Thread 0 issues every copy; all threads wait on its barrier.  A wait
    // that times out stops the block's work (the flag reports it), and
    // thread 0 then waits once more, bounded, for the copies it left in
    // flight before the block's shared memory is released.
    // bit b of phase: the parity of buffer b's next copy; bit b of pend: a
    // copy into buffer b issued and not yet waited for
    uint32_t phase = 0u, pend = 0u;
    int k = 0;
    if ((int)blockIdx.x >= n_items)
        return;
    Item next = item_at(blockIdx.x);
    if (threadIdx.x == 0)
        issue(next, 0);
    pend |= (next.t != special) ? 1u : 0u;
    for (int j = blockIdx.x; j < n_items; j += gridDim.x, ++k) {
        const int buf = k & 1;
        const int t = next.t;
        const int s0 = (int)next.s0, cntj = (int)next.cnt;
        if (j + (int)gridDim.x < n_items) {  // the next item's copies run while this one is summed
            next = item_at(j + (int)gridDim.x);
            if (threadIdx.x == 0)
                issue(next, buf ^ 1);
            if (next.t != special)
                pend |= 1u << (buf ^ 1);
        }
        if (t != special) {
            if (mbar_wait(buf ? bar1 : bar0, (phase >> buf) & 1u)) {
                phase ^= 1u << buf;
                pend &= ~(1u << buf);
            } else {
                atomicOr(&sum->flags, FLAG_TIMEOUT);
                failed = 1;
            }
            __syncthreads();
            if (failed)
                break;
        }
        const float2 *win = reinterpret_cast<const float2 *>(wbase + (buf ? a.win_stride : 0));
        const float4 *rb = raw + (buf ? BIN_ITEM : 0);
        const int tx = t % a.nx, ty = t / a.nx;
        constexpr int P = 2 * R + 1;
        if (t == special) {  // no patch sums: l = -inf (non-finite) or 0 (no pixel in the image)
            for (int r = s0 + threadIdx.x; r < s0 + cntj; r += blockDim.x) {
                const float4 q = rec[r];
                int cx, cy;
                float gx[P], gy[P], C, l;
                patch_setup<R>(geom, q.x, q.y, q.z, cx, cy, gx, gy, C, &l);
                a.l[r] = l;
            }
        } else {
            // Sort the item's records by patch anchor (a counting sort over the
            // T x T anchors of the tile), so that the lanes of a warp hold
            // neighbouring anchors and their window reads share shared-memory
            // words instead of colliding in the banks.
            for (int u = threadIdx.x; u < a.T * a.T; u += blockDim.x)
                hist[u] = 0u;
            __syncthreads();
            uint32_t an[BIN_SORT_PER_THREAD];  // anchor and rank
#pragma unroll
            for (int e = 0; e < BIN_SORT_PER_THREAD; ++e) {
                const int r = threadIdx.x + e * (int)blockDim.x;
                const float2 xy = r < cntj ? *reinterpret_cast<const float2 *>(rb + r) : make_float2(0.0f, 0.0f);
                const int lu = (int)floorf(xy.x + 0.5f) + R - tx * a.T;
                const int lv = (int)floorf(xy.y + 0.5f) + R - ty * a.T;
                const bool ok = r < cntj && PPF_DCHECK(lu >= 0 && lu < a.T && lv >= 0 && lv < a.T, &sum->flags,
                                                       FLAG_INTERNAL);
                const uint32_t u = (uint32_t)(lv * a.T + lu);
                an[e] = ok ? u | (atomicAdd(&hist[u], 1u) << 16) : 0xFFFFFFFFu;
            }
            __syncthreads();
            int sorted = cntj;
            // exclusive prefix of the T x T counts
            {
                const int na = a.T * a.T, per = (na + blockDim.x - 1) / blockDim.x, u0 = threadIdx.x * per;
                uint64_t sm = 0;
                for (int u = u0; u < u0 + per && u < na; ++u)
                    sm += hist[u];
                uint64_t tot;
                uint64_t run = block_excl_scan_u64(sm, red, &tot);
                // (the debug build: without the records its anchor check left out)
                if (!PPF_DCHECK(tot == (uint64_t)cntj, &sum->flags, FLAG_INTERNAL))
                    sorted = (int)tot;
                for (int u = u0; u < u0 + per && u < na; ++u) {
                    const uint32_t c = hist[u];
                    hist[u] = (uint32_t)run;
                    run += c;
                }
            }
            __syncthreads();
#pragma unroll
            for (int e = 0; e < BIN_SORT_PER_THREAD; ++e)
                if (an[e] != 0xFFFFFFFFu)
                    srt[hist[an[e] & 0xFFFFu] + (an[e] >> 16)] = (uint16_t)(threadIdx.x + e * blockDim.x);
            __syncthreads();
            for (int j = threadIdx.x; j < sorted; j += blockDim.x) {
                const uint32_t r = srt[j];
                const float4 v = rb[r];
                int cx, cy;
                float gx[P], gy[P], C, l;
                if (patch_setup<R>(geom, v.x, v.y, v.z, cx, cy, gx, gy, C, &l)) {
                    const int lu = cx + R - tx * a.T, lv = cy + R - ty * a.T;
                    const float Bs = patch_rows<R, true, true>(win + lv * a.pitch + lu, a.pitch, gx, gy);
                    l = v.z * fmaf(-0.5f * v.z, C, Bs) * a.inv_sxi2;
                }
                a.l[s0 + r] = l;
            }
        }
        __syncthreads();  // this window is free for the copy two items on
    }
    if (failed && threadIdx.x == 0) {
        if (pend & 1u)
            mbar_wait(bar0, phase & 1u);
        if (pend & 2u)
            mbar_wait(bar1, (phase >> 1) & 1u);
    }
}

// ------------------------------------------------------------ host side
namespace {

// pairs in a row of the window: whole turns of the 32 banks (see bin_loglik_kernel)
int win_pitch(int box) { return (box + 15) / 16 * 16; }

int win_stride_bytes(int box)
{
    const int b = box * win_pitch(box) * 8;
    return (b + 127) / 128 * 128;
}

size_t scatter_smem(int nbins)
{
    // staged records, their bins, and four words per bin
    return sizeof(float4) * BIN_CHUNK + sizeof(uint16_t) * BIN_CHUNK + 4 * sizeof(uint32_t) * (size_t)nbins;
}

bool wide_tiles(int T) { return T > 32; }

size_t loglik_smem(int box, int T, int nbins)
{
    const size_t item = wide_tiles(T) ? BinShape<true>::ITEM : BinShape<false>::ITEM;
    // two windows, the alignment slack, two items' records and their order, the anchor counts, the bin prefixes
    return 2 * (size_t)win_stride_bytes(box) + 128 + (2 * sizeof(float4) + sizeof(uint16_t)) * item +
           sizeof(uint32_t) * (T * T + 2 * ((size_t)nbins + 1));
}

// The dynamic shared memory limit of a kernel is raised to the device's
// opt-in maximum less the kernel's static shared memory (a limit, not a
// reservation): contexts with other window sizes then never lower it under
// one another.
template <typename K>
cudaError_t raise_smem_limit(K kernel, size_t need)
{
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess)
        return e;
    const int lim = optin - (int)fa.sharedSizeBytes;
    if ((int64_t)need > lim)
        return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
}

template <int R, bool WIDE>
cudaError_t loglik_attr(size_t smem, int *per_sm)
{
    cudaError_t e = raise_smem_limit(bin_loglik_kernel<R, WIDE>, smem);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, bin_loglik_kernel<R, WIDE>, BinShape<WIDE>::THREADS,
                                                          smem);
    return e;
}

template <bool WIDE>
cudaError_t loglik_setup(int R, size_t smem, int *per_sm)
{
    switch (R) {
    case 0: return loglik_attr<0, WIDE>(smem, per_sm);
    case 1: return loglik_attr<1, WIDE>(smem, per_sm);
    case 2: return loglik_attr<2, WIDE>(smem, per_sm);
    case 3: return loglik_attr<3, WIDE>(smem, per_sm);
    case 4: return loglik_attr<4, WIDE>(smem, per_sm);
    case 5: return loglik_attr<5, WIDE>(smem, per_sm);
    case 6: return loglik_attr<6, WIDE>(smem, per_sm);
    case 7: return loglik_attr<7, WIDE>(smem, per_sm);
    default: return loglik_attr<8, WIDE>(smem, per_sm);
    }
}

template <typename T>
cudaError_t dalloc(T **p, size_t count)
{
    *p = nullptr;
    return cudaMalloc((void **)p, sizeof(T) * (count ? count : 1));
}

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

}  // namespace

cudaError_t bin_setup(ppf_ctx *c)
{
    const int R = c->m.patch_radius;
    if (c->m.likelihood != 0)
        return cudaSuccess;  // pcSIR: one lookup per particle, no patch to stage
    int T = 32;
    auto bins = [&](int t) { return (int64_t)((c->m.width + 2 * R + t - 1) / t) * ((c->m.height + 2 * R + t - 1) / t) + 1; };
    while (bins(T) > BIN_MAX_BINS && T + 2 * R <= BIN_MAX_BOX / 2)
        T *= 2;
    if (bins(T) > BIN_MAX_BINS || T + 2 * R > BIN_MAX_BOX)
        return cudaSuccess;  // frames this large keep the direct path
    c->bin_T = T;
    c->bin_nx = (c->m.width + 2 * R + T - 1) / T;
    c->bin_nbins = (int32_t)bins(T);
    const int box = T + 2 * R;
    const size_t smem = loglik_smem(box, T, c->bin_nbins);
    int per_sm = 0;
    cudaError_t e = wide_tiles(T) ? loglik_setup<true>(R, smem, &per_sm) : loglik_setup<false>(R, smem, &per_sm);
    if (e != cudaSuccess)
        return e;
    c->bin_grid = c->num_sms * (per_sm > 0 ? (per_sm < 4 ? per_sm : 4) : 1);
    e = raise_smem_limit(bin_scatter_kernel, scatter_smem(c->bin_nbins));
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bin_scatter_kernel, BIN_THREADS, scatter_smem(c->bin_nbins));
    if (e != cudaSuccess)
        return e;
    c->bin_scatter_grid = c->num_sms * (per_sm > 0 ? per_sm : 1);
    if ((e = dalloc(&c->bin_key, (size_t)c->N)) != cudaSuccess ||
        (e = dalloc(&c->bin_l, (size_t)c->N)) != cudaSuccess ||
        (e = dalloc(&c->bin_tot, 2 * ((size_t)c->bin_nbins + 1))) != cudaSuccess ||
        (e = dalloc(&c->bin_rec, (size_t)c->N)) != cudaSuccess)
        return e;
    // the prepared frame as a 2D float tensor (2 Wp floats per row, Hp rows);
    // a window is 2 win_pitch(box) floats by box rows, copied with zero fill outside
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
        return e != cudaSuccess ? e : cudaErrorNotSupported;
    const cuuint64_t dims[2] = {(cuuint64_t)2 * c->Wp, (cuuint64_t)c->Hp};
    const cuuint64_t strides[1] = {(cuuint64_t)2 * c->Wp * sizeof(float)};
    const cuuint32_t boxd[2] = {(cuuint32_t)(2 * win_pitch(box)), (cuuint32_t)box};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = reinterpret_cast<EncodeTiled>(fn)(
        &c->bin_tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, c->Zp, dims, strides, boxd, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    return bin_set_next(c, 1);  // the prior draw is spread over the frame
}

cudaError_t bin_set_next(ppf_ctx *c, int binned)
{
    if (!c->bin_key)
        return cudaSuccess;
    const int32_t v = binned ? 1 : 0;
    cudaError_t e = cudaMemcpyAsync((char *)c->sum + offsetof(DevSummary, bin_next), &v, sizeof(v),
                                    cudaMemcpyHostToDevice, c->stream);
    return e == cudaSuccess ? cudaStreamSynchronize(c->stream) : e;
}

template <int R>
static void launch_loglik_r(const CUtensorMap &tm, const BinLikArgs &a, int grid, size_t smem, cudaStream_t s)
{
    if (wide_tiles(a.T))
        launch_pdl(bin_loglik_kernel<R, true>, grid, BinShape<true>::THREADS, smem, s, tm, a);
    else
        launch_pdl(bin_loglik_kernel<R, false>, grid, BinShape<false>::THREADS, smem, s, tm, a);
}

cudaError_t launch_binned(ppf_ctx *c)
{
    const int R = c->m.patch_radius;
    const int nb = c->bin_nbins;
    float *dst = c->state[c->cur ^ 1];
    const int64_t chunks = (c->N + BIN_CHUNK - 1) / BIN_CHUNK;
    const int gscat = (int)(chunks < (int64_t)c->bin_scatter_grid ? chunks : (int64_t)c->bin_scatter_grid);
    launch_pdl(bin_scatter_kernel, gscat, BIN_THREADS, scatter_smem(nb), c->stream, (const float *)dst, c->N, nb, c->bin_key,
               (const uint32_t *)c->bin_tot, c->bin_tot + nb + 1, c->bin_rec, c->sum);
    BinLikArgs a;
    memset(&a, 0, sizeof(a));
    a.N = c->N;
    a.W = c->m.width;
    a.H = c->m.height;
    a.T = c->bin_T;
    a.nx = c->bin_nx;
    a.nbins = nb;
    a.box = c->bin_T + 2 * R;
    a.pitch = win_pitch(a.box);
    a.win_stride = win_stride_bytes(a.box);
    a.inv2s2 = 1.0f / (2.0f * c->m.psf_sigma * c->m.psf_sigma);
    a.inv_sxi2 = 1.0f / (c->m.sigma_xi * c->m.sigma_xi);
    for (int q = 0; q < MAX_RADIUS; ++q)
        a.Kc[q] = (float)exp(-(2.0 * q + 1.0) * (double)a.inv2s2);
    a.rec = c->bin_rec;
    a.size = c->bin_tot;
    a.l = c->bin_l;
    a.sum = c->sum;
    const size_t smem = loglik_smem(a.box, a.T, nb);
    switch (R) {
    case 0: launch_loglik_r<0>(c->bin_tmap, a, c->bin_grid, smem, c->stream); break;
    case 1: launch_loglik_r<1>(c->bin_tmap, a, c->bin_grid, smem, c->stream); break;
    case 2: launch_loglik_r<2>(c->bin_tmap, a, c->bin_grid, smem, c->stream); break;
    case 3: launch_loglik_r<3>(c->bin_tmap, a, c->bin_grid, smem, c->stream); break;
    case 4: launch_loglik_r<4>(c->bin_tmap, a, c->bin_grid, smem, c->stream); break;
    case 5: launch_loglik_r<5>(c->bin_tmap, a, c->bin_grid, smem, c->stream); break;
    case 6: launch_loglik_r<6>(c->bin_tmap, a, c->bin_grid, smem, c->stream); break;
    case 7: launch_loglik_r<7>(c->bin_tmap, a, c->bin_grid, smem, c->stream); break;
    default: launch_loglik_r<8>(c->bin_tmap, a, c->bin_grid, smem, c->stream); break;
    }
    c->launches += 2;
    return cudaGetLastError();
}

}  // namespace ppf
