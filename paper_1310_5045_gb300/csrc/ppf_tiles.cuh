// ppf_tiles.cuh -- block-level building blocks of the fixed-point resampling
// (Alg. 1 resampling step): tile staging, tile scans, and the parents of a
// range of systematic tickets.  Shared by the single-filter, RNA and batched
// resampling kernels.
#pragma once

#include <cstdint>

#include "ppf_device.cuh"
#include "ppf_internal.h"

namespace ppf {

// A tile is held in registers: thread t of TILE_THREADS has the 16 consecutive
// particles [16 t, 16 t + 16), a warp 512 of them (a strip), their weights
// quantised and summed there.  The sums before a warp come from the totals
// pass, which leaves the prefix of every tile's 8 strips, or, where a group
// does not start on a tile, from a scan over the block's warps.
//
// The weights come as 16-byte vectors wherever the plane starts: the address
// is rounded down to a 16-byte boundary, a fifth vector is read when it was
// not on one, and the (block-uniform) remainder picks the 16 values.  A
// thread whose vectors would leave [0, N) of the plane loads its values one by
// one.  -inf (weight 0) beyond n.  Lanes read 64 bytes apart, so a load
// instruction touches every other sector of its lines, but all sectors are
// used by the thread's own next loads, and no shared-memory transposition
// (16 stores, 16 loads and a barrier per tile) is needed.
__device__ __forceinline__ void tile_load16(const float *__restrict__ lw, int64_t N, int64_t lo, int n,
                                            float (&v)[TILE_ITEMS])
{
    const int e0 = (int)threadIdx.x * TILE_ITEMS;
    const int a = (int)((reinterpret_cast<uintptr_t>(lw + lo) >> 2) & 3u);
    const int64_t i0 = lo + e0 - a;
    if (e0 >= n) {
#pragma unroll
        for (int k = 0; k < TILE_ITEMS; ++k)
            v[k] = -INFINITY;
        return;
    }
    if (i0 >= 0 && i0 + (a ? TILE_ITEMS + 4 : TILE_ITEMS) <= N) {
        const float4 *p4 = reinterpret_cast<const float4 *>(lw + i0);
#pragma unroll
        for (int q = 0; q < TILE_ITEMS / 4; ++q) {
            const float4 x = __ldg(p4 + q);
            v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
        }
        if (a) {
            const float4 x = __ldg(p4 + TILE_ITEMS / 4);
            const float e[3] = {x.x, x.y, x.z};
#pragma unroll
            for (int k = 0; k < TILE_ITEMS; ++k) {
                const float v1 = k + 1 < TILE_ITEMS ? v[k + 1 < TILE_ITEMS ? k + 1 : 0] : e[0];
                const float v2 = k + 2 < TILE_ITEMS ? v[k + 2 < TILE_ITEMS ? k + 2 : 0] : e[k + 2 - TILE_ITEMS];
                const float v3 = k + 3 < TILE_ITEMS ? v[k + 3 < TILE_ITEMS ? k + 3 : 0] : e[k + 3 - TILE_ITEMS];
                v[k] = a == 1 ? v1 : (a == 2 ? v2 : v3);
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < TILE_ITEMS; ++k)
            v[k] = (e0 + k < n) ? __ldg(lw + lo + e0 + k) : -INFINITY;
    }
    if (e0 + TILE_ITEMS > n) {
#pragma unroll
        for (int k = 0; k < TILE_ITEMS; ++k)
            v[k] = (e0 + k < n) ? v[k] : -INFINITY;
    }
}

// The fixed-point sums of a tile: loc[k] the thread's weights up to and with
// its k-th, pre the tile's weights before the thread.
struct TileSums {
    uint64_t loc[TILE_ITEMS];
    uint64_t pre;
};

__device__ __forceinline__ void tile_quantise(const float (&v)[TILE_ITEMS], float M, int s, TileSums &ts)
{
#pragma unroll
    for (int k = 0; k < TILE_ITEMS; k += 2)
        quantise2(v[k], v[k + 1], M, s, ts.loc[k], ts.loc[k + 1]);
#pragma unroll
    for (int k = 1; k < TILE_ITEMS; ++k)
        ts.loc[k] += ts.loc[k - 1];
}

// The weights of the warps before are known (below): no barrier.
__device__ __forceinline__ void strip_scan(TileSums &ts, uint64_t below)
{
    const uint64_t mine = ts.loc[TILE_ITEMS - 1];
    ts.pre = below + warp_incl_scan_u64(mine) - mine;
}

// floor(x / d) for a fixed divisor d >= 1 and any x < 2^64, from the
// precomputed m = floor((2^64 - 1) / d): the product estimate floor(x m / 2^64)
// lies within 2 below the quotient and never above it.
struct Divisor {
    uint64_t m;
    uint32_t d;
};

__host__ __device__ inline Divisor make_divisor(uint32_t d)
{
    Divisor v;
    v.m = ~0ull / d;
    v.d = d;
    return v;
}

__device__ __forceinline__ uint64_t div_by(uint64_t x, Divisor v, uint32_t *rem)
{
    uint64_t q = __umul64hi(x, v.m);
    uint64_t r = x - q * v.d;
    while (r >= v.d) {
        ++q;
        r -= v.d;
    }
    *rem = (uint32_t)r;
    return q;
}

// The ticket grid of one systematic draw: nt tickets at (u + jQ)/nt of the
// cumulative fixed-point weight, Q = qN nt + qR.
struct TicketGrid {
    uint64_t Q, u, qN;
    uint32_t qR;
    Divisor nt;
};

__device__ __forceinline__ TicketGrid ticket_grid(uint64_t Q, uint64_t u, uint64_t qN, uint32_t qR, Divisor nt)
{
    TicketGrid g;
    g.Q = Q;
    g.u = u;
    g.qN = qN;
    g.qR = qR;
    g.nt = nt;
    return g;
}

// The threshold of ticket j, thr_j = floor((u + jQ)/nt) = j qN + floor((u + j qR)/nt):
// exact in 64-bit arithmetic (j < nt < 2^31 and u < Q <= 2^63, so
// u + j qR < 2^64).
__device__ __forceinline__ uint64_t ticket_threshold(int64_t j, const TicketGrid &tg)
{
    uint32_t r;
    return (uint64_t)j * tg.qN + div_by(tg.u + (uint64_t)j * tg.qR, tg.nt, &r);
}

// Number of tickets below cumulative weight c, #{j in [0, nt) : u + jQ < nt c}
// = #{j : thr_j < c} (thr_j < c iff (u + jQ)/nt < c for integer c): a float
// estimate c nt / Q, corrected once by the float estimate of the distance
// from c to the estimate's exact threshold, then moved to the exact boundary
// by comparing thresholds (they do not decrease with j).  No 128-bit or FP64
// arithmetic.
__device__ __forceinline__ int64_t tickets_below_grid(uint64_t c, const TicketGrid &tg)
{
    const int64_t n = tg.nt.d;
    const float rstep = (float)n / (float)tg.Q;
    int64_t j = (int64_t)((float)c * rstep);
    j = j < 0 ? 0 : (j > n - 1 ? n - 1 : j);
    const int64_t d = (int64_t)(c - ticket_threshold(j, tg));
    j += (int64_t)floorf((float)d * rstep);
    j = j < 0 ? 0 : (j > n ? n : j);
    while (j > 0 && ticket_threshold(j - 1, tg) >= c)
        --j;
    while (j < n && ticket_threshold(j, tg) < c)
        ++j;
    return j;
}

// The parents of a run of tickets among the particles of one tile.
//
// Ticket j of a draw sits at p_j = (u + jQ)/nt of the cumulative weight; its
// parent is the first particle whose inclusive sum C exceeds floor(p_j).  So
// the particle with sums (C-, C] holds the run's tickets [b(C-), b(C)),
// b(C) = #{m in [0, L): thr_{j_lo + m} < C}.  Every thread counts b for its
// own 16 sums in registers and writes the particle's index at the place of its
// first ticket in shared memory (a "head"; nothing for a particle without
// tickets).  Then the warps take chunks of 256 places and fill the gaps by a
// running maximum, within a chunk and over the chunks' last heads.  (Chunks of
// places, not each warp its own particles' tickets: a strip can hold several
// times another's.)
// About 40 instructions per particle and 8 per ticket; the merge of the sums
// with the thresholds that this replaces walked every particle and every
// ticket serially behind a shared-memory read (205 per particle and ticket
// together).
//
// The count is a fixed-point quotient, y = (C - p_{j_lo}) nt / Q: a distance
// scaled into 32 bits times v = nt / Q scaled to 2^30..2^32, the upper half of
// the product in units of 2^-16 ticket.  The roundings of the distance, of v,
// of the product and of the first ticket's place stay below 6 units in all, so
// when the fraction is not within 8 units of a whole ticket the count is
// certain; otherwise (2.4e-4 of the particles) it is settled by comparing C
// with that ticket's exact threshold.  A run that holds all tickets of its tile
// measures the distance from the tile's start (below L + 2 tickets); one of
// several runs of a tile measures it from its own first ticket, the sums
// clamped to the run first.
constexpr int STRIPS = TILE_THREADS / 32;        // strips (warps) of a tile
constexpr int CHUNK = 256;                       // places a warp fills at a time
constexpr int COUNT_MARGIN = 8;                  // units of 2^-16 ticket
static_assert(ITEM_TICKETS < (1 << 13), "the counts' fixed point holds runs below 2^13 tickets");

// Shared memory of a block of NT threads that draws parents: 32 places per
// thread, up to 3 of them before a run's first ticket.
template <int NT>
struct ParentSmemT {
    static constexpr int RUN = 32 * NT - 8;  // tickets of a run, at most
    alignas(16) uint16_t place[32 * NT];
    uint64_t red[NT / 32];
    uint32_t last[32 * NT / CHUNK];  // the last head of each chunk of places
};
typedef ParentSmemT<TILE_THREADS> ParentSmem;
static_assert(ParentSmem::RUN == ITEM_TICKETS && 32 * TILE_THREADS <= 32 * CHUNK, "one lane per chunk");

// The scan of the threads' sums over a block of NT threads.  red: one word per
// warp, the warp totals.  One barrier (the caller separates two uses of red by
// another).
template <int NT>
__device__ __forceinline__ void tile_scan(TileSums &ts, ParentSmemT<NT> &sm)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t mine = ts.loc[TILE_ITEMS - 1];
    const uint64_t incl = warp_incl_scan_u64(mine);
    if (lane == 31)
        sm.red[warp] = incl;
    __syncthreads();
    // the totals of the warps before: one word per lane, summed over NW lanes
    uint64_t below = (lane & (NW - 1)) < warp ? sm.red[lane & (NW - 1)] : 0ull;
#pragma unroll
    for (int o = 1; o < NW; o <<= 1)
        below += __shfl_xor_sync(0xffffffffu, below, o);
    ts.pre = below + incl - mine;
}

// its total, after the scan
template <int NT>
__device__ __forceinline__ uint64_t tile_total(const ParentSmemT<NT> &sm)
{
    uint64_t total = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w)
        total += sm.red[w];
    return total;
}

// nt / Q of a draw: y = (C - ..) 2^-sr 2^sl v 2^-48, v in [2^30, 2^32)
struct TicketScale {
    uint32_t v;
    int32_t sr, sl;  // right and left shift of the distance (one of them 0)
};

__device__ __forceinline__ TicketScale ticket_scale(uint64_t Q, uint32_t nt)
{
    const int lq = __clzll((long long)Q), ln = __clz((int)nt);  // Q >= 1, nt >= 1
    const uint32_t qt = (uint32_t)((Q << lq) >> 32), nn = nt << ln;
    TicketScale s;
    s.v = (uint32_t)(((uint64_t)nn << 31) / qt);
    const int e = 15 - lq + ln;
    s.sr = e > 0 ? e : 0;
    s.sl = e < 0 ? -e : 0;
    return s;
}

__device__ __forceinline__ uint32_t scaled_distance(uint64_t d, const TicketScale &s)
{
    return (uint32_t)(d >> s.sr) << s.sl;
}

// The place of ticket j, the first of a tile's tickets, above the tile's start
// c0, in units, taken from the margin: what the estimates of a run that holds
// all tickets of its tile add (whole), or of one measured from ticket j.
__device__ __forceinline__ int32_t run_offset(uint64_t c0, const TicketGrid &tg, const TicketScale &sc, int64_t j,
                                              bool whole)
{
    uint32_t rem;
    const uint64_t t0 = (uint64_t)j * tg.qN + div_by(tg.u + (uint64_t)j * tg.qR, tg.nt, &rem);
    // the threshold's fraction rem / nt counts when distances are scaled up
    const uint32_t fr = sc.sl ? (uint32_t)(((uint64_t)rem << sc.sl) / tg.nt.d) : 0u;
    return COUNT_MARGIN - (int32_t)__umulhi(fr, sc.v) -
           (whole ? (int32_t)__umulhi(scaled_distance(t0 - c0, sc), sc.v) : 0);
}

// One run of tickets of a tile, the same in every thread.
struct TicketRun {
    uint64_t c0;     // cumulative weight of the draw that the sums count from
    int64_t j_lo;    // first ticket
    int32_t L;       // tickets, at most ITEM_TICKETS
    int32_t off;     // run_offset
};

// The run of L tickets from j_lo, one of several of a tile that starts at c0:
// the tile's sums become distances from the run's first threshold, those
// below it 0 and those beyond its last one past the last.
__device__ __forceinline__ TicketRun part_run(TileSums &ts, uint64_t c0, const TicketGrid &tg, const TicketScale &sc,
                                              int64_t j_lo, int L)
{
    const uint64_t t0 = ticket_threshold(j_lo, tg), first = t0 - c0;
    const uint64_t span = ticket_threshold(j_lo + L - 1, tg) - t0 + 1;
    auto clamped = [&](uint64_t c) -> uint64_t {
        const uint64_t d = c > first ? c - first : 0ull;
        return d < span ? d : span;
    };
    const uint64_t pre = clamped(ts.pre);
#pragma unroll
    for (int k = 0; k < TILE_ITEMS; ++k)
        ts.loc[k] = clamped(ts.pre + ts.loc[k]) - pre;
    ts.pre = pre;
    return TicketRun{t0, j_lo, L, run_offset(c0, tg, sc, j_lo, false)};
}

// two 16-bit lanes
__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// The thread's counts of a run: before its particles, and up to and with each
// of them (two to a word).
struct ThreadCounts {
    int before;
    uint32_t upto[TILE_ITEMS / 2];
};

// grid(): the draw's ticket grid, only for the counts that need a threshold.
template <typename Grid>
__device__ __forceinline__ void count_tickets(const TileSums &ts, const TicketRun &run, const Grid &grid,
                                              const TicketScale &sc, ThreadCounts &tc)
{
    // the count in the upper half, the fraction (with the margin) in the lower
    const int32_t add = run.off + (1 << 16);
    auto estimate = [&](uint64_t c) -> uint32_t {
        return __umulhi(scaled_distance(c, sc), sc.v) + (uint32_t)add;
    };
    const uint32_t L2 = (uint32_t)run.L * 0x10001u;
    const uint32_t tb = estimate(ts.pre);
    uint32_t frac = tb & 0xFFFFu;
    frac |= frac << 16;
    tc.before = min((int)(tb >> 16), run.L);
#pragma unroll
    for (int k = 0; k < TILE_ITEMS; k += 2) {
        const uint32_t t0 = estimate(ts.pre + ts.loc[k]), t1 = estimate(ts.pre + ts.loc[k + 1]);
        tc.upto[k / 2] = min_u16x2(__byte_perm(t0, t1, 0x7632), L2);
        frac = min_u16x2(frac, __byte_perm(t0, t1, 0x5410));
    }
    if (min(frac & 0xFFFFu, frac >> 16) >= 2 * COUNT_MARGIN)
        return;
    // some estimate lies near a whole ticket (0.4 % of the threads)
    const TicketGrid tg = grid();
    uint32_t near = (tb & 0xFFFFu) < 2 * COUNT_MARGIN ? 1u << TILE_ITEMS : 0u;
#pragma unroll
    for (int k = 0; k < TILE_ITEMS; ++k)
        near |= (estimate(ts.pre + ts.loc[k]) & 0xFFFFu) < 2 * COUNT_MARGIN ? 1u << k : 0u;
    while (near) {
        uint64_t c = ts.pre;  // the last near item's sum
#pragma unroll
        for (int q = 0; q < TILE_ITEMS; ++q)
            c = (near >> q) & 1u ? ts.pre + ts.loc[q] : c;
        // the whole ticket it lies near is the one below the estimate, which
        // carries the margin: that ticket's threshold decides
        int b = (int)(estimate(c) >> 16) - 1;
        b = (b >= 0 && b < run.L && ticket_threshold(run.j_lo + b, tg) >= run.c0 + c) ? b : min(b + 1, run.L);
        // for every item with that sum (many particles weigh nothing)
        if (c == ts.pre) {
            tc.before = b;
            near &= (1u << TILE_ITEMS) - 1u;
        }
#pragma unroll
        for (int q = 0; q < TILE_ITEMS; ++q)
            if (ts.pre + ts.loc[q] == c) {
                tc.upto[q / 2] = __byte_perm(tc.upto[q / 2], (uint32_t)b, (q & 1) ? 0x5410 : 0x3254);
                near &= ~(1u << q);
            }
    }
}

// Clears the places of a run whose first ticket is at place a; a barrier must follow.
template <int NT>
__device__ __forceinline__ void clear_places(ParentSmemT<NT> &sm, int a, int L)
{
    uint4 *place4 = reinterpret_cast<uint4 *>(sm.place);
    for (int i = threadIdx.x; 8 * i < a + L; i += NT)
        place4[i] = make_uint4(0u, 0u, 0u, 0u);
}

// The parents of a run's tickets; the places are cleared and a barrier has
// passed since.  a = em.lead(j_lo): the empty places (0..3) before the first.
// With Emit::DIRECT em.four(x, y, j) gets the parents (local indices, 16 bits
// each) of four places that lie wholly inside the run, j the ticket of the
// first, and em.one the tickets of the two edges; else em.staged(place, L,
// j_lo) all filled places, after a barrier.  Called by every thread of the
// block; two barriers, and the caller puts one before the places are cleared again.
template <int NT, typename Grid, typename Emit>
__device__ __forceinline__ void block_parents(const TileSums &ts, const TicketRun &run, const Grid &grid,
                                              const TicketScale &sc, ParentSmemT<NT> &sm, const Emit &em)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    ThreadCounts tc;
    count_tickets(ts, run, grid, sc, tc);
    const int L = run.L, a = em.lead(run.j_lo);
    uint16_t *at = sm.place + a;
    const int i0 = (int)threadIdx.x * TILE_ITEMS;
    int prev = tc.before;
#pragma unroll
    for (int k = 0; k < TILE_ITEMS; k += 2) {
        const int b0 = (int)(tc.upto[k / 2] & 0xFFFFu), b1 = (int)(tc.upto[k / 2] >> 16);
        if (b0 > prev)
            at[prev] = (uint16_t)(i0 + k);
        if (b1 > b0)
            at[b0] = (uint16_t)(i0 + k + 1);
        prev = b1;
    }
    __syncthreads();
    // A chunk is two halves of 128 places, four consecutive places of each per
    // lane: the two scans over the lanes share a register, and a lane's four
    // parents of a half are one 16-byte store next to its neighbours'.
    constexpr int NW = NT / 32, PER_WARP = 32 * NT / CHUNK / NW;
    const int end = a + L;
    uint2 x[PER_WARP], y[PER_WARP];
    uint32_t before[PER_WARP];  // in the chunk: the last head before the lane's places, per half
#pragma unroll
    for (int q = 0; q < PER_WARP; ++q) {
        const int ch = warp + NW * q;
        if (CHUNK * ch < end) {
            const uint2 *w = reinterpret_cast<const uint2 *>(sm.place + CHUNK * ch) + lane;
            const int p0 = CHUNK * ch + 4 * lane, p1 = p0 + CHUNK / 2;
            x[q] = p0 < end ? w[0] : make_uint2(0u, 0u);
            y[q] = p1 < end ? w[32] : make_uint2(0u, 0u);
            x[q].x = max_u16x2(x[q].x, x[q].x << 16);
            y[q].x = max_u16x2(y[q].x, y[q].x << 16);
            x[q].y = max_u16x2(max_u16x2(x[q].y, x[q].y << 16), __byte_perm(x[q].x, 0u, 0x3232));
            y[q].y = max_u16x2(max_u16x2(y[q].y, y[q].y << 16), __byte_perm(y[q].x, 0u, 0x3232));
            uint32_t s = __byte_perm(x[q].y, y[q].y, 0x7632);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1)  // a lane without a lower neighbour gets its own value
                s = max_u16x2(s, __shfl_up_sync(0xffffffffu, s, o));
            const uint32_t all = __shfl_sync(0xffffffffu, s, 31);
            const uint32_t c = __shfl_up_sync(0xffffffffu, s, 1);
            before[q] = max_u16x2(lane == 0 ? 0u : c, all << 16);  // the second half follows the first
            if (lane == 0)
                sm.last[ch] = max(all & 0xFFFFu, all >> 16);
        }
    }
    __syncthreads();
    const uint32_t lasts = CHUNK * lane < end ? sm.last[lane] : 0u;
#pragma unroll
    for (int q = 0; q < PER_WARP; ++q) {
        const int ch = warp + NW * q;
        if (CHUNK * ch < end) {
            const uint32_t h = __reduce_max_sync(0xffffffffu, lane < ch ? lasts : 0u);
            const int p0 = CHUNK * ch + 4 * lane, p1 = p0 + CHUNK / 2;
            const uint32_t c = max_u16x2(before[q], h * 0x10001u);
            const uint32_t c0 = __byte_perm(c, 0u, 0x1010), c1 = __byte_perm(c, 0u, 0x3232);
            const uint2 f = make_uint2(max_u16x2(x[q].x, c0), max_u16x2(x[q].y, c0));
            const uint2 g = make_uint2(max_u16x2(y[q].x, c1), max_u16x2(y[q].y, c1));
            if constexpr (Emit::DIRECT) {
                if (p0 >= a && p1 + 4 <= end) {
                    em.four(f.x, f.y, run.j_lo + (p0 - a));
                    em.four(g.x, g.y, run.j_lo + (p1 - a));
                } else {  // at an edge of the run
                    const uint32_t v[4] = {f.x, f.y, g.x, g.y};
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int p = (e < 4 ? p0 : p1 - 4) + e;
                        if (p >= a && p < end)
                            em.one((int32_t)((v[e >> 1] >> (16 * (e & 1))) & 0xFFFFu), run.j_lo + (p - a));
                    }
                }
            } else {
                uint2 *w = reinterpret_cast<uint2 *>(sm.place + CHUNK * ch) + lane;
                if (p0 < end)
                    w[0] = f;
                if (p1 < end)
                    w[32] = g;
            }
        }
    }
    if constexpr (!Emit::DIRECT) {
        __syncthreads();
        em.staged(at, L, run.j_lo);
    }
}

// out[j] = base + parent, a 16-byte store per four places: the lead puts the
// places on the output's 16-byte boundaries.  The debug build checks every
// parent against [0, n) and every slot against [0, j_max).
struct EmitContig {
    static constexpr bool DIRECT = true;
    int32_t *__restrict__ out;
    int32_t base;
    int n;
    int64_t j_max;
    const int32_t *flags;
    __device__ __forceinline__ int lead(int64_t j) const
    {
        return (int)((reinterpret_cast<uintptr_t>(out + j) >> 2) & 3u);
    }
    __device__ __forceinline__ void four(uint32_t x, uint32_t y, int64_t j) const
    {
        const int4 v = make_int4((int32_t)(x & 0xFFFFu), (int32_t)(x >> 16), (int32_t)(y & 0xFFFFu), (int32_t)(y >> 16));
        if (PPF_DCHECK(v.x < n && v.y < n && v.z < n && v.w < n && j >= 0 && j + 4 <= j_max, flags, FLAG_INTERNAL))
            *reinterpret_cast<int4 *>(out + j) = make_int4(base + v.x, base + v.y, base + v.z, base + v.w);
    }
    __device__ __forceinline__ void one(int32_t i, int64_t j) const
    {
        if (PPF_DCHECK(i < n && j >= 0 && j < j_max, flags, FLAG_INTERNAL))
            out[j] = base + i;
    }
};

// o[k] = base + st[k] for k < m, called by every thread of the block: up to
// three single stores reach a 16-byte boundary of o, then four tickets per
// thread and iteration as int4.  The debug build checks every parent against [0, n).
__device__ __forceinline__ void store_staged(int32_t *__restrict__ o, const uint16_t *st, int m, int32_t base,
                                             int n, const int32_t *flags)
{
    const int head = (int)((4u - ((uint32_t)(reinterpret_cast<uintptr_t>(o) >> 2) & 3u)) & 3u);
    const int h = head < m ? head : m;
    const int m4 = (m - h) >> 2;
    const int t0 = h + 4 * m4;
    const int k = threadIdx.x;
    if (k < h && PPF_DCHECK(st[k] < n, flags, FLAG_INTERNAL))
        o[k] = base + st[k];
    int4 *o4 = reinterpret_cast<int4 *>(o + h);
    for (int q = k; q < m4; q += blockDim.x) {
        const int e = h + 4 * q;
        const int32_t p0 = st[e], p1 = st[e + 1], p2 = st[e + 2], p3 = st[e + 3];
        if (PPF_DCHECK(p0 < n && p1 < n && p2 < n && p3 < n, flags, FLAG_INTERNAL))
            o4[q] = make_int4(base + p0, base + p1, base + p2, base + p3);
    }
    if (k < m - t0 && PPF_DCHECK(st[t0 + k] < n, flags, FLAG_INTERNAL))
        o[t0 + k] = base + st[t0 + k];
}

// The tickets [j_lo, j_hi) of a tile, run by run.  all: they are all tickets
// of the tile's sums; off: their run_offset then.  A second run (a tile with
// more than a run's) gets the sums again from `again`.
template <int NT, typename Emit, typename Again>
__device__ __forceinline__ void draw_parents(TileSums &ts, uint64_t c0, const TicketGrid &tg, const TicketScale &sc,
                                             int64_t j_lo, int64_t j_hi, bool all, int32_t off,
                                             ParentSmemT<NT> &sm, const Emit &em, Again again)
{
    constexpr int RUN = ParentSmemT<NT>::RUN;
    for (int64_t c = j_lo; c < j_hi; c += RUN) {
        const int L = (int)((j_hi - c < RUN) ? j_hi - c : RUN);
        if (c > j_lo) {
            __syncthreads();  // the run before has left the places
            again(ts);
        }
        clear_places(sm, em.lead(c), L);
        TicketRun run{c0, c, L, off};
        if (!all || j_hi - j_lo > RUN)
            run = part_run(ts, c0, tg, sc, c, L);
        __syncthreads();
        block_parents(ts, run, [&]() { return tg; }, sc, sm, em);
    }
}

// A thread's weights of its warp's strip of a tile in strides (element
// strip + 32 k + lane), -inf beyond n: for sums, whose order does not matter.
// Aligned full strips are read as 16-byte vectors (element strip + 128 k + 4 lane ..).
__device__ __forceinline__ void strip_load(const float *__restrict__ lw, int n, float (&v)[TILE_ITEMS])
{
    const int lane = threadIdx.x & 31, s0 = (int)(threadIdx.x >> 5) * (TILE / STRIPS);
    if (s0 + TILE / STRIPS <= n && (reinterpret_cast<uintptr_t>(lw) & 15) == 0) {
        const float4 *p4 = reinterpret_cast<const float4 *>(lw + s0) + lane;
#pragma unroll
        for (int k = 0; k < TILE_ITEMS / 4; ++k) {
            const float4 x = __ldg(p4 + 32 * k);
            v[4 * k] = x.x; v[4 * k + 1] = x.y; v[4 * k + 2] = x.z; v[4 * k + 3] = x.w;
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < TILE_ITEMS; ++k) {
        const int e = s0 + 32 * k + lane;
        v[k] = e < n ? __ldg(lw + e) : -INFINITY;
    }
}

// The strips' totals (wsum, after a barrier) as a prefix into strip[0..STRIPS)
// and the tile's total into *total: warp 0.
__device__ __forceinline__ void store_strips(const uint64_t *wsum, uint64_t *__restrict__ strip,
                                             uint64_t *__restrict__ total)
{
    if (threadIdx.x >= 32)
        return;
    const int lane = threadIdx.x;
    const uint64_t x = lane < STRIPS ? wsum[lane] : 0ull;
    uint64_t incl = x;
#pragma unroll
    for (int o = 1; o < STRIPS; o <<= 1) {
        const uint64_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += t;
    }
    if (lane < STRIPS)
        strip[lane] = incl - x;
    if (lane == STRIPS - 1)
        *total = incl;
}

// A tile's sums: load, quantise, scan (one barrier, and one before for a
// second use of red).
template <int NT>
__device__ __forceinline__ void tile_sums(const float *__restrict__ lw, int64_t N, int64_t lo, int n, float M, int s,
                                          TileSums &ts, ParentSmemT<NT> &sm)
{
    float v[TILE_ITEMS];
    tile_load16(lw, N, lo, n, v);
    tile_quantise(v, M, s, ts);
    tile_scan(ts, sm);
}

}  // namespace ppf
