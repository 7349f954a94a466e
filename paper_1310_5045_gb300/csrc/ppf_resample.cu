// ppf_resample.cu -- the resampling step of Alg. 1 on 64-bit fixed-point
// weights, and the distributed schemes of Sec. 3-4 mapped onto particle groups:
//   systematic  one global offset u, ticket j at (u + jQ)/N of the cumulative
//               weight; the parent of ticket j is the first particle whose
//               cumulative weight C_i satisfies N C_i > u + jQ.
//   RPA         the same global tickets (proportional allocation); group g
//               holds the tickets of its own cumulative range, keeps the first
//               ones and routes its surplus to receivers following the Greedy
//               (Alg. 2), Sorted Greedy (Alg. 3) or Largest Gradient (Alg. 4)
//               schedule.
//   RNA         every group resamples its own slots from its own weights with
//               its own offset (non-proportional allocation); its offspring
//               carry the group weight, and the last floor(alpha min n_g) slots
//               of every group migrate to the next group of the ring.
// Every resampling kernel takes the N_eff threshold of Alg. 1: when the
// step's effective sample size is not below it, the kernels do nothing but
// mark the particles as kept (the next step carries their weights).
#include <cmath>
#include <cstddef>

#include "ppf_device.cuh"
#include "ppf_internal.h"
#include "ppf_tiles.cuh"

namespace ppf {

// Alg. 1 resamples only while N_eff < N_threshold (NaN N_eff: resample, which
// then reports the degenerate weights).
__device__ __forceinline__ bool kept_by_ess(const DevSummary *sum, double ess_thr)
{
    return sum->ess >= ess_thr;
}

// Balanced layout: group g holds n_g = q + [g < r] slots, q = floor(N/G) and
// r = N mod G (divided once on the host: 64-bit division is a long software
// sequence on the device), starting at off_g = g q + min(g, r).
struct Balanced {
    int64_t q, r;
};

inline Balanced balanced_layout(int64_t N, int32_t G)
{
    return Balanced{N / G, N % G};
}

__device__ __forceinline__ int64_t target_of(const Balanced &b, int32_t g)
{
    return b.q + ((int64_t)g < b.r ? 1 : 0);
}

__device__ __forceinline__ int64_t balanced_offset(const Balanced &b, int32_t g)
{
    return (int64_t)g * b.q + ((int64_t)g < b.r ? (int64_t)g : b.r);
}

// ---------------------------------------------------------------- R1 tiles
// Tile totals Q_t and the prefix of every tile's strips: every warp loads its
// strip (coalesced, all 16 values in flight together) and quantises them two
// at a time; the warp sums meet in shared memory.  Integer sums: any order.
// 33 us at 38M particles (48 before the quantiser's floor by a rounded-down
// addition), 22 us at the copy bandwidth.
__global__ void __launch_bounds__(TILE_THREADS, 5) tile_totals_kernel(const float *__restrict__ lw, int64_t N,
                                                                      const DevSummary *__restrict__ sum,
                                                                      double ess_thr, uint64_t *__restrict__ Qt,
                                                                      uint64_t *__restrict__ St)
{
    // Blocks take tiles blockIdx.x, + gridDim.x, ... (one each when the grid
    // has a block per tile).  A full, aligned tile's loads go out one tile
    // ahead, so that they are in flight while the block quantises the tile
    // before and waits at its reduction; any other tile is loaded when it is
    // its turn.
    if (!pdl_wait())
        return;
    pdl_trigger();
    if (kept_by_ess(sum, ess_thr))
        return;
    __shared__ uint64_t wsum[2][STRIPS];
    const int32_t T = (int32_t)((N + TILE - 1) / TILE);
    const int32_t T_full = (reinterpret_cast<uintptr_t>(lw) & 15) == 0 ? (int32_t)(N / TILE) : 0;
    const float M = sum->M;
    const int s = scale_bits(N);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float4 *v4 = reinterpret_cast<const float4 *>(lw) + warp * (TILE / STRIPS / 4) + lane;
    auto load = [&](int32_t t, float (&v)[TILE_ITEMS]) {
#pragma unroll
        for (int k = 0; k < TILE_ITEMS / 4; ++k) {
            const float4 x = __ldg(v4 + (int64_t)t * (TILE / 4) + 32 * k);
            v[4 * k] = x.x; v[4 * k + 1] = x.y; v[4 * k + 2] = x.z; v[4 * k + 3] = x.w;
        }
    };
    int buf = 0;
    auto finish = [&](int32_t t, const float (&v)[TILE_ITEMS]) {
        uint64_t acc = 0;
#pragma unroll
        for (int k = 0; k < TILE_ITEMS; k += 2) {
            uint64_t a, b;
            quantise2(v[k], v[k + 1], M, s, a, b);
            acc += a + b;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0)
            wsum[buf][warp] = acc;
        __syncthreads();  // (two buffers: the next tile's sums never meet this one's readers)
        if (threadIdx.x <= STRIPS) {
            uint64_t below = 0;
            for (int w = 0; w < (int)threadIdx.x; ++w)
                below += wsum[buf][w];
            if (threadIdx.x < STRIPS)
                St[(int64_t)t * STRIPS + threadIdx.x] = below;
            else
                Qt[t] = below;
        }
        buf ^= 1;
    };
    int32_t t = blockIdx.x;
    float v[TILE_ITEMS];
    if (t < T_full)
        load(t, v);
    for (; t < T_full; t += (int32_t)gridDim.x) {
        const int32_t tn = t + (int32_t)gridDim.x;
        float vn[TILE_ITEMS];
        if (tn < T_full)
            load(tn, vn);
        finish(t, v);
#pragma unroll
        for (int k = 0; k < TILE_ITEMS; ++k)
            v[k] = vn[k];
    }
    for (; t < T; t += (int32_t)gridDim.x) {
        const int64_t lo = (int64_t)t * TILE;
        strip_load(lw + lo, (int)(N - lo < TILE ? N - lo : TILE), v);
        finish(t, v);
    }
}

// Tile totals for RPA and ARNA, and for every group start inside the tile the
// local prefix before it.  A balanced layout puts one or two group starts in
// a tile: their prefixes are masked sums of the weights the threads already
// hold, reduced together with the total.  A tile with more starts (small
// groups, or the unequal groups LGS leaves) scans its weights in shared
// memory and reads the prefixes there.  Every tile also records the first
// group starting at or after it and how many start inside it (GT_MASKED + 1
// meaning more), for the fill's routing of kept tickets.
constexpr int GT_MASKED = 4;  // group starts per tile handled by masked sums

// The thread's part of the tile total (acc[GT_MASKED]) and of the prefix
// before each of the NS group starts at local positions spos[j] (acc[j]).
// A thread holds the quads of its warp's strip that strip_load gives it: a
// quad lies wholly below or above a start except the one quad that holds it,
// so each start costs a select of the quad's sum, and the partial quad a few more.
template <int NS>
__device__ __forceinline__ void masked_sums(const float (&v)[TILE_ITEMS], const int32_t *spos, float M, int s,
                                            uint64_t (&acc)[GT_MASKED + 1])
{
    constexpr int V = TILE_ITEMS / 4;
    const int q0 = (int)(threadIdx.x >> 5) * (TILE / STRIPS) + 4 * (int)(threadIdx.x & 31);
    int p[NS > 0 ? NS : 1];
#pragma unroll
    for (int j = 0; j < NS; ++j)
        p[j] = spos[j];
#pragma unroll
    for (int j = 0; j <= GT_MASKED; ++j)
        acc[j] = 0;
#pragma unroll
    for (int k = 0; k < V; ++k) {
        uint64_t w0, w1, w2, w3;
        quantise2(v[4 * k], v[4 * k + 1], M, s, w0, w1);
        quantise2(v[4 * k + 2], v[4 * k + 3], M, s, w2, w3);
        const uint64_t w01 = w0 + w1, qs = w01 + w2 + w3;
        acc[GT_MASKED] += qs;
        const int e0 = q0 + 128 * k;
#pragma unroll
        for (int j = 0; j < NS; ++j) {
            const int d = p[j] - e0;  // elements of the quad below start j
            const uint64_t part = d >= 4 ? qs : (d == 3 ? w01 + w2 : (d == 2 ? w01 : (d == 1 ? w0 : 0ull)));
            acc[j] += d > 0 ? part : 0ull;
        }
    }
}

__global__ void __launch_bounds__(TILE_THREADS, 5) tile_group_totals_kernel(
    const float *__restrict__ lw, int64_t N, const DevSummary *__restrict__ sum, double ess_thr,
    uint64_t *__restrict__ Qt, uint64_t *__restrict__ St, const int64_t *__restrict__ goff, int32_t G,
    uint64_t *__restrict__ Cbl, int32_t *__restrict__ tile_g)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    if (kept_by_ess(sum, ess_thr))
        return;
    __shared__ uint64_t sums[TILE];  // the tile's inclusive sums (only for tiles with many group starts)
    __shared__ uint64_t red[STRIPS];
    __shared__ int32_t gfirst, nstart;
    __shared__ int32_t spos[GT_MASKED];
    __shared__ uint64_t wsum[STRIPS][GT_MASKED], stot[STRIPS];
    const int64_t lo = (int64_t)blockIdx.x * TILE;
    const int n = (int)(N - lo < TILE ? N - lo : TILE);
    // the weights first, so that their loads are in flight during the search
    // warp 0 does for the tile's group starts
    const bool full = n == TILE && ((reinterpret_cast<uintptr_t>(lw + lo) & 15) == 0);
    float v[TILE_ITEMS];
    if (full)
        strip_load(lw + lo, n, v);
    if (threadIdx.x < 32) {
        // warp 0: the first g with goff[g] >= lo (goff[G] = N >= lo, so it
        // exists).  The first round probes the 32 groups around the balanced
        // layout's guess lo G / N, which holds the answer for a balanced
        // layout; otherwise 32-way rounds narrow [a, b] (invariant: the
        // answer lies in it) by a factor 32 each.
        const int lane = threadIdx.x;
        const int32_t guess = (int32_t)(lo * (int64_t)G / N);
        int32_t a = guess > 0 ? guess - 1 : 0, b = a + 31 < G ? a + 31 : G;
        {
            const int32_t p = a + lane;
            const unsigned m = __ballot_sync(0xffffffffu, p <= b && goff[p] >= lo);
            if (m & 1u) {          // goff[a] >= lo: the answer is at or before a
                b = a;
                a = 0;
            } else if (m != 0u) {  // the first lane at or past lo
                a = b = a + __ffs(m) - 1;
            } else {               // every probe below lo
                a = b + 1;
                b = G;
            }
        }
        while (a < b) {
            const int32_t step = (b - a + 30) / 31;  // 31 steps reach b
            const int32_t p = a + lane * step;
            const unsigned m = __ballot_sync(0xffffffffu, p <= b && goff[p] >= lo);
            if (m & 1u) {
                b = a;
            } else if (m != 0u) {
                const int f = __ffs(m) - 1;  // probes f - 1 below lo, f at or past it
                b = a + f * step;
                a = a + (f - 1) * step + 1;
            } else {
                const int last = (b - a) / step;  // the last probe (at or below b)
                a = a + last * step + 1;
            }
        }
        // the group starts inside the tile: lanes 0 .. GT_MASKED look at
        // goff[a + lane] (a prefix of them lie inside; lane GT_MASKED tells
        // whether there are more than GT_MASKED)
        const int32_t gg = a + lane;
        const bool inside = lane <= GT_MASKED && gg <= G && goff[gg] < lo + n;
        const unsigned mi = __ballot_sync(0xffffffffu, inside);
        const int ns = __popc(mi);
        if (inside && lane < GT_MASKED)
            spos[lane] = (int)(goff[gg] - lo);
        if (lane == 0) {
            gfirst = a;
            nstart = ns;
            tile_g[2 * blockIdx.x] = a;
            tile_g[2 * blockIdx.x + 1] = ns;
        }
    }
    __syncthreads();
    const int ns = nstart;
    const float M = sum->M;
    const int s = scale_bits(N);
    if (ns <= GT_MASKED && full) {
        uint64_t acc[GT_MASKED + 1];
        switch (ns) {  // uniform over the block: only the starts the tile has
        case 0: masked_sums<0>(v, spos, M, s, acc); break;
        case 1: masked_sums<1>(v, spos, M, s, acc); break;
        case 2: masked_sums<2>(v, spos, M, s, acc); break;
        case 3: masked_sums<3>(v, spos, M, s, acc); break;
        default: masked_sums<4>(v, spos, M, s, acc); break;
        }
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int j = 0; j <= GT_MASKED; ++j) {
            if (j < ns || j == GT_MASKED) {
                uint64_t x = acc[j];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    x += __shfl_xor_sync(0xffffffffu, x, o);
                if (lane == 0) {
                    if (j == GT_MASKED)
                        stot[warp] = x;
                    else
                        wsum[warp][j] = x;
                }
            }
        }
        __syncthreads();
        store_strips(stot, St + (int64_t)blockIdx.x * STRIPS, Qt + blockIdx.x);
        if (threadIdx.x >= 32 && threadIdx.x < 32 + ns) {
            uint64_t x = 0;
            for (int w = 0; w < STRIPS; ++w)
                x += wsum[w][threadIdx.x - 32];
            Cbl[gfirst + threadIdx.x - 32] = x;
        }
        return;
    }
    float w[TILE_ITEMS];
    tile_load16(lw, N, lo, n, w);
    __shared__ uint64_t bred[33];
    uint64_t btot;
    TileSums ts;
    tile_quantise(w, M, s, ts);
    const uint64_t pre = block_excl_scan_u64(ts.loc[TILE_ITEMS - 1], bred, &btot);
#pragma unroll
    for (int k = 0; k < TILE_ITEMS; ++k)
        sums[threadIdx.x * TILE_ITEMS + k] = pre + ts.loc[k];
    __syncthreads();
    if (threadIdx.x < STRIPS)
        red[threadIdx.x] = sums[TILE / STRIPS * (threadIdx.x + 1) - 1] -
                           (threadIdx.x ? sums[TILE / STRIPS * threadIdx.x - 1] : 0ull);
    __syncwarp();
    store_strips(red, St + (int64_t)blockIdx.x * STRIPS, Qt + blockIdx.x);
    __syncthreads();
    for (int32_t g = gfirst + threadIdx.x; g <= G; g += blockDim.x) {
        const int64_t pos = goff[g];
        if (pos >= lo + n)
            break;
        const int k = (int)(pos - lo);
        Cbl[g] = (k == 0) ? 0ull : sums[k - 1];
    }
}

// ---------------------------------------------------------------- R2 scan
// One block: exclusive tile prefix, total Q, ticket offset u, the scale of the
// ticket counts.  A proportional draw (rpa != 2) at a low N_eff also sets the
// next step to the direct likelihood path.
//
// PER > 0: a thread holds PER consecutive tile totals in registers, all its
// loads in flight together (T <= PER x threads); PER = 0 walks the tiles in
// rounds of blockDim, each closed by a block scan.  What the one thread used
// to do in turn after the scan (the spacing's division, the scale's, the
// offset's Philox block) four warps do at once.  At T = 9278 (38M) the prefix
// takes 5 us instead of 9, at T = 512 with as many groups everything 5 instead of 8.
//
// FULL (T <= SCAN_FULL_TILES, and as many groups for RPA and ARNA): the block
// also counts the tickets below each tile start and, for rpa != 0, each group
// start, one thread each, and lists the fill's further runs; otherwise
// tile_tickets_kernel does.
constexpr int SCAN_FULL_TILES = 1023;  // tile or group starts counted by the scan's own block

struct ScanArgs {
    int64_t N;
    int32_t T;
    const uint64_t *__restrict__ Qt;
    uint64_t *__restrict__ Ct;
    int64_t *__restrict__ Tt;
    int32_t *__restrict__ To;
    DevSummary *sum;
    double ess_thr;
    uint64_t seed;
    uint32_t fid, frame;
    const int64_t *__restrict__ goff;
    int32_t G, rpa;  // rpa: 0 systematic, 1 RPA, 2 ARNA
    const uint64_t *__restrict__ Cbl;
    int64_t *__restrict__ Tg;
    Divisor ndiv;
    int2 *__restrict__ extra;
};

// a tile's further runs (t, k), k >= 1, into the fill's list (in any order)
__device__ __forceinline__ void list_runs(DevSummary *sum, int2 *__restrict__ extra, int32_t t, int64_t tickets)
{
    const int64_t runs = (tickets + ITEM_TICKETS - 1) / ITEM_TICKETS;
    if (runs > 1) {
        const int32_t pos = atomicAdd(&sum->n_extra, (int32_t)(runs - 1));
        for (int64_t k = 1; k < runs; ++k)
            extra[pos + k - 1] = make_int2(t, (int32_t)k);
    }
}

template <int PER, bool FULL>
__global__ void __launch_bounds__(1024) tile_scan_kernel(ScanArgs A)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    static_assert(!FULL || PER == 1, "the block counts tickets for one tile per thread");
    __shared__ uint64_t red[33];
    __shared__ uint64_t s_u, s_qN;
    __shared__ uint32_t s_qR;
    __shared__ TicketScale s_sc;
    __shared__ uint64_t sC[FULL ? SCAN_FULL_TILES + 1 : 1];
    __shared__ int64_t sT[FULL ? SCAN_FULL_TILES + 1 : 1];
    DevSummary *sum = A.sum;
    const int32_t T = A.T;
    const int64_t N = A.N;
    uint64_t v[PER > 0 ? PER : 1];
    const int t0 = (int)threadIdx.x * PER;
#pragma unroll
    for (int k = 0; k < PER; ++k)
        v[k] = t0 + k < T ? __ldg(A.Qt + t0 + k) : 0ull;
    if (threadIdx.x == 0) {
        sum->n_split = 0;  // the two-stage draw's split list is rebuilt after the scan
        sum->n_runs = 0;
        sum->n_extra = 0;  // and the fill's list of further ticket runs
    }
    if (kept_by_ess(sum, A.ess_thr)) {  // N_eff test: keep the particles and the layout
        if (threadIdx.x == 0) {
            sum->degenerate = 1;
            sum->flags |= FLAG_KEPT;
            sum->links = 0;
            sum->moved = 0;
        }
        return;
    }
    uint64_t total = 0;
    if (PER > 0) {
        uint64_t loc = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k)
            loc += v[k];
        uint64_t run = block_excl_scan_u64(loc, red, &total);
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            if (t0 + k < T) {
                A.Ct[t0 + k] = run;  // exclusive tile prefix
                if (FULL)
                    sC[t0 + k] = run;
            }
            run += v[k];
        }
    } else {
        for (int base = 0; base < T; base += blockDim.x) {
            const int t = base + threadIdx.x;
            const uint64_t x = (t < T) ? A.Qt[t] : 0ull;
            uint64_t tot;
            const uint64_t ex = block_excl_scan_u64(x, red, &tot);
            if (t < T)
                A.Ct[t] = total + ex;
            total += tot;
        }
    }
    const bool deg = total == 0ull;
    if (threadIdx.x == 0) {
        A.Ct[T] = total;
        sum->Q = total;
        sum->degenerate = deg ? 1 : 0;
        if (deg)
            sum->flags |= FLAG_DEGENERATE;
        else if (A.rpa != 2 && sum->ess < (double)N / BIN_CONCENTRATE)
            sum->bin_next = 0;  // a concentrating proportional draw: the next step is direct
        if (!deg && !A.rpa) {
            // systematic keeps the group layout (the summary already holds its
            // extent, set whenever the layout changes); no routing
            sum->links = 0;
            sum->moved = 0;
        }
    } else if (threadIdx.x == 32) {
        uint32_t r;
        s_qN = div_by(total, A.ndiv, &r);
        s_qR = r;
        sum->qN = s_qN;
        sum->qR = r;
    } else if (threadIdx.x == 64 && !deg) {
        const TicketScale sc = ticket_scale(total, (uint32_t)N);
        s_sc = sc;
        sum->tsv = sc.v;
        sum->tsr = sc.sr;
        sum->tsl = sc.sl;
    } else if (threadIdx.x == 96) {
        s_u = deg ? 0ull : ticket_offset(A.seed, A.fid, A.frame, PURPOSE_RESAMPLE, 0u, total);
        sum->u = s_u;
    }
    if (!FULL || deg)
        return;
    __syncthreads();
    const TicketGrid tg = ticket_grid(total, s_u, s_qN, s_qR, A.ndiv);
    // the tickets below the tile starts, then those below the group starts
    const int starts = T + 1 + (A.rpa ? A.G + 1 : 0);
    for (int i = threadIdx.x; i < starts; i += blockDim.x) {
        const int g = i - (T + 1);
        const int64_t pos = g < 0 ? 0 : A.goff[g];
        const bool end = g < 0 ? i == T : pos >= N;
        const uint64_t c = end ? total : (g < 0 ? sC[i] : sC[pos / TILE] + A.Cbl[g]);
        const int64_t j = end ? N : tickets_below_grid(c, tg);
        if (g >= 0) {
            A.Tg[g] = j;
            continue;
        }
        A.Tt[i] = sT[i] = j;
        if (i < T)
            A.To[i] = run_offset(c, tg, s_sc, j, true);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < T; t += blockDim.x)
        list_runs(sum, A.extra, t, sT[t + 1] - sT[t]);
}

// The tickets below every tile start and, for RPA and ARNA, every group
// start, one thread each, after tile_scan_kernel's prefix, and the fill's
// list of further runs.
__global__ void __launch_bounds__(256) tile_tickets_kernel(ScanArgs A)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    DevSummary *__restrict__ sum = A.sum;
    if (sum->degenerate)
        return;  // kept by the N_eff test, or no usable weight
    const int32_t T = A.T;
    const int64_t N = A.N;
    const TicketGrid tg = ticket_grid(sum->Q, sum->u, sum->qN, sum->qR, A.ndiv);
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i <= T) {
        const int64_t a = (i == T) ? N : tickets_below_grid(A.Ct[i], tg);
        A.Tt[i] = a;
        if (i < T) {
            A.To[i] = run_offset(A.Ct[i], tg, TicketScale{sum->tsv, sum->tsr, sum->tsl}, a, true);
            list_runs(sum, A.extra, i, ((i + 1 == T) ? N : tickets_below_grid(A.Ct[i + 1], tg)) - a);
        }
    }
    if (A.rpa && i <= A.G) {
        const int64_t pos = A.goff[i];
        const uint64_t c = (pos >= N) ? sum->Q : A.Ct[pos / TILE] + A.Cbl[i];
        A.Tg[i] = (pos >= N) ? N : tickets_below_grid(c, tg);
    }
}

// The scan and the ticket counts; returns the launches made.
static int launch_scan(const ScanArgs &A, cudaStream_t stream)
{
    const int32_t T = A.T, most = A.rpa && A.G > T ? A.G : T;
    if (most <= SCAN_FULL_TILES) {
        const int starts = T + 1 + (A.rpa ? A.G + 1 : 0);
        int threads = (starts + 31) / 32 * 32;
        threads = threads < 128 ? 128 : (threads > 1024 ? 1024 : threads);
        launch_pdl(tile_scan_kernel<1, true>, 1, threads, 0, stream, A);
        return 1;
    }
    if (T <= 4 * 1024)
        launch_pdl(tile_scan_kernel<4, false>, 1, 1024, 0, stream, A);
    else if (T <= 16 * 1024)
        launch_pdl(tile_scan_kernel<16, false>, 1, 1024, 0, stream, A);
    else
        launch_pdl(tile_scan_kernel<0, false>, 1, 1024, 0, stream, A);
    launch_pdl(tile_tickets_kernel, (most + 256) / 256, 256, 0, stream, A);
    return 2;
}

// ------------------------------------------------ kept tickets, GS and SGS
// GS and SGS leave every group at its balanced size n_g: a sender keeps n_g
// of its o_g tickets and sends the rest, a receiver keeps all o_g < n_g and
// is filled up.  The first keep_g = min(o_g, n_g) tickets of group g (tickets
// Tg[g] <= j < Tg[g+1], in ticket order) therefore land in slots off_g +
// (j - Tg[g]) of the balanced layout whatever the schedule pairs; the fill
// writes them there directly and only the sent tickets go to their ticket
// slot of anc_sys, for the routing copy of the links.
constexpr int KT_GROUPS = GT_MASKED + 1;  // groups holding one tile's particles, at most, for the table
struct KeptTable {
    int n;                         // groups in the table; -1: too many, look every ticket up
    int64_t start[KT_GROUPS + 1];  // first ticket of each group, then the end of the last one
    int64_t keep_end[KT_GROUPS];   // first ticket each group sends
    int64_t shift[KT_GROUPS];      // a kept ticket j goes to slot j + shift
};

// The kept / sent split of the parents of tickets [c, c + m): every group's
// kept piece goes to anc (shifted to its balanced slot) and its sent piece to
// anc_sys + sent_shift, each as one store_staged run.  With kt.n < 0
// every ticket finds its group among Tg[0..G] by bisection (a tile crossed by
// more than KT_GROUPS groups).
struct EmitRouted {
    static constexpr bool DIRECT = false;
    const KeptTable &kt;
    int32_t *__restrict__ anc;
    int32_t *__restrict__ anc_sys;
    int64_t sent_shift;
    int32_t base;
    int n;
    int64_t N;
    int32_t G;
    const Balanced &bl;
    const int64_t *__restrict__ Tg;
    const int32_t *flags;
    __device__ __forceinline__ int lead(int64_t) const { return 0; }
    __device__ __forceinline__ void piece(int32_t *dst, int64_t slot, const uint16_t *st, int m) const
    {
        if (slot >= 0 && slot + m <= N)
            store_staged(dst + slot, st, m, base, n, flags);
        else if (threadIdx.x == 0)
            atomicOr(const_cast<int32_t *>(flags), FLAG_INTERNAL);  // inconsistent counts: never write out of bounds
    }
    __device__ __forceinline__ void staged(const uint16_t *st, int m, int64_t c) const
    {
        const int64_t ce = c + m;
        if (kt.n >= 0) {
            for (int e = 0; e < kt.n; ++e) {
                const int64_t a0 = c > kt.start[e] ? c : kt.start[e];
                const int64_t a1 = ce < kt.keep_end[e] ? ce : kt.keep_end[e];
                if (a0 < a1)
                    piece(anc, a0 + kt.shift[e], st + (a0 - c), (int)(a1 - a0));
                const int64_t b0 = c > kt.keep_end[e] ? c : kt.keep_end[e];
                const int64_t b1 = ce < kt.start[e + 1] ? ce : kt.start[e + 1];
                if (b0 < b1)
                    piece(anc_sys, b0 + sent_shift, st + (b0 - c), (int)(b1 - b0));
            }
            return;
        }
        for (int k = threadIdx.x; k < m; k += TILE_THREADS) {
            const int64_t j = c + k;
            int32_t a = 0, b = G - 1;  // the last g with Tg[g] <= j (Tg[0] = 0 <= j)
            while (a < b) {
                const int32_t mid = (a + b + 1) >> 1;
                if (__ldg(Tg + mid) <= j)
                    a = mid;
                else
                    b = mid - 1;
            }
            const int64_t s0 = __ldg(Tg + a), o = __ldg(Tg + a + 1) - s0;
            const int64_t nk = target_of(bl, a);
            const int64_t keep = o < nk ? o : nk;
            const int64_t slot = (j - s0 < keep) ? balanced_offset(bl, a) + (j - s0) : j + sent_shift;
            int32_t *dst = (j - s0 < keep) ? anc : anc_sys;
            if (slot >= 0 && slot < N && PPF_DCHECK(st[k] < n, flags, FLAG_INTERNAL))
                dst[slot] = base + st[k];
            else if (slot < 0 || slot >= N)
                atomicOr(const_cast<int32_t *>(flags), FLAG_INTERNAL);
        }
    }
};

// ------------------------------------------- the GS and SGS links, in a block
// What the RPA schedules read and write (see the RPA schedule below).
struct SchedArgs {
    int64_t N;
    int32_t G;
    int scheme;
    const int64_t *goff;
    int64_t *goff_new;
    const int64_t *Tg;
    uint64_t *key;      // [2 * G]  (sender keys, receiver keys)
    int64_t *val;       // [2 * G]  (sent, received; LGS)
    int32_t *seg_chunk; // [2G + 2]
    int64_t *seg_tick, *seg_dst, *seg_len;  // [2G + 1]
    DevSummary *sum;
    Balanced bl;     // the balanced targets n_g
};

// first index in sorted a[0..n) with a[i] > v
__device__ __forceinline__ int upper_bound_i32(const int32_t *a, int n, int32_t v)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (a[mid] > v)
            hi = mid;
        else
            lo = mid + 1;
    }
    return lo;
}

// Up to this many groups the GS and SGS schedule runs in the fill's own first
// block (their fills write the kept tickets, so only the links are left): its
// lists fit 33 KB next to the fill's buffers at four blocks per SM, and it
// needs no second stream, events or launch.  By itself the one-block schedule
// of a side stream took 33 us at 8 groups and 80 us at 1954, most of it a
// register sort that every thread ran whatever the count and global round
// trips; a fill of 8M particles takes 30 us.
constexpr int SCHED_SMALL = 2048;

__host__ __device__ inline int pow2_at_least(int n)
{
    int p = 64;
    while (p < n)
        p *= 2;
    return p;
}

inline size_t sched_small_bytes(int32_t G)
{
    return sizeof(uint64_t) * pow2_at_least(G) + sizeof(int32_t) * (2 * (size_t)G + 4);
}

// The links of GS and SGS: the senders' and receivers' amounts in list order
// (group order for GS; for SGS by amount, descending, ties by group) are
// pieces of [0, D), and every distinct piece start begins a link.  All starts
// of senders are links; a receiver's is one unless a sender starts there too.
// Output: the balanced offsets and one routing segment per sender and
// receiver (empty where its start is no link) with its copy work items.
// Called by every thread of one block; mem: sched_small_bytes(G).
__device__ void schedule_small(const SchedArgs &A, unsigned char *mem)
{
    __shared__ uint64_t red[33];
    const int32_t G = A.G;
    const Balanced &bl = A.bl;
    DevSummary *sum = A.sum;
    if (sum->degenerate) {
        for (int g = threadIdx.x; g <= G; g += blockDim.x)
            A.goff_new[g] = A.goff[g];
        if (threadIdx.x == 0) {
            sum->n_chunks = 0;
            sum->links = 0;
            sum->moved = 0;
        }
        return;
    }
    // key: class (receivers above), descending amount, group
    uint64_t *key = reinterpret_cast<uint64_t *>(mem);
    int32_t *tg = reinterpret_cast<int32_t *>(key + pow2_at_least(G));
    int32_t *P = tg + G + 1;  // prefix sums: the senders' and D, then the receivers' and D
    auto amount = [](uint64_t k) -> int32_t { return 0x7FFFFFFF - (int32_t)((k >> 32) & 0x7FFFFFFFu); };
    auto group = [](uint64_t k) -> int32_t { return (int32_t)(k & 0xFFFFu); };
    for (int g = threadIdx.x; g <= G; g += blockDim.x) {
        tg[g] = (int32_t)A.Tg[g];
        A.goff_new[g] = balanced_offset(bl, g);
    }
    __syncthreads();
    int nS, nR;
    {
        const int per = (G + (int)blockDim.x - 1) / (int)blockDim.x, g0 = (int)threadIdx.x * per;
        uint64_t c = 0;
        for (int g = g0; g < g0 + per && g < G; ++g) {
            const int32_t d = tg[g + 1] - tg[g] - (int32_t)target_of(bl, g);
            c += d > 0 ? 1ull : (d < 0 ? 1ull << 32 : 0ull);
        }
        uint64_t total;
        const uint64_t at = block_excl_scan_u64(c, red, &total);
        nS = (int)(uint32_t)total;
        nR = (int)(total >> 32);
        int ps = (int)(uint32_t)at, pr = nS + (int)(at >> 32);
        for (int g = g0; g < g0 + per && g < G; ++g) {
            const int32_t d = tg[g + 1] - tg[g] - (int32_t)target_of(bl, g);
            if (d > 0)
                key[ps++] = ((uint64_t)(uint32_t)(0x7FFFFFFF - d) << 32) | (uint64_t)g;
            else if (d < 0)
                key[pr++] = (1ull << 63) | ((uint64_t)(uint32_t)(0x7FFFFFFF + d) << 32) | (uint64_t)g;
        }
    }
    const int n = nS + nR;
    if (A.scheme != PPF_RPA_GS) {
        // bitonic sort in shared memory, one pair per thread and round; steps
        // within 64 keys stay within a warp
        const int n2 = pow2_at_least(n);
        for (int i = n + threadIdx.x; i < n2; i += blockDim.x)
            key[i] = ~0ull;
        __syncthreads();
        for (int k = 2; k <= n2; k *= 2)
            for (int j = k / 2; j > 0; j /= 2) {
                for (int p = threadIdx.x; p < n2 / 2; p += blockDim.x) {
                    const int i = 2 * p - (p & (j - 1));
                    const uint64_t x = key[i], y = key[i + j];
                    if ((x > y) == ((i & k) == 0)) {
                        key[i] = y;
                        key[i + j] = x;
                    }
                }
                if (j >= 64 || (j == 1 && k >= 64))
                    __syncthreads();
                else
                    __syncwarp();
            }
    }
    __syncthreads();
    const int per = (n + (int)blockDim.x - 1) / (int)blockDim.x;
    const int i0 = (int)threadIdx.x * per, i1 = i0 + per < n ? i0 + per : n;
    int32_t D;
    {
        uint64_t s = 0, total;
        for (int i = i0; i < i1; ++i)
            s += (uint64_t)(uint32_t)amount(key[i]);
        uint64_t run = block_excl_scan_u64(s, red, &total);
        D = (int32_t)(total / 2);  // what the senders give is what the receivers take
        for (int i = i0; i < i1; ++i) {
            P[i < nS ? i : i + 1] = (int32_t)(i < nS ? run : run - (uint64_t)D);
            run += (uint64_t)(uint32_t)amount(key[i]);
        }
        if (threadIdx.x == 0)
            P[nS] = P[n + 1] = D;
    }
    __syncthreads();
    const int32_t *PS = P, *PR = P + nS + 1;
    uint64_t c = 0;  // links above, copy work items below
    for (int i = i0; i < i1; ++i) {
        int si, rj;
        int32_t a;
        bool link = true;
        if (i < nS) {
            si = i;
            a = PS[i];
            rj = upper_bound_i32(PR, nR, a) - 1;
        } else {
            rj = i - nS;
            a = PR[rj];
            si = upper_bound_i32(PS, nS, a) - 1;
            link = PS[si] != a;
        }
        const int32_t e = PS[si + 1] < PR[rj + 1] ? PS[si + 1] : PR[rj + 1];
        const int32_t gs = group(key[si]), gr = group(key[nS + rj]);
        // a sender keeps n_s; a receiver keeps its o_r and is filled after them
        A.seg_tick[i] = tg[gs] + target_of(bl, gs) + (a - PS[si]);
        A.seg_dst[i] = balanced_offset(bl, gr) + (tg[gr + 1] - tg[gr]) + (a - PR[rj]);
        A.seg_len[i] = link ? e - a : 0;
        if (link)
            c += (1ull << 32) + (uint64_t)((e - a + COPY_CHUNK - 1) / COPY_CHUNK);
    }
    uint64_t total;
    uint32_t run = (uint32_t)block_excl_scan_u64(c, red, &total);
    for (int i = i0; i < i1; ++i) {
        A.seg_chunk[i] = (int32_t)run;
        run += (uint32_t)((A.seg_len[i] + COPY_CHUNK - 1) / COPY_CHUNK);
    }
    if (threadIdx.x == 0) {
        A.seg_chunk[n] = (int32_t)(uint32_t)total;
        A.seg_chunk[2 * G + 1] = n;  // the segment count
        sum->n_chunks = (int32_t)(uint32_t)total;
        sum->links = (int64_t)(total >> 32);
        sum->moved = D;
        sum->max_group = bl.q + (bl.r > 0 ? 1 : 0);
        sum->min_group = bl.q;
    }
}

// ---------------------------------------------------------------- R3 fill
// Block t < T takes tile t's first ITEM_TICKETS tickets, block T + e the e-th
// entry (t, k) of the list of further runs; a tile without tickets ends its
// block at once.  The tile's weights are quantised and summed in registers and
// the parents of the run's tickets drawn among them, straight to out[j]
// (systematic, LGS) or split into kept and sent tickets (GS, SGS: kr.anc set).
// Bound by instruction issue (65 thread instructions per particle and ticket,
// IPC 2.4, 64 registers): 98 us at 38M particles (208 before, with the merge),
// 22 us at 8M (47); with the kept / sent split 29 us at 8M (52).
struct KeptRoute {
    int32_t *anc;           // final ancestors; nullptr: every ticket to out[j]
    const int64_t *Tg;      // [G+1] tickets below each group start
    const int32_t *tile_g;  // [2T] per tile: first group starting at or after it, starts inside (capped)
    int32_t G;
    Balanced bl;            // the balanced layout GS and SGS leave
};

struct FillArgs {
    const float *__restrict__ lw;
    int64_t N;
    int32_t T;
    Divisor ndiv;
    const DevSummary *__restrict__ sum;
    const uint64_t *__restrict__ Ct;
    const int64_t *__restrict__ Tt;
    const int32_t *__restrict__ To;
    const uint64_t *__restrict__ St;
    const int2 *__restrict__ extra;
    int32_t *__restrict__ out;
    KeptRoute kr;
    int sched;      // the first block runs the schedule
    SchedArgs sa;
};

template <bool ROUTE>
__global__ void __launch_bounds__(TILE_THREADS, 4) fill_tiles_kernel(FillArgs A)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    const DevSummary *__restrict__ sum = A.sum;
    // the tile's bounds are read together with the flags that may end the block
    const int32_t deg = sum->degenerate, n_extra = sum->n_extra;
    int32_t t = blockIdx.x, k = 0;
    if (ROUTE && A.sched) {
        if (t == 0) {
            extern __shared__ uint64_t sched_mem[];  // sched_small_bytes(G)
            schedule_small(A.sa, reinterpret_cast<unsigned char *>(sched_mem));
            return;
        }
        --t;
    }
    if (t >= A.T) {
        if (deg || t - A.T >= n_extra)
            return;
        const int2 e = A.extra[t - A.T];
        t = e.x;
        k = e.y;
    }
    const int64_t tt0 = A.Tt[t], tt1 = A.Tt[t + 1];
    TicketRun run;
    run.c0 = A.Ct[t];
    run.off = A.To[t];
    run.j_lo = tt0 + (int64_t)k * ITEM_TICKETS;
    run.L = (int32_t)(tt1 - run.j_lo < ITEM_TICKETS ? tt1 - run.j_lo : ITEM_TICKETS);
    if (deg || run.L <= 0)
        return;  // kept by the N_eff test, no usable weight, or a tile without tickets
    __shared__ ParentSmem sm;
    __shared__ KeptTable kt;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t N = A.N, lo = (int64_t)t * TILE;
    const int n = (int)(N - lo < TILE ? N - lo : TILE);
    float v[TILE_ITEMS];
    tile_load16(A.lw, N, lo, n, v);
    const uint64_t below = A.St[(int64_t)t * STRIPS + warp];
    const TicketScale sc{sum->tsv, sum->tsr, sum->tsl};
    auto grid = [&]() {  // (read where it is needed, not held in registers)
        return ticket_grid(__ldcg(&sum->Q), __ldcg(&sum->u), __ldcg(&sum->qN), __ldcg(&sum->qR), A.ndiv);
    };
    if (ROUTE && warp == STRIPS - 1) {
        // the groups holding the tile's particles, one lane each (ga, the
        // group of the tile's first particle, to gb, the last group starting
        // inside it)
        const KeptRoute &kr = A.kr;
        const int32_t gf = __ldg(kr.tile_g + 2 * t), ns = __ldg(kr.tile_g + 2 * t + 1);
        if (ns > GT_MASKED) {
            if (lane == 0)
                kt.n = -1;
        } else {
            const int32_t ga = gf > 0 ? gf - 1 : 0, gb = gf + ns - 1;  // gf = 0 only for tile 0, with ns >= 1
            const int ng = gb - ga + 1;
            if (lane <= ng) {
                const int32_t g = ga + lane;
                const int64_t t0 = __ldg(kr.Tg + g);
                kt.start[lane] = t0;
                if (lane < ng) {
                    const int64_t o = __ldg(kr.Tg + g + 1) - t0, nk = target_of(kr.bl, g);
                    kt.keep_end[lane] = t0 + (o < nk ? o : nk);
                    kt.shift[lane] = balanced_offset(kr.bl, g) - t0;
                }
            }
            if (lane == 0)
                kt.n = ng;
        }
    }
    auto draw = [&](const auto &em) {
        clear_places(sm, em.lead(run.j_lo), run.L);
        TileSums ts;
        tile_quantise(v, sum->M, scale_bits(N), ts);
        strip_scan(ts, below);
        if (tt1 - tt0 > ITEM_TICKETS)
            run = part_run(ts, run.c0, grid(), sc, run.j_lo, run.L);
        __syncthreads();  // the cleared places and the table
        block_parents(ts, run, grid, sc, sm, em);
    };
    if constexpr (ROUTE)
        draw(EmitRouted{kt, A.kr.anc, A.out, 0, (int32_t)lo, n, N, A.kr.G, A.kr.bl, A.kr.Tg, &sum->flags});
    else
        draw(EmitContig{A.out, (int32_t)lo, n, N, &sum->flags});
}

static cudaError_t launch_fill(const FillArgs &A, cudaStream_t stream)
{
    const int runs = A.T + (int)(A.N / ITEM_TICKETS) + 1;
    if (A.kr.anc)
        launch_pdl(fill_tiles_kernel<true>, runs + (A.sched ? 1 : 0), TILE_THREADS,
                   A.sched ? sched_small_bytes(A.sa.G) : 0, stream, A);
    else
        launch_pdl(fill_tiles_kernel<false>, runs, TILE_THREADS, 0, stream, A);
    return cudaGetLastError();
}

// The systematic draw on the caller's buffers (the allocation-free entry
// point): tile totals, scan, ticket counts, fill.  Resamples every time.
cudaError_t launch_draw_plain(const float *lw, int64_t N, DevSummary *sum, uint64_t *Qt, uint64_t *St, uint64_t *Ct,
                              int64_t *Tt, int32_t *To, int2 *extra, uint64_t seed, uint32_t fid, uint32_t frame,
                              int32_t *out, cudaStream_t stream)
{
    const int32_t T = (int32_t)((N + TILE - 1) / TILE);
    const Divisor nd = make_divisor((uint32_t)N);
    launch_pdl(tile_totals_kernel, T, TILE_THREADS, 0, stream, lw, N, (const DevSummary *)sum, (double)INFINITY, Qt, St);
    launch_scan(ScanArgs{N, T, Qt, Ct, Tt, To, sum, INFINITY, seed, fid, frame, nullptr, 0, 0, nullptr, nullptr, nd,
                         extra},
                stream);
    const KeptRoute none{nullptr, nullptr, nullptr, 0, Balanced{0, 0}};
    return launch_fill(FillArgs{lw, N, T, nd, sum, Ct, Tt, To, St, extra, out, none, 0, SchedArgs{}}, stream);
}

// ------------------------------------------------ two-stage RPA, stage 2
// Every group g draws its N_g = Tg[g+1] - Tg[g] offspring (stage 1: the
// global tickets of its cumulative range) again inside the group, by its own
// systematic draw over the same fixed-point weights with the offset from
// Philox(seed; g, frame, filter, GROUP).  They are written, in ticket order,
// where the global draw would have put them (ticket slots Tg[g] ..), so the
// RPA schedule and routing copy apply unchanged; with kept_anc set (GS, SGS)
// the group's first keep_g tickets go straight to its balanced slots in
// kept_anc instead, as in the one-stage fill.
//
// The group's total and the cumulative weight below any tile start inside it
// come from the global prefix of the tile pass (C(p) = Ct[p / TILE] + the
// local prefix at p; integer sums, so exactly the group's own sums), which
// lets a large group be split at tile boundaries: a group spanning more
// than GROUP_SPLIT particles is drawn by one block for its head (up to the
// first tile boundary) and one block per interior tile.  A smaller group
// with more than ITEM_TICKETS offspring is split by tickets instead: its
// block draws the first ITEM_TICKETS, and one more block each further run
// of ITEM_TICKETS, so that no block carries a heavy group alone.
constexpr int64_t GROUP_SPLIT = 2 * TILE;

// One thread per group: the group's draw; a large group lists all its tile
// parts (tile, g, run 0), a heavy small group its further runs (-1, g, r),
// r >= 1, in the split list (four ints an entry; the order of the list does
// not matter: every entry writes its own tickets).
__global__ void __launch_bounds__(256) group_grid_kernel(
    int64_t N, int32_t G, const int64_t *__restrict__ goff, const int64_t *__restrict__ Tg,
    const uint64_t *__restrict__ Ct, const uint64_t *__restrict__ Cbl, DevSummary *__restrict__ sum, double ess_thr,
    uint64_t seed, uint32_t fid, uint32_t frame, GroupGrid *__restrict__ grid, int4 *__restrict__ split,
    Balanced bl)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G || kept_by_ess(sum, ess_thr) || sum->degenerate)
        return;
    const uint64_t Q = sum->Q;
    const int64_t a = goff[g], e = goff[g + 1];
    const uint64_t ca = (a >= N) ? Q : Ct[a / TILE] + Cbl[g];
    const uint64_t ce = (e >= N) ? Q : Ct[e / TILE] + Cbl[g + 1];
    const int64_t nt = Tg[g + 1] - Tg[g];
    GroupGrid gg;
    gg.Ca = ca;
    gg.Q = ce - ca;
    gg.nt = (nt > 0 && gg.Q > 0) ? (uint32_t)nt : 0u;
    gg.u = gg.qN = gg.dm = 0;
    gg.qR = gg.tsv = 0;
    gg.tsr = gg.tsl = gg.off = 0;
    gg.p0 = a;
    gg.p1 = e;
    gg.tg0 = Tg[g];
    {
        const int64_t nk = target_of(bl, g);
        gg.keep = nt < nk ? nt : nk;
        gg.shift = balanced_offset(bl, g);
    }
    if (gg.nt > 0) {
        gg.u = ticket_offset(seed, fid, frame, PURPOSE_GROUP, (uint32_t)g, gg.Q);
        gg.dm = make_divisor(gg.nt).m;
        gg.qN = gg.Q / gg.nt;
        gg.qR = (uint32_t)(gg.Q % gg.nt);
        const TicketScale sc = ticket_scale(gg.Q, gg.nt);
        gg.tsv = sc.v;
        gg.tsr = sc.sr;
        gg.tsl = sc.sl;
        gg.off = run_offset(0, ticket_grid(gg.Q, gg.u, gg.qN, gg.qR, Divisor{gg.dm, gg.nt}), sc, 0, true);
    }
    grid[g] = gg;
    if (gg.nt == 0)
        return;
    if (e - a > GROUP_SPLIT) {
        const int64_t t1 = a / TILE, t2 = (e - 1) / TILE;  // every tile the group reaches
        const int32_t pos = atomicAdd(&sum->n_split, (int32_t)(t2 - t1 + 1));
        for (int64_t t = t1; t <= t2; ++t)
            split[pos + (t - t1)] = make_int4((int32_t)t, g, 0, 0);
    } else if (nt > ITEM_TICKETS) {
        const int32_t runs = (int32_t)((nt + ITEM_TICKETS - 1) / ITEM_TICKETS);
        const int32_t pos = atomicAdd(&sum->n_split, runs - 1);
        for (int32_t r = 1; r < runs; ++r)
            split[pos + r - 1] = make_int4(-1, g, r, 0);
    }
}

// The part of a large group in one tile: its particles and the group's
// cumulative weight below them.
__device__ __forceinline__ void tile_part(const GroupGrid &gg, int32_t t, const uint64_t *__restrict__ Ct,
                                          int64_t &p0, int64_t &p1, uint64_t &carry)
{
    const int64_t lo = (int64_t)t * TILE;
    p0 = lo > gg.p0 ? lo : gg.p0;
    p1 = lo + TILE < gg.p1 ? lo + TILE : gg.p1;
    carry = p0 == gg.p0 ? 0ull : Ct[t] - gg.Ca;
}

// One thread per tile part listed by group_grid_kernel: a part with more than
// ITEM_TICKETS offspring appends its further runs (tile, g, r), r >= 1, so
// that a heavy tile of a large group is drawn by several blocks too.
__global__ void __launch_bounds__(256) split_runs_kernel(const uint64_t *__restrict__ Ct,
                                                         const GroupGrid *__restrict__ grid, int4 *__restrict__ split,
                                                         DevSummary *__restrict__ sum, double ess_thr)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    if (kept_by_ess(sum, ess_thr) || sum->degenerate)
        return;
    const int32_t n0 = sum->n_split;  // the entries group_grid_kernel listed; the runs go after them
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n0; i += gridDim.x * blockDim.x) {
        const int4 en = split[i];
        if (en.x < 0 || en.z != 0)
            continue;
        const GroupGrid gg = grid[en.y];
        int64_t p0, p1;
        uint64_t c_lo;
        tile_part(gg, en.x, Ct, p0, p1, c_lo);
        const uint64_t c_hi = p1 == gg.p1 ? gg.Q : Ct[en.x + 1] - gg.Ca;
        const int64_t nt = gg.nt;
        const int64_t j_lo = c_lo == 0 ? 0 : tickets_below(c_lo, nt, gg.u, gg.Q);
        const int64_t j_hi = c_hi == gg.Q ? nt : tickets_below(c_hi, nt, gg.u, gg.Q);
        if (j_hi - j_lo > ITEM_TICKETS) {
            const int32_t runs = (int32_t)((j_hi - j_lo + ITEM_TICKETS - 1) / ITEM_TICKETS);
            const int32_t pos = n0 + atomicAdd(&sum->n_runs, runs - 1);
            for (int32_t r = 1; r < runs; ++r)
                split[pos + r - 1] = make_int4(en.x, en.y, r, 0);
        }
    }
}

// One work item of the two-stage draw: particles [p0, p1) of group gg, carry
// the group's cumulative weight below p0.  Its tickets: the group's [j0, j1)
// among them (run < 0), or run `run` of ITEM_TICKETS among the tickets of a
// one-tile part (run >= 0).
__device__ __forceinline__ void group_fill_item(const float *__restrict__ lw, int64_t N, int32_t G,
                                                const int64_t *__restrict__ Tg, const GroupGrid &gg, int64_t p0,
                                                int64_t p1, int64_t j0, int64_t j1, int32_t run, uint64_t carry,
                                                float M, int s, const DevSummary *__restrict__ sum,
                                                int32_t *__restrict__ out, int32_t *__restrict__ kept_anc,
                                                const Balanced &bl, ParentSmem &sm)
{
    const int64_t nt = gg.nt;
    Divisor dv;
    dv.m = gg.dm;
    dv.d = gg.nt;
    const TicketGrid tg = ticket_grid(gg.Q, gg.u, gg.qN, gg.qR, dv);
    KeptTable kt;  // one group, in local ticket numbers
    kt.n = 1;
    kt.start[0] = 0;
    kt.start[1] = nt;
    kt.keep_end[0] = kept_anc ? gg.keep : 0;  // LGS: every ticket to its ticket slot
    kt.shift[0] = gg.shift;
    // chunks of at most TILE particles; the local tickets of a chunk with
    // cumulative weight [carry, carry + total) inside the group are
    // [T(carry), T(carry + total)), T the count below of the nt tickets
    for (int64_t c0 = p0; c0 < p1; c0 += TILE) {
        const int n = (int)(p1 - c0 < TILE ? p1 - c0 : TILE);
        TileSums ts;
        tile_sums(lw, N, c0, n, M, s, ts, sm);
        const uint64_t tot = tile_total(sm);
        // no ticket lies below the group's start, all of them below its end
        const int64_t c_lo = carry == 0 ? 0 : tickets_below(carry, nt, gg.u, gg.Q);
        const int64_t c_hi = c0 + n == gg.p1 ? nt : tickets_below(carry + tot, nt, gg.u, gg.Q);
        int64_t t_lo, t_hi;
        if (run >= 0) {
            t_lo = c_lo + (int64_t)run * ITEM_TICKETS;
            t_hi = (t_lo + ITEM_TICKETS < c_hi) ? t_lo + ITEM_TICKETS : c_hi;
        } else {
            t_lo = c_lo > j0 ? c_lo : j0;
            t_hi = c_hi < j1 ? c_hi : j1;
        }
        if (t_lo < t_hi) {  // (at most ITEM_TICKETS: one run)
            const TicketScale sc{gg.tsv, gg.tsr, gg.tsl};
            const int L = (int)(t_hi - t_lo);
            clear_places(sm, 0, L);
            TicketRun rn{carry, t_lo, L, gg.off};
            if (t_lo != c_lo || t_hi != c_hi)
                rn = part_run(ts, carry, tg, sc, t_lo, L);
            else if (carry > 0)
                rn.off = run_offset(carry, tg, sc, t_lo, true);
            __syncthreads();
            block_parents(ts, rn, [&]() { return tg; }, sc, sm,
                          EmitRouted{kt, kept_anc, out, gg.tg0, (int32_t)c0, n, N, G, bl, Tg, &sum->flags});
        }
        carry += tot;
        __syncthreads();
    }
}

// Blocks [0, n_workers) take the split list's entries in turn; block
// n_workers + g takes a small group g whole, or its first ITEM_TICKETS
// tickets when it is heavy (a large group is all in the split list).
// s: scale_bits(N).
__global__ void __launch_bounds__(TILE_THREADS, 3) group_fill_kernel(
    const float *__restrict__ lw, int64_t N, int32_t G, const int64_t *__restrict__ Tg,
    const uint64_t *__restrict__ Ct, const GroupGrid *__restrict__ grid, const int4 *__restrict__ split,
    int32_t n_workers, const DevSummary *__restrict__ sum, double ess_thr, int32_t *__restrict__ out,
    int32_t *__restrict__ kept_anc, Balanced bl, int s, int sched, SchedArgs sa)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    int32_t block = blockIdx.x;
    if (sched) {  // the first block runs the schedule
        if (block == 0) {
            extern __shared__ uint64_t sched_mem[];  // sched_small_bytes(G)
            schedule_small(sa, reinterpret_cast<unsigned char *>(sched_mem));
            return;
        }
        --block;
    }
    __shared__ ParentSmem sm;
    if (block >= n_workers) {  // a group block: one item, no loop
        const GroupGrid gg = grid[block - n_workers];
        const double ess = sum->ess;
        const int32_t deg = sum->degenerate;
        const float M = sum->M;
        if (ess >= ess_thr || deg || gg.nt == 0 || gg.p1 - gg.p0 > GROUP_SPLIT)
            return;  // kept by the N_eff test, no usable weight, no offspring, or a large group
        const int64_t j1 = gg.nt > ITEM_TICKETS ? ITEM_TICKETS : gg.nt;  // a heavy group's first run
        group_fill_item(lw, N, G, Tg, gg, gg.p0, gg.p1, 0, j1, -1, 0, M, s, sum, out, kept_anc, bl, sm);
        return;
    }
    if (sum->ess >= ess_thr || sum->degenerate)
        return;
    const float M = sum->M;
    const int32_t n_items = sum->n_split + sum->n_runs;
    for (int32_t it = block; it < n_items; it += n_workers) {
        const int4 en = split[it];
        const GroupGrid gg = grid[en.y];
        if (en.x >= 0) {  // run en.z of a large group's part in tile en.x
            int64_t p0, p1;
            uint64_t carry;
            tile_part(gg, en.x, Ct, p0, p1, carry);
            group_fill_item(lw, N, G, Tg, gg, p0, p1, 0, 0, en.z, carry, M, s, sum, out, kept_anc, bl, sm);
        } else {  // run en.z of a heavy small group
            const int64_t j0 = (int64_t)en.z * ITEM_TICKETS;
            const int64_t j1 = (j0 + ITEM_TICKETS < (int64_t)gg.nt) ? j0 + ITEM_TICKETS : (int64_t)gg.nt;
            group_fill_item(lw, N, G, Tg, gg, gg.p0, gg.p1, j0, j1, -1, 0, M, s, sum, out, kept_anc, bl, sm);
        }
    }
}

// ------------------------------------------------------------ RPA schedule
// One block.  Senders / receivers from the offspring counts o_g = T_{g+1} -
// T_g and the balanced targets n_g; SGS and LGS sort both lists by amount,
// descending, ties by group index (a merge sort in shared memory).  GS/SGS
// links are the pieces of [0, D) cut at every sender and receiver prefix
// boundary (D = total surplus = total deficit); LGS pairs the i-th sender
// with the i-th receiver.  Output: new group offsets and the routing
// segments (ticket start, slot start, length) with their copy work items
// (GS and SGS: the links only, from schedule_links_balanced).
// block-wide exclusive scan of an int64 array in place (single block)
__device__ void block_scan_i64(int64_t *a, int n, uint64_t *red, int64_t *total_out)
{
    const int per = (n + blockDim.x - 1) / blockDim.x;
    const int i0 = threadIdx.x * per;
    uint64_t s = 0;
    for (int k = 0; k < per; ++k)
        if (i0 + k < n)
            s += (uint64_t)a[i0 + k];
    uint64_t total;
    uint64_t run = block_excl_scan_u64(s, red, &total);
    __syncthreads();
    for (int k = 0; k < per; ++k)
        if (i0 + k < n) {
            const int64_t v = a[i0 + k];
            a[i0 + k] = (int64_t)run;
            run += (uint64_t)v;
        }
    if (total_out)
        *total_out = (int64_t)total;
    __syncthreads();
}

// Sort (ascending) of n <= cap distinct u64 keys, one block of 1024 threads.
// sm: cap keys, then two index buffers of cap u16 (sort_smem_bytes(cap) in
// all, cap <= MAX_SCHED_GROUPS); g may be sm itself.  A merge sort on
// indices: every thread sorts a run of 16 in registers, then the merge
// levels, each thread writing 16 outputs after a merge-path search of its
// diagonal.  Launches size the buffer by their G, not by the largest G, so
// that the rest of the SM's 256 KB stays L1 cache for the kernel's global
// reads.
constexpr int SORT_PER = 16;
// every key needs a thread: the 1024 threads' runs cover the largest group count
static_assert(SORT_PER * 1024 >= MAX_SCHED_GROUPS, "block_sort_u64 covers at most SORT_PER x 1024 keys");
constexpr size_t SORT_SMEM_BYTES = (sizeof(uint64_t) + 2 * sizeof(uint16_t)) * MAX_SCHED_GROUPS;
__host__ __device__ inline size_t sort_smem_bytes(int cap)
{
    return (sizeof(uint64_t) + 2 * sizeof(uint16_t)) * (size_t)(cap > 0 ? cap : 1);
}

__device__ void block_sort_u64(uint64_t *g, int n, uint64_t *sm, int cap)
{
    uint16_t *ia = reinterpret_cast<uint16_t *>(sm + cap), *ib = ia + cap;
    if (g != sm)
        for (int i = threadIdx.x; i < n; i += blockDim.x)
            sm[i] = g[i];
    __syncthreads();
    const int t0 = threadIdx.x * SORT_PER;
    if (t0 < n) {
        uint64_t k[SORT_PER];
        uint16_t id[SORT_PER];
#pragma unroll
        for (int e = 0; e < SORT_PER; ++e) {
            k[e] = (t0 + e < n) ? sm[t0 + e] : ~0ull;  // past the end: sorts last
            id[e] = (uint16_t)(t0 + e);
        }
#pragma unroll
        for (int e = 1; e < SORT_PER; ++e)
#pragma unroll
            for (int f = e; f > 0; --f)
                if (k[f] < k[f - 1]) {
                    const uint64_t tk = k[f];
                    k[f] = k[f - 1];
                    k[f - 1] = tk;
                    const uint16_t ti = id[f];
                    id[f] = id[f - 1];
                    id[f - 1] = ti;
                }
#pragma unroll
        for (int e = 0; e < SORT_PER; ++e)
            if (t0 + e < n)
                ia[t0 + e] = id[e];
    }
    __syncthreads();
    uint16_t *src = ia, *dst = ib;
    for (int w = SORT_PER; w < n; w *= 2) {
        if (t0 < n) {
            const int base = (t0 / (2 * w)) * (2 * w);
            const int an = (n - base < w) ? n - base : w;
            const int b0 = base + w;
            const int bn = (n - b0 <= 0) ? 0 : ((n - b0 < w) ? n - b0 : w);
            const int d = t0 - base;
            int lo = d - bn > 0 ? d - bn : 0, hi = d < an ? d : an;
            while (lo < hi) {  // merge path: i taken from the first run, d - i from the second
                const int mid = (lo + hi) >> 1;
                if (sm[src[base + mid]] < sm[src[b0 + d - mid - 1]])
                    lo = mid + 1;
                else
                    hi = mid;
            }
            int i = lo, j = d - lo;
            const int cnt = (an + bn - d < SORT_PER) ? an + bn - d : SORT_PER;
            for (int e = 0; e < cnt; ++e) {
                const bool take_a = i < an && (j >= bn || sm[src[base + i]] < sm[src[b0 + j]]);
                dst[t0 + e] = take_a ? src[base + i] : src[b0 + j];
                i += take_a ? 1 : 0;
                j += take_a ? 0 : 1;
            }
        }
        __syncthreads();
        uint16_t *t = src;
        src = dst;
        dst = t;
    }
    uint64_t k[SORT_PER];
#pragma unroll
    for (int e = 0; e < SORT_PER; ++e)
        k[e] = (t0 + e < n) ? sm[src[t0 + e]] : 0ull;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < SORT_PER; ++e)
        if (t0 + e < n)
            g[t0 + e] = k[e];
    __syncthreads();
}

__device__ __forceinline__ int lower_bound_i32(const int32_t *a, int n, int32_t v)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (a[mid] < v)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// exclusive prefix of a[0..n) in place, a[n] = the total (one block; every
// thread takes one contiguous segment)
__device__ void block_scan_smem_i32(int32_t *a, int n, uint64_t *red)
{
    const int per = (n + blockDim.x - 1) / blockDim.x;
    const int i0 = threadIdx.x * per;
    uint64_t loc = 0;
    for (int k = 0; k < per; ++k)
        if (i0 + k < n)
            loc += (uint32_t)a[i0 + k];
    uint64_t total;
    uint64_t run = block_excl_scan_u64(loc, red, &total);
    for (int k = 0; k < per; ++k)
        if (i0 + k < n) {
            const int32_t v = a[i0 + k];
            a[i0 + k] = (int32_t)run;
            run += (uint32_t)v;
        }
    if (threadIdx.x == 0)
        a[n] = (int32_t)total;
    __syncthreads();
}

// Shared memory of schedule_kernel: the sort's buffer, and at least what
// schedule_links_balanced lays out (two u16 id lists, three int32 arrays).
__host__ __device__ inline size_t sched_smem_bytes(int G)
{
    const size_t need = 10 * (size_t)(G > 0 ? G : 1) + 64;
    const size_t sort = sort_smem_bytes(G);
    return sort > need ? sort : need;
}

// GS and SGS: every group ends at its balanced size, so the new offsets are
// the balanced ones and every sender keeps exactly n_g of its tickets (the
// fill already wrote those).  What remains are the links: the pieces of
// [0, D) cut at every sender and receiver prefix boundary, in the senders'
// and receivers' list order (group order for GS, sorted for SGS), and the
// copy work items of the links.  Everything but Tg stays in shared memory:
// the list order's group ids (u16), the prefix sums of the amounts (int32,
// with the total D as a sentinel), and the merge of the two prefix lists.
__device__ void schedule_links_balanced(const SchedArgs &A, int nS, int nR, bool sorted, uint64_t *sm,
                                        uint64_t *red)
{
    const int32_t G = A.G;
    const Balanced &bl = A.bl;
    DevSummary *sum = A.sum;
    const uint64_t *Skey = A.key, *Rkey = A.key + G;
    uint16_t *gS = reinterpret_cast<uint16_t *>(sm);
    uint16_t *gR = gS + nS;
    int32_t *PS = reinterpret_cast<int32_t *>(sm) + ((nS + nR + 1) / 2 + 1);  // after the ids, 4-byte aligned
    int32_t *PR = PS + nS + 1;
    int32_t *MG = PR + nR + 1;
    auto amount = [&](uint64_t k) -> int32_t {
        return sorted ? (int32_t)(0xFFFFFFFFFFull - (k >> 24)) : (int32_t)(k >> 24);
    };
    // 1. ids and amounts in list order; the balanced offsets and extent
    for (int i = threadIdx.x; i < nS; i += blockDim.x) {
        const uint64_t k = Skey[i];
        gS[i] = (uint16_t)(k & 0xFFFFFFull);
        PS[i] = amount(k);
    }
    for (int j = threadIdx.x; j < nR; j += blockDim.x) {
        const uint64_t k = Rkey[j];
        gR[j] = (uint16_t)(k & 0xFFFFFFull);
        PR[j] = amount(k);
    }
    for (int g = threadIdx.x; g <= G; g += blockDim.x)
        A.goff_new[g] = balanced_offset(bl, g);
    if (threadIdx.x == 0) {
        sum->max_group = bl.q + (bl.r > 0 ? 1 : 0);
        sum->min_group = bl.q;
    }
    __syncthreads();
    // 2. exclusive prefix sums (PS[nS] = PR[nR] = D)
    block_scan_smem_i32(PS, nS, red);
    block_scan_smem_i32(PR, nR, red);
    // 3. the merge of the two start lists (senders first on ties)
    for (int i = threadIdx.x; i < nS; i += blockDim.x)
        MG[i + lower_bound_i32(PR, nR, PS[i])] = PS[i];
    for (int j = threadIdx.x; j < nR; j += blockDim.x)
        MG[j + upper_bound_i32(PS, nS, PR[j])] = PR[j];
    __syncthreads();
    // 4. one link per distinct start, in order; each thread takes one
    //    contiguous range of the merge and knows its links' places
    const int nm = nS + nR;
    const int per = (nm + blockDim.x - 1) / blockDim.x;
    const int i0 = threadIdx.x * per;
    uint64_t c = 0;
    for (int k = 0; k < per; ++k) {
        const int i = i0 + k;
        if (i < nm && (i == 0 || MG[i] != MG[i - 1]))
            ++c;
    }
    uint64_t L;
    const uint64_t pos0 = block_excl_scan_u64(c, red, &L);
    uint64_t pos = pos0, chunks = 0;
    for (int k = 0; k < per; ++k) {
        const int i = i0 + k;
        if (i < nm && (i == 0 || MG[i] != MG[i - 1])) {
            const int32_t a = MG[i];
            const int si = upper_bound_i32(PS, nS, a) - 1;  // the sender piece holding a
            const int rj = upper_bound_i32(PR, nR, a) - 1;
            const int32_t e = PS[si + 1] < PR[rj + 1] ? PS[si + 1] : PR[rj + 1];
            const int32_t gs = gS[si], gr = gR[rj];
            const int64_t ts = A.Tg[gs], tr0 = A.Tg[gr], tr1 = A.Tg[gr + 1];
            // a sender keeps n_s; a receiver keeps its o_r and is filled after them
            A.seg_tick[G + pos] = ts + target_of(bl, gs) + (a - PS[si]);
            A.seg_dst[G + pos] = balanced_offset(bl, gr) + (tr1 - tr0) + (a - PR[rj]);
            A.seg_len[G + pos] = e - a;
            chunks += (uint64_t)((e - a + COPY_CHUNK - 1) / COPY_CHUNK);
            ++pos;
        }
    }
    // 5. copy work items: none for the kept segments [0, G), then the links
    uint64_t total_chunks;
    uint64_t run = block_excl_scan_u64(chunks, red, &total_chunks);
    for (int g = threadIdx.x; g < G; g += blockDim.x)
        A.seg_chunk[g] = 0;
    for (uint64_t p = pos0; p < pos; ++p) {
        A.seg_chunk[G + p] = (int32_t)run;
        run += (uint64_t)((A.seg_len[G + p] + COPY_CHUNK - 1) / COPY_CHUNK);
    }
    if (threadIdx.x == 0) {
        const int32_t nseg = G + (int32_t)L;
        A.seg_chunk[nseg] = (int32_t)total_chunks;
        A.seg_chunk[2 * G + 1] = nseg;  // the segment count
        sum->n_chunks = (int32_t)total_chunks;
        sum->links = (int64_t)L;
        sum->moved = PS[nS];
    }
}

__global__ void __launch_bounds__(1024) schedule_kernel(SchedArgs A)
{
    extern __shared__ uint64_t sm[];   // sched_smem_bytes(G)
    __shared__ uint64_t red[33];
    __shared__ int nS_s, nR_s;
    const int32_t G = A.G;
    DevSummary *sum = A.sum;
    if (sum->degenerate) {
        for (int g = threadIdx.x; g <= G; g += blockDim.x)
            A.goff_new[g] = A.goff[g];
        if (threadIdx.x == 0) {
            sum->n_chunks = 0;
            sum->links = 0;
            sum->moved = 0;
        }
        return;
    }
    uint64_t *Skey = A.key, *Rkey = A.key + G;
    // 1. senders / receivers, compacted in group order.  key = amount << 24 | g
    //    (amount <= N < 2^31 fits 40 bits; g < 2^24).  For sorting by amount
    //    descending then g ascending we sort ((2^40-1-amount) << 24 | g).
    if (threadIdx.x == 0) {
        nS_s = 0;
        nR_s = 0;
    }
    __syncthreads();
    // stable compaction via block scan of flags over contiguous per-thread ranges
    {
        const int per = (G + blockDim.x - 1) / blockDim.x;
        const int g0 = threadIdx.x * per;
        uint64_t cs = 0, cr = 0;
        for (int k = 0; k < per; ++k) {
            const int g = g0 + k;
            if (g < G) {
                const int64_t o = A.Tg[g + 1] - A.Tg[g], t = target_of(A.bl, g);
                cs += (o > t);
                cr += (o < t);
            }
        }
        uint64_t ts, tr;
        uint64_t ps = block_excl_scan_u64(cs, red, &ts);
        uint64_t pr = block_excl_scan_u64(cr, red, &tr);
        const bool sorted = (A.scheme != PPF_RPA_GS);
        for (int k = 0; k < per; ++k) {
            const int g = g0 + k;
            if (g < G) {
                const int64_t o = A.Tg[g + 1] - A.Tg[g], t = target_of(A.bl, g);
                if (o > t) {
                    const uint64_t amt = (uint64_t)(o - t);
                    Skey[ps++] = sorted ? (((0xFFFFFFFFFFull - amt) << 24) | (uint64_t)g) : ((amt << 24) | (uint64_t)g);
                }
                if (o < t) {
                    const uint64_t amt = (uint64_t)(t - o);
                    Rkey[pr++] = sorted ? (((0xFFFFFFFFFFull - amt) << 24) | (uint64_t)g) : ((amt << 24) | (uint64_t)g);
                }
            }
        }
        if (threadIdx.x == 0) {
            nS_s = (int)ts;
            nR_s = (int)tr;
        }
    }
    __syncthreads();
    const int nS = nS_s, nR = nR_s;
    const bool sorted = (A.scheme != PPF_RPA_GS);
    if (sorted) {
        block_sort_u64(Skey, nS, sm, G);
        block_sort_u64(Rkey, nR, sm, G);
    }
    if (A.scheme != PPF_RPA_LGS) {  // the fill wrote the kept tickets already
        schedule_links_balanced(A, nS, nR, sorted, sm, red);
        return;
    }
    auto amount = [&](uint64_t k) -> int64_t { return (int64_t)(0xFFFFFFFFFFull - (k >> 24)); };
    auto group = [&](uint64_t k) -> int32_t { return (int32_t)(k & 0xFFFFFFull); };
    // per-group sent / received totals
    int64_t *sent = A.val, *recv = A.val + G;
    for (int g = threadIdx.x; g < G; g += blockDim.x) {
        sent[g] = 0;
        recv[g] = 0;
    }
    __syncthreads();
    const int L = nS < nR ? nS : nR;
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        const int64_t a = amount(Skey[i]), b = amount(Rkey[i]);
        const int64_t c = a < b ? a : b;
        sent[group(Skey[i])] = c;
        recv[group(Rkey[i])] = c;
    }
    __syncthreads();
    // 2. new sizes and offsets: m'_g = o_g - sent_g + recv_g
    int64_t *off = A.goff_new;
    for (int g = threadIdx.x; g < G; g += blockDim.x)
        off[g] = (A.Tg[g + 1] - A.Tg[g]) - sent[g] + recv[g];
    __syncthreads();
    {
        int64_t mx = 0, mn = INT64_MAX;
        for (int g = threadIdx.x; g < G; g += blockDim.x) {
            mx = off[g] > mx ? off[g] : mx;
            mn = off[g] < mn ? off[g] : mn;
        }
        __shared__ long long smx[32], smn[32];
        for (int o = 16; o > 0; o >>= 1) {
            const long long a = __shfl_xor_sync(0xffffffffu, (long long)mx, o);
            const long long b = __shfl_xor_sync(0xffffffffu, (long long)mn, o);
            mx = a > mx ? a : mx;
            mn = b < mn ? b : mn;
        }
        if ((threadIdx.x & 31) == 0) {
            smx[threadIdx.x >> 5] = mx;
            smn[threadIdx.x >> 5] = mn;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            long long a = 0, b = INT64_MAX;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
                a = smx[w] > a ? smx[w] : a;
                b = smn[w] < b ? smn[w] : b;
            }
            sum->max_group = a;
            sum->min_group = b;
        }
        __syncthreads();
    }
    int64_t tot;
    block_scan_i64(off, G, red, &tot);
    if (threadIdx.x == 0)
        off[G] = tot;
    __syncthreads();
    // 3. kept segments: group g keeps its first o_g - sent_g tickets
    int64_t *seg_len = A.seg_len, *seg_tick = A.seg_tick, *seg_dst = A.seg_dst;
    for (int g = threadIdx.x; g < G; g += blockDim.x) {
        seg_tick[g] = A.Tg[g];
        seg_dst[g] = off[g];
        seg_len[g] = (A.Tg[g + 1] - A.Tg[g]) - sent[g];
    }
    // 4. links
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        const int32_t s = group(Skey[i]), r = group(Rkey[i]);
        const int64_t c = sent[s];
        const int64_t keep_s = (A.Tg[s + 1] - A.Tg[s]) - c;
        const int64_t keep_r = A.Tg[r + 1] - A.Tg[r];
        seg_tick[G + i] = A.Tg[s] + keep_s;
        seg_dst[G + i] = off[r] + keep_r;
        seg_len[G + i] = c;
    }
    __syncthreads();
    const int nseg = G + L;
    // 5. copy work items per segment
    {
        const int per = (nseg + blockDim.x - 1) / blockDim.x;
        const int i0 = threadIdx.x * per;
        uint64_t c = 0, mv = 0;
        for (int k = 0; k < per; ++k) {
            const int i = i0 + k;
            if (i < nseg) {
                c += (uint64_t)((seg_len[i] + COPY_CHUNK - 1) / COPY_CHUNK);
                if (i >= G)
                    mv += (uint64_t)seg_len[i];
            }
        }
        uint64_t tc, tmv;
        uint64_t run = block_excl_scan_u64(c, red, &tc);
        block_excl_scan_u64(mv, red, &tmv);
        for (int k = 0; k < per; ++k) {
            const int i = i0 + k;
            if (i < nseg) {
                A.seg_chunk[i] = (int32_t)run;
                run += (uint64_t)((seg_len[i] + COPY_CHUNK - 1) / COPY_CHUNK);
            }
        }
        if (threadIdx.x == 0) {
            A.seg_chunk[nseg] = (int32_t)tc;
            sum->n_chunks = (int32_t)tc;
            sum->links = L;
            sum->moved = (int64_t)tmv;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0)
        A.seg_chunk[2 * G + 1] = nseg;  // remember the segment count
}

// routing copy: anc[dst + k] = anc_sys[tick + k] for every segment, in work
// items of COPY_CHUNK slots; blocks loop over the items.  The first warp finds
// an item's segment (the last with seg_chunk <= b) by a 32-way search: each
// round probes 32 evenly spaced entries at once, so about three dependent
// loads locate it among tens of thousands of segments.
__global__ void __launch_bounds__(256) route_copy_kernel(const int32_t *__restrict__ anc_sys,
                                                         int32_t *__restrict__ anc, int32_t G,
                                                         const int32_t *__restrict__ seg_chunk,
                                                         const int64_t *__restrict__ seg_tick,
                                                         const int64_t *__restrict__ seg_dst,
                                                         const int64_t *__restrict__ seg_len, int64_t N,
                                                         DevSummary *__restrict__ sum)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    __shared__ int32_t sseg;
    const int32_t nb = sum->n_chunks;
    const int32_t nseg = seg_chunk[2 * G + 1];
    const int lane = threadIdx.x & 31;
    for (int32_t b = blockIdx.x; b < nb; b += gridDim.x) {
        if (threadIdx.x < 32) {
            int32_t lo = 0, hi = nseg;  // seg_chunk[lo] <= b < seg_chunk[hi] (hi may be nseg)
            while (hi - lo > 1) {
                const int32_t step = (hi - lo + 31) / 32;
                const int32_t p = lo + lane * step;
                const bool le = p < hi && __ldg(seg_chunk + p) <= b;
                const unsigned m = __ballot_sync(0xffffffffu, le);  // a prefix of the lanes
                const int32_t last = 31 - __clz(m);
                lo = lo + last * step;
                const int32_t nh = lo + step;
                hi = nh < hi ? nh : hi;
            }
            if (lane == 0)
                sseg = lo;
        }
        __syncthreads();
        const int32_t s = sseg;
        const int64_t k0 = (int64_t)(b - __ldg(seg_chunk + s)) * COPY_CHUNK;
        const int64_t len = __ldg(seg_len + s);
        const int64_t k1 = (k0 + COPY_CHUNK < len) ? k0 + COPY_CHUNK : len;
        const int64_t src = __ldg(seg_tick + s), dst = __ldg(seg_dst + s);
        if (src < 0 || dst < 0 || k0 < 0 || src + k1 > N || dst + k1 > N) {
            if (threadIdx.x == 0)
                atomicOr(&sum->flags, FLAG_INTERNAL);  // inconsistent schedule: never write out of bounds
        } else {
            // four loads in flight per thread before the stores
            for (int64_t k = k0 + threadIdx.x; k < k1; k += 4 * (int64_t)blockDim.x) {
                int32_t v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int64_t kk = k + q * (int64_t)blockDim.x;
                    v[q] = kk < k1 ? __ldg(anc_sys + src + kk) : 0;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int64_t kk = k + q * (int64_t)blockDim.x;
                    if (kk < k1)
                        anc[dst + kk] = v[q];
                }
            }
        }
        __syncthreads();  // sseg is rewritten for the next item
    }
}

// ------------------------------------------------------------------- RNA
// A group's offspring: ticket s2 goes to the group's own slot lo + s2, the last
// mig of them to the tail of the next group of the ring (at `tail`).
struct EmitRing {
    static constexpr bool DIRECT = false;
    int32_t *__restrict__ anc;
    float *__restrict__ lwp;
    float lwg;
    int32_t base;
    int n;
    int64_t lo, keep, tail, N;  // own slots [lo, lo + keep), then tail ..
    const int32_t *flags;
    __device__ __forceinline__ int lead(int64_t) const { return 0; }
    // m offspring to the slots from d on, their weight beside them
    __device__ __forceinline__ void piece(int64_t d, const uint16_t *st, int m) const
    {
        if (!PPF_DCHECK(d >= 0 && d + m <= N, flags, FLAG_INTERNAL))
            return;
        store_staged(anc + d, st, m, base, n, flags);
        float *o = lwp + d;
        const int head = (int)((4u - ((uint32_t)(reinterpret_cast<uintptr_t>(o) >> 2) & 3u)) & 3u);
        const int h = head < m ? head : m, m4 = (m - h) >> 2, t0 = h + 4 * m4, k = threadIdx.x;
        if (k < h)
            o[k] = lwg;
        for (int q = k; q < m4; q += blockDim.x)
            reinterpret_cast<float4 *>(o + h)[q] = make_float4(lwg, lwg, lwg, lwg);
        if (k < m - t0)
            o[t0 + k] = lwg;
    }
    __device__ __forceinline__ void staged(const uint16_t *st, int m, int64_t c) const
    {
        const int own = c < keep ? (keep - c < m ? (int)(keep - c) : m) : 0;
        if (own > 0)
            piece(lo + c, st, own);
        if (own < m)
            piece(tail + (c + own - keep), st + own, m - own);
    }
};

// The draw of a group larger than the block's 16 NT particles, in chunks of
// them; the tickets of a chunk are [T(carry), T(carry + total)), T the count
// below of the group's sz tickets.  (A call: its registers stay out of the
// kernel's common path.)  The weights are read three times, and 284 to 448 bytes
// a thread spill: a frame of RNA at 2,000,000 particles takes 72.7 us in groups
// of 4096, 87.5 in groups of 5000 and 98.4 in groups of 16384.
template <int NT>
static __device__ __noinline__ void rna_chunks(const float *__restrict__ lw, int64_t N, int64_t lo, int64_t sz, float Mg,
                                               int s, TicketGrid tg, TicketScale sc, ParentSmemT<NT> *sm, EmitRing em)
{
    constexpr int PART = NT * TILE_ITEMS;
    uint64_t carry = 0;
    for (int64_t c0 = 0; c0 < sz; c0 += PART) {
        const int n = (int)(sz - c0 < PART ? sz - c0 : PART);
        TileSums ts;
        tile_sums(lw, N, lo + c0, n, Mg, s, ts, *sm);
        const uint64_t tot = tile_total(*sm);
        const int64_t t_lo = tickets_below(carry, sz, tg.u, tg.Q);
        const int64_t t_hi = tickets_below(carry + tot, sz, tg.u, tg.Q);
        em.base = (int32_t)(lo + c0);
        em.n = n;
        draw_parents(ts, carry, tg, sc, t_lo, t_hi, true, run_offset(carry, tg, sc, t_lo, true), *sm, em,
                     [&](TileSums &t) { tile_sums(lw, N, lo + c0, n, Mg, s, t, *sm); });
        carry += tot;
        __syncthreads();
    }
}

// One block per group: group max, fixed-point weights, local total and group
// weight (FP64 against the global total of the step), local systematic
// tickets, then every offspring is written to its slot -- the last `mig`
// slots of the group go to the tail of the next group of the ring (group
// g + 1 mod G, or succ[g] for ARNA's ring).
//
// NT threads hold 16 NT particles: 64 for groups up to 1024, 128 up to 2048,
// else 256 (so that a small group does not leave most warps idle at the
// barriers).  Sums of e^(lw - Mg) are taken in one order for every NT: as if
// by 256 threads in strides of 256, lane sums by the warps' butterfly, the 8
// warps in turn.  Bound by the block's chain of barriers and its FP64
// logarithms (two per group: two lanes take one each): 20.6 us at 3.1M
// particles in groups of 4001 (31.5 before), 16.2 us at 2M (20.6).
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT - 1) rna_kernel(
    const float *__restrict__ lw, int64_t N, int32_t G, const int64_t *__restrict__ goff,
    const int32_t *__restrict__ succ, DevSummary *sum, double ess_thr, uint64_t seed, uint32_t fid, uint32_t frame,
    int32_t *__restrict__ anc, float *__restrict__ lwp, Divisor d_small, Divisor d_large)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    if (kept_by_ess(sum, ess_thr))
        return;
    const int64_t mig = sum->mig;
    constexpr int NW = NT / 32, VT = 256 / NT;  // virtual threads of the 256 per thread
    __shared__ ParentSmemT<NT> sm;
    __shared__ float smf[8];
    __shared__ float lwg_s;
    __shared__ uint64_t Qs, us, qNs;
    __shared__ uint32_t qRs;
    __shared__ Divisor dvs;
    __shared__ TicketScale scs;
    __shared__ int32_t offs;
    const int32_t g = blockIdx.x;
    const int64_t lo = goff[g], sz = goff[g + 1] - lo;
    if (sz <= 0)
        return;
    const int32_t gn = succ ? succ[g] : (g + 1) % G;
    const int64_t gn_lo = goff[gn], gn_sz = goff[gn + 1] - gn_lo;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const EmitRing em{anc, lwp, 0.0f, (int32_t)lo, (int)(sz < TILE ? sz : TILE), lo, sz - mig, gn_lo + gn_sz - mig, N,
                      &sum->flags};
    const bool one = sz <= NT * TILE_ITEMS;  // the whole group in the block's registers
    const int s = scale_bits(sz);
    float Mg = -INFINITY;
    auto group_max = [&](float m) {
        m = warp_max(m);
        if (lane == 0)
            smf[warp] = m;
        __syncthreads();
        for (int w = 0; w < NW; ++w)
            Mg = fmaxf(Mg, smf[w]);
        __syncthreads();  // every thread has read smf
    };
    TileSums ts;
    uint64_t q_all = 0;
    if (one) {
        // loaded in strides for the maximum and the sum of e^(lw - Mg), then
        // consecutively, from L1, for the quantised scan (whose total is the
        // group's Q)
        const int n = (int)sz;
        constexpr int PER = TILE_ITEMS / VT;
        float v[TILE_ITEMS];
        float m = -INFINITY;
#pragma unroll
        for (int j = 0; j < VT; ++j)
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int e = (int)threadIdx.x + j * NT + k * 256;
                v[j * PER + k] = (e < n) ? __ldg(lw + lo + e) : -INFINITY;
                m = fmaxf(m, v[j * PER + k]);
            }
        group_max(m);
#pragma unroll
        for (int j = 0; j < VT; ++j) {
            float es = 0.0f;
#pragma unroll
            for (int k = 0; k < PER; ++k)
                if (v[j * PER + k] > -INFINITY)
                    es += __expf(v[j * PER + k] - Mg);
            es = warp_sum(es);
            if (lane == 0)
                smf[warp + j * NW] = es;
        }
        tile_load16(lw, N, lo, n, v);
        tile_quantise(v, Mg, s, ts);
        clear_places(sm, 0, n);
        tile_scan(ts, sm);  // its barrier also publishes smf and the cleared places
        q_all = tile_total(sm);
    } else {
        float m = -INFINITY;
        for (int64_t i = threadIdx.x; i < sz; i += NT)
            m = fmaxf(m, __ldg(lw + lo + i));
        group_max(m);
        uint64_t qs = 0;
        for (int j = 0; j < VT; ++j) {
            float es = 0.0f;
            for (int64_t i = threadIdx.x + j * NT; i < sz; i += 512) {
                // two strided elements at a time
                const int64_t i2 = i + 256;
                const float v = __ldg(lw + lo + i);
                const float w = (i2 < sz) ? __ldg(lw + lo + i2) : -INFINITY;
                uint64_t a, b;
                quantise2(v, w, Mg, s, a, b);
                qs += a + b;
                if (v > -INFINITY)
                    es += __expf(v - Mg);
                if (w > -INFINITY)
                    es += __expf(w - Mg);
            }
            es = warp_sum(es);
            if (lane == 0)
                smf[warp + j * NW] = es;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            qs += __shfl_xor_sync(0xffffffffu, qs, o);
        if (lane == 0)
            sm.red[warp] = qs;
        __syncthreads();
        q_all = tile_total(sm);
    }
    // the group's draw: the FP64 weight by two lanes of warp 0 (one logarithm
    // each), the ticket grid by warp 1
    if (warp == 0) {
        float e = 0.0f;
        for (int w = 0; w < 8; ++w)
            e += smf[w];
        const double lg = log(lane == 1 ? (double)sz : (double)e);
        const double lsz = __shfl_sync(0xffffffffu, lg, 1);
        if (lane == 0)
            lwg_s = q_all == 0ull ? -INFINITY : (float)(((double)Mg + lg) - sum->log_total - lsz);
    }
    if (threadIdx.x == 32) {
        Qs = q_all;
        dvs = sz == (int64_t)d_small.d ? d_small : (sz == (int64_t)d_large.d ? d_large : make_divisor((uint32_t)sz));
        uint32_t r;
        qNs = div_by(q_all, dvs, &r);
        qRs = r;
        us = 0ull;
        if (q_all != 0ull) {
            us = ticket_offset(seed, fid, frame, PURPOSE_GROUP, (uint32_t)g, q_all);
            scs = ticket_scale(q_all, (uint32_t)sz);
            offs = run_offset(0, ticket_grid(q_all, us, qNs, qRs, dvs), scs, 0, true);
        }
    }
    __syncthreads();
    EmitRing ring = em;
    ring.lwg = lwg_s;
    if (q_all == 0ull) {  // no usable weight in the group: it keeps its slots
        for (int64_t s2 = threadIdx.x; s2 < sz; s2 += NT) {
            const int64_t d = s2 < em.keep ? lo + s2 : em.tail + (s2 - em.keep);
            if (!PPF_DCHECK(d >= 0 && d < N, &sum->flags, FLAG_INTERNAL))
                continue;
            anc[d] = (int32_t)(lo + s2);
            lwp[d] = ring.lwg;
        }
        return;
    }
    if (one) {
        const TicketRun run{0, 0, (int32_t)sz, offs};  // one ticket per particle: one run
        block_parents(ts, run, [&]() { return ticket_grid(Qs, us, qNs, qRs, dvs); }, scs, sm, ring);
    } else {
        rna_chunks<NT>(lw, N, lo, sz, Mg, s, ticket_grid(Qs, us, qNs, qRs, dvs), scs, &sm, ring);
    }
}

__global__ void __launch_bounds__(1024) rna_prep_kernel(const int64_t *__restrict__ goff, int32_t G, float alpha,
                                                        DevSummary *sum, double ess_thr)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    __shared__ long long smx[32], smn[32];
    long long mx = 0, mn = INT64_MAX;
    for (int g = threadIdx.x; g < G; g += blockDim.x) {
        const long long sz = goff[g + 1] - goff[g];
        mx = sz > mx ? sz : mx;
        mn = sz < mn ? sz : mn;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const long long a = __shfl_xor_sync(0xffffffffu, mx, o);
        const long long b = __shfl_xor_sync(0xffffffffu, mn, o);
        mx = a > mx ? a : mx;
        mn = b < mn ? b : mn;
    }
    if ((threadIdx.x & 31) == 0) {
        smx[threadIdx.x >> 5] = mx;
        smn[threadIdx.x >> 5] = mn;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long a = 0, b = INT64_MAX;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            a = smx[w] > a ? smx[w] : a;
            b = smn[w] < b ? smn[w] : b;
        }
        const bool kept = kept_by_ess(sum, ess_thr);  // N_eff test: no resampling, no exchange
        const int64_t mig = kept ? 0 : (int64_t)floor((double)alpha * (double)b);
        sum->mig = mig;
        sum->max_group = a;
        sum->min_group = b;
        sum->links = (G > 1 && mig > 0) ? G : 0;
        sum->moved = (G > 1) ? mig * G : 0;
        sum->degenerate = kept ? 1 : 0;
        if (kept)
            sum->flags |= FLAG_KEPT;
    }
}

// ------------------------------------------------------------------ ARNA
// One block, after the RPA tile passes have counted the tickets below every
// group start (Tg): the involved groups (proportional allocation gives them
// at least their own size), the adaptive number of migrants
// mig = floor(alpha (G - |I|) min_g n_g / G) (FP64, in that order), and the
// ring -- redrawn when the step's log-evidence is negative (the object
// counts as lost): the groups in increasing order of the first Philox word of
// (seed; g, frame, filter, RING), ties by index (the merge sort of
// word << 32 | g).  Then every group's successor on the ring.
// Dynamic shared memory: sort_smem_bytes(G) (G <= MAX_SCHED_GROUPS).
__global__ void __launch_bounds__(1024) arna_prep_kernel(const int64_t *__restrict__ goff, int32_t G, float alpha,
                                                         DevSummary *sum, double ess_thr,
                                                         const int64_t *__restrict__ Tg, int32_t *__restrict__ ring,
                                                         int32_t *__restrict__ succ, uint64_t seed, uint32_t fid,
                                                         uint32_t frame)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    extern __shared__ uint64_t sm[];
    __shared__ long long smx[32], smn[32];
    __shared__ int sinv[32];
    __shared__ bool s_lost;
    const bool kept = kept_by_ess(sum, ess_thr);  // N_eff test: no resampling, no exchange, ring kept
    const bool usable = !kept && sum->Q != 0ull;  // Tg holds the tickets only when some weight is usable
    long long mx = 0, mn = INT64_MAX;
    int inv = 0;
    for (int g = threadIdx.x; g < G; g += blockDim.x) {
        const long long sz = goff[g + 1] - goff[g];
        mx = sz > mx ? sz : mx;
        mn = sz < mn ? sz : mn;
        if (usable && Tg[g + 1] - Tg[g] >= sz)
            ++inv;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const long long a = __shfl_xor_sync(0xffffffffu, mx, o);
        const long long b = __shfl_xor_sync(0xffffffffu, mn, o);
        mx = a > mx ? a : mx;
        mn = b < mn ? b : mn;
        inv += __shfl_xor_sync(0xffffffffu, inv, o);
    }
    if ((threadIdx.x & 31) == 0) {
        smx[threadIdx.x >> 5] = mx;
        smn[threadIdx.x >> 5] = mn;
        sinv[threadIdx.x >> 5] = inv;
    }
    if (threadIdx.x == 0)
        s_lost = !kept && !(sum->log_evidence >= 0.0);
    __syncthreads();
    if (s_lost) {
        for (int g = threadIdx.x; g < G; g += blockDim.x) {
            const uint4 r = draw(seed, (uint32_t)g, frame, fid, PURPOSE_RING, 0);
            sm[g] = ((uint64_t)r.x << 32) | (uint32_t)g;
        }
        __syncthreads();
        block_sort_u64(sm, G, sm, G);
        for (int p = threadIdx.x; p < G; p += blockDim.x)
            ring[p] = (int32_t)(uint32_t)sm[p];
        __syncthreads();
    }
    for (int p = threadIdx.x; p < G; p += blockDim.x)
        succ[ring[p]] = ring[(p + 1) % G];
    if (threadIdx.x == 0) {
        long long a = 0, b = INT64_MAX;
        int in = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            a = smx[w] > a ? smx[w] : a;
            b = smn[w] < b ? smn[w] : b;
            in += sinv[w];
        }
        const int64_t mig =
            kept ? 0 : (int64_t)floor((double)alpha * (double)(G - in) * (double)b / (double)G);
        sum->mig = mig;
        sum->involved = in;
        sum->max_group = a;
        sum->min_group = b;
        sum->links = (G > 1 && mig > 0) ? G : 0;
        sum->moved = (G > 1) ? mig * G : 0;
        sum->degenerate = kept ? 1 : 0;
        if (kept)
            sum->flags |= FLAG_KEPT;
        if (s_lost)
            sum->flags |= FLAG_RING;
    }
}

// ancestors / starting log-weights the next step will use
__global__ void pending_kernel(int64_t N, int mode, const int32_t *__restrict__ anc, const float *__restrict__ lwp,
                               const float *__restrict__ lw_cur, const int32_t *__restrict__ degenerate,
                               int32_t *__restrict__ anc_out, float *__restrict__ lwp_out)
{
    const int m = (mode != MODE_CARRY && *degenerate) ? MODE_CARRY : mode;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        if (anc_out)
            anc_out[i] = (m == MODE_CARRY) ? (int32_t)i : anc[i];
        if (lwp_out)
            lwp_out[i] = (m == MODE_CARRY) ? lw_cur[i] : (m == MODE_UNIFORM ? 0.0f : lwp[i]);
    }
}

__global__ void identity_kernel(int32_t *__restrict__ a, int64_t N)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = (int32_t)i;
}

// New particles were set: identity ancestry (a non-null), no degenerate
// resample before them, and the binned path next if the context has it.
// One launch for what were an ancestor fill and two staged copies of four bytes
// from the host (4,000,000 particles set: 60 us, 51 with this).
__global__ void restart_kernel(int32_t *__restrict__ a, int64_t N, DevSummary *sum, int binned)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sum->degenerate = 0;
        if (binned)
            sum->bin_next = 1;
    }
    if (!a)
        return;
    const int64_t nv = N >> 2;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t i = (int32_t)(4 * v);
        reinterpret_cast<int4 *>(a)[v] = make_int4(i, i + 1, i + 2, i + 3);
    }
    if (blockIdx.x == 0 && threadIdx.x < (N & 3))
        a[4 * nv + threadIdx.x] = (int32_t)(4 * nv + threadIdx.x);
}

__global__ void fill_f32_kernel(float *__restrict__ a, int64_t N, float v)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = v;
}

// ---------------------------------------------------------------- launchers
// Opt the dynamic-shared-memory kernels of this file into their sizes (current
// device; called when a context is created).
cudaError_t resample_kernel_attributes()
{
    cudaError_t e = cudaSuccess;
    e = cudaFuncSetAttribute(fill_tiles_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sched_small_bytes(SCHED_SMALL));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(group_fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sched_small_bytes(SCHED_SMALL));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(schedule_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)SORT_SMEM_BYTES);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(arna_prep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)SORT_SMEM_BYTES);
    return e;
}

// The context's scan.  rpa: 0 systematic, 1 RPA, 2 ARNA.
static void launch_tile_tickets(ppf_ctx *c, double ess_thr, int rpa)
{
    const ScanArgs A{c->N, c->T, c->sc.Qt, c->sc.Ct, c->sc.Tt, c->sc.To, c->sum, ess_thr, c->m.seed, c->m.filter_id,
                     (uint32_t)c->last_frame, c->goff, c->G, rpa, c->sc.Cbl, c->sc.Tg, make_divisor((uint32_t)c->N),
                     reinterpret_cast<int2 *>(c->sc.extra)};
    c->launches += launch_scan(A, c->stream) - 1;
}

static SchedArgs sched_args(ppf_ctx *c, int scheme, bool two_stage)
{
    SchedArgs A;
    A.N = c->N;
    A.G = c->G;
    A.scheme = two_stage ? scheme - (PPF_RPA2_GS - PPF_RPA_GS) : scheme;  // the schedule
    A.goff = c->goff;
    A.goff_new = c->goff_new;
    A.Tg = c->sc.Tg;
    A.key = c->sc.skey;
    A.val = c->sc.sval;
    A.seg_chunk = c->sc.seg_chunk;
    A.seg_tick = c->sc.seg_tick;
    A.seg_dst = c->sc.seg_dst;
    A.seg_len = c->sc.seg_len;
    A.sum = c->sum;
    A.bl = balanced_layout(c->N, c->G);
    return A;
}

// The RPA schedule of more than SCHED_SMALL groups, or of LGS, on the context's
// side stream, after the tile scan (an event on the main stream), its
// completion recorded in ev_sched.
static cudaError_t launch_schedule(ppf_ctx *c, const SchedArgs &A)
{
    cudaError_t e = cudaEventRecord(c->ev_scan, c->stream);
    if (e == cudaSuccess)
        e = cudaStreamWaitEvent(c->side_stream, c->ev_scan, 0);
    if (e != cudaSuccess)
        return e;
    schedule_kernel<<<1, 1024, sched_smem_bytes(c->G), c->side_stream>>>(A);
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaEventRecord(c->ev_sched, c->side_stream);
    return e;
}

cudaError_t launch_resample_global(ppf_ctx *c, int scheme, double ess_thr)
{
    const bool rpa = (scheme != PPF_SYSTEMATIC);
    const float *lw = c->state[c->cur] + 5 * c->N;
    const int T = c->T;
    prof_mark(c, PH_RESAMPLE, 0);
    c->launches += rpa ? 4 : 3;
    if (rpa)
        launch_pdl(tile_group_totals_kernel, T, TILE_THREADS, 0, c->stream, lw, c->N, (const DevSummary *)c->sum,
                   ess_thr, c->sc.Qt, c->sc.St, (const int64_t *)c->goff, c->G, c->sc.Cbl, c->sc.tile_g);
    else  // five blocks per SM (48 registers), each tile's loads one tile ahead
        launch_pdl(tile_totals_kernel, T < 5 * c->num_sms ? T : 5 * c->num_sms, TILE_THREADS, 0, c->stream, lw, c->N,
                   (const DevSummary *)c->sum, ess_thr, c->sc.Qt, c->sc.St);
    launch_tile_tickets(c, ess_thr, rpa ? 1 : 0);
    int32_t *out = rpa ? c->anc_sys : c->anc;
    const bool two_stage = (scheme >= PPF_RPA2_GS && scheme <= PPF_RPA2_LGS);
    // GS and SGS: the kept tickets go straight to their balanced slots
    const bool kept_direct = rpa && scheme != PPF_RPA_LGS && scheme != PPF_RPA2_LGS;
    // The routing schedule needs only the tile scan (offspring counts per
    // group), not the fill, and runs beside it on one SM: as the fill's first
    // block where its lists are small, else on a side stream that the copy joins.
    const bool in_fill = kept_direct && c->G <= SCHED_SMALL;
    const SchedArgs sa = rpa ? sched_args(c, scheme, two_stage) : SchedArgs{};
    if (rpa && !in_fill) {
        cudaError_t e0 = launch_schedule(c, sa);
        if (e0 != cudaSuccess)
            return e0;
        c->launches += 1;
    }
    if (two_stage) {  // stage 2: every group draws its own offspring
        int4 *split = reinterpret_cast<int4 *>(c->sc.split);
        group_grid_kernel<<<(c->G + 255) / 256, 256, 0, c->stream>>>(
            c->N, c->G, c->goff, c->sc.Tg, c->sc.Ct, c->sc.Cbl, c->sum, ess_thr, c->m.seed, c->m.filter_id,
            (uint32_t)c->last_frame, c->sc.ggrid, split, balanced_layout(c->N, c->G));
        launch_pdl(split_runs_kernel, c->num_sms, 256, 0, c->stream, (const uint64_t *)c->sc.Ct,
                   (const GroupGrid *)c->sc.ggrid, split, c->sum, ess_thr);
        const int n_workers = 4 * c->num_sms;
        launch_pdl(group_fill_kernel, n_workers + c->G + (in_fill ? 1 : 0), TILE_THREADS,
                   in_fill ? sched_small_bytes(c->G) : 0, c->stream, lw, c->N, c->G,
                   (const int64_t *)c->sc.Tg, (const uint64_t *)c->sc.Ct, (const GroupGrid *)c->sc.ggrid,
                   (const int4 *)split, n_workers, (const DevSummary *)c->sum, ess_thr, out,
                   kept_direct ? c->anc : nullptr, balanced_layout(c->N, c->G), scale_bits(c->N), in_fill ? 1 : 0, sa);
        c->launches += 2;
    } else {
        const KeptRoute kr{kept_direct ? c->anc : nullptr, c->sc.Tg, c->sc.tile_g, c->G, balanced_layout(c->N, c->G)};
        const FillArgs A{lw, c->N, T, make_divisor((uint32_t)c->N), c->sum, c->sc.Ct, c->sc.Tt, c->sc.To, c->sc.St,
                         reinterpret_cast<const int2 *>(c->sc.extra), out, kr, in_fill ? 1 : 0, sa};
        launch_fill(A, c->stream);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !rpa) {
        prof_mark(c, PH_RESAMPLE, 1);
        return e;
    }
    if (!in_fill) {
        e = cudaStreamWaitEvent(c->stream, c->ev_sched, 0);  // join the schedule
        if (e != cudaSuccess)
            return e;
    }
    const int max_chunks = 2 * c->G + 1 + (int)((c->N + COPY_CHUNK - 1) / COPY_CHUNK);
    const int gcopy = max_chunks < 8 * c->num_sms ? max_chunks : 8 * c->num_sms;
    if (in_fill)
        launch_pdl(route_copy_kernel, gcopy, 256, 0, c->stream, (const int32_t *)c->anc_sys, c->anc, c->G,
                   (const int32_t *)c->sc.seg_chunk, (const int64_t *)c->sc.seg_tick, (const int64_t *)c->sc.seg_dst,
                   (const int64_t *)c->sc.seg_len, c->N, c->sum);
    else
        route_copy_kernel<<<gcopy, 256, 0, c->stream>>>(c->anc_sys, c->anc, c->G, c->sc.seg_chunk, c->sc.seg_tick,
                                                         c->sc.seg_dst, c->sc.seg_len, c->N, c->sum);
    prof_mark(c, PH_RESAMPLE, 1);
    return cudaGetLastError();
}

// RNA's per-group kernel, the block sized by the balanced groups (any layout
// is drawn right; groups beyond the block's particles go in chunks).
static void launch_rna(ppf_ctx *c, double ess_thr, const int32_t *succ)
{
    const float *lw = c->state[c->cur] + 5 * c->N;
    const Balanced bl = balanced_layout(c->N, c->G);
    const Divisor d0 = make_divisor((uint32_t)(bl.q > 0 ? bl.q : 1)), d1 = make_divisor((uint32_t)(bl.q + 1));
    const int64_t top = c->uneven ? TILE : bl.q + (bl.r > 0 ? 1 : 0);
    auto go = [&](auto kernel, int nt) {
        launch_pdl(kernel, c->G, nt, 0, c->stream, lw, c->N, c->G, (const int64_t *)c->goff, succ, c->sum, ess_thr,
                   c->m.seed, c->m.filter_id, (uint32_t)c->last_frame, c->anc, c->lwp, d0, d1);
    };
    if (top <= 64 * TILE_ITEMS)
        go(rna_kernel<64>, 64);
    else if (top <= 128 * TILE_ITEMS)
        go(rna_kernel<128>, 128);
    else
        go(rna_kernel<256>, 256);
}

cudaError_t launch_resample_rna(ppf_ctx *c, float alpha, double ess_thr)
{
    prof_mark(c, PH_RESAMPLE, 0);
    launch_pdl(rna_prep_kernel, 1, 1024, 0, c->stream, (const int64_t *)c->goff, c->G, alpha, c->sum, ess_thr);
    launch_rna(c, ess_thr, nullptr);
    prof_mark(c, PH_RESAMPLE, 1);
    c->launches += 2;
    return cudaGetLastError();
}

// ARNA: the RPA tile passes count each group's proportional offspring, one
// block settles the exchange and the ring, then RNA's per-group kernel.
cudaError_t launch_resample_arna(ppf_ctx *c, float alpha, double ess_thr)
{
    const float *lw = c->state[c->cur] + 5 * c->N;
    const int T = c->T;
    prof_mark(c, PH_RESAMPLE, 0);
    launch_pdl(tile_group_totals_kernel, T, TILE_THREADS, 0, c->stream, lw, c->N, (const DevSummary *)c->sum, ess_thr,
               c->sc.Qt, c->sc.St, (const int64_t *)c->goff, c->G, c->sc.Cbl, c->sc.tile_g);
    launch_tile_tickets(c, ess_thr, 2);
    launch_pdl(arna_prep_kernel, 1, 1024, sort_smem_bytes(c->G), c->stream, (const int64_t *)c->goff, c->G, alpha,
               c->sum, ess_thr, (const int64_t *)c->sc.Tg, c->ring, c->succ, c->m.seed, c->m.filter_id,
               (uint32_t)c->last_frame);
    launch_rna(c, ess_thr, c->succ);
    prof_mark(c, PH_RESAMPLE, 1);
    c->launches += 4;
    return cudaGetLastError();
}

cudaError_t launch_pending(ppf_ctx *c, int32_t *anc_out, float *lwp_out)
{
    const int grid = (int)((c->N + 255) / 256 < 8192 ? (c->N + 255) / 256 : 8192);
    c->launches += 1;
    pending_kernel<<<grid, 256, 0, c->stream>>>(c->N, c->mode, c->anc, c->lwp, c->state[c->cur] + 5 * c->N,
                                                &c->sum->degenerate, anc_out, lwp_out);
    return cudaGetLastError();
}

cudaError_t launch_identity(ppf_ctx *c, int32_t *dst)
{
    const int grid = (int)((c->N + 255) / 256 < 8192 ? (c->N + 255) / 256 : 8192);
    c->launches += 1;
    identity_kernel<<<grid, 256, 0, c->stream>>>(dst, c->N);
    return cudaGetLastError();
}

cudaError_t launch_restart(ppf_ctx *c, bool identity)
{
    const int64_t need = identity ? (c->N / 4 + 255) / 256 + 1 : 1;
    const int grid = (int)(need < 8 * (int64_t)c->num_sms ? need : 8 * (int64_t)c->num_sms);
    c->launches += 1;
    launch_pdl(restart_kernel, grid, 256, 0, c->stream, identity ? c->anc : nullptr, c->N, c->sum, c->bin_key ? 1 : 0);
    return cudaGetLastError();
}

// the ppf_estimate_t fields of the device summary, one 8-byte word per lane
// (for ppf_estimate_async; out is the caller's host buffer as the device sees
// it, so no copy follows)
__global__ void format_estimate_kernel(const DevSummary *__restrict__ sum, ppf_estimate_t *__restrict__ out)
{
    if (!pdl_wait())
        return;
    pdl_trigger();
    static_assert(sizeof(ppf_estimate_t) == 13 * 8 && offsetof(ppf_estimate_t, frame) == 64 &&
                      offsetof(ppf_estimate_t, status_flags) == 68 && offsetof(ppf_estimate_t, links) == 72,
                  "the estimate's words");
    const int w = threadIdx.x;
    unsigned long long v;
    if (w < 5)
        v = (unsigned long long)__double_as_longlong(sum->mean[w]);
    else if (w < 8)
        v = (unsigned long long)__double_as_longlong(w == 5 ? sum->log_evidence : w == 6 ? sum->ess : sum->max_lw);
    else if (w == 8)
        v = (unsigned long long)(uint32_t)sum->frame | ((unsigned long long)(uint32_t)sum->flags << 32);
    else
        v = (unsigned long long)(w == 9 ? sum->links : w == 10 ? sum->moved : w == 11 ? sum->max_group : sum->min_group);
    if (w < 13)
        reinterpret_cast<unsigned long long *>(out)[w] = v;
}

cudaError_t launch_format_estimate(ppf_ctx *c, ppf_estimate_t *out)
{
    launch_pdl(format_estimate_kernel, 1, 32, 0, c->stream, (const DevSummary *)c->sum, out);
    c->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_fill_f32(ppf_ctx *c, float *dst, float v)
{
    const int grid = (int)((c->N + 255) / 256 < 8192 ? (c->N + 255) / 256 : 8192);
    fill_f32_kernel<<<grid, 256, 0, c->stream>>>(dst, c->N, v);
    return cudaGetLastError();
}

}  // namespace ppf
