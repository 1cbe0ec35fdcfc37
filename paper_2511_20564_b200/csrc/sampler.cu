// k-hop neighbour sampling, frontier relabelling and block transposition.
//
// Everything here is integer work whose result is fixed by (graph, seeds, fanouts,
// seed, step): Philox4x32-10 draws keyed by the global node id, a bitmap + rank scan
// that yields the new frontier nodes in ascending id order, and a stable least-
// significant-digit radix sort that orders the transposed block by (source, position).
// All element counts stay on the device; grids are sized for the worst case and the
// surplus threads leave at once.
#include "common.cuh"
#include "scan.cuh"
#include "internal.cuh"
#include "radix.cuh"

#include <algorithm>

namespace e2egrec {

// ---------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplies with a
// Weyl key schedule.
// ---------------------------------------------------------------------------------------
__device__ inline uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

// ---------------------------------------------------------------------------------------
// Scratch layout (host and device agree through this struct).
// ---------------------------------------------------------------------------------------
constexpr int kDstTile = 128;          // most destinations per block of the sampling kernel
constexpr int kDstTileMin = 4;
constexpr int kDstThreads = 256;       // its threads: one per destination for the counts, then all of them draw
constexpr int kWordTile = 512;         // bitmap words per block of the frontier kernel (2048: 8 blocks on 500 k nodes)

// Destinations per block: about 1024 slots, four per thread, where that gives two blocks per SM and more; about 256 below,
// where the time is that of one block's chain of loads.  With 64 destinations whatever the fanout, 4096 seeds at fanout
// 100 were 64 blocks of 25 slots per thread.
//
// At most kDstBlocks blocks, three times what the machine holds, up to 64 destinations each: the host knows capacities, rows are
// shorter, and a block of eight destinations with ten entries each costs what one with a hundred each does (B200,
// 100 k seeds at fanout 128 on rows of 40 entries on average: 127 us with 12 500 blocks, 73 with 1563; on rows of 130 289 and 283).
constexpr int64_t kDstBlocks = 148 * 16;
static inline int dst_tile(int32_t cap_dst, int32_t fanout)
{
    const int64_t slots = (int64_t)cap_dst * fanout >= 2 * 148 * 1024 ? 1024 : 256;
    int t = kDstTileMin;
    while (t < kDstTile && 2ll * t * fanout <= slots) t *= 2;
    while (t < 64 && ceil_div(cap_dst, t) > kDstBlocks) t *= 2;
    return t;
}

// Everything one block transposition (radix sort by column + offsets) needs; one lane per hop, so that the
// transposition of hop h can run beside the sampling of hop h+1.
struct SortLane {
    int32_t  *edge_row;    // [max cap_edges]   destination of each block entry
    uint2    *pair;        // [max cap_edges]   the passes alternate between these and the block's arrays
    SortState sort;        // counts and tickets zeroed before relabel, which zeroes the live tiles' scan state
};

struct SamplerScratch {
    uint32_t *step_offset; // [1]         added to the `step` argument of every call (see e2egrec_sampler_set_step)
    int32_t  *local_id;    // [n_nodes]   -1 when idle, else position in the current frontier
    uint32_t *bitmap;      // [n_words]   newly reached nodes of the hop in progress; 0 when idle
    // everything from here to the chain states' used end is zeroed by the first kernel of a call
    char     *zero;
    unsigned *tickets;                 // [2 per hop, 1 for the seeds of a joint step]
    unsigned *ghist[kMaxHops];         // digit counts and tickets of the lanes' sorts
    unsigned long long *chain;         // per frontier (seeds of a joint step, hops): word tiles; then per hop: dst tiles
    int64_t   word_tiles;
    SortLane  lane[kMaxHops];
    size_t    bytes;
    int64_t   n_words;
};

static SamplerScratch carve(int64_t n_nodes, int64_t max_dst, int64_t max_src, int64_t max_edges, void *base)
{
    (void)max_src;
    SamplerScratch s;
    s.n_words = ceil_div(n_nodes, 32);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *p = base ? static_cast<char *>(base) + off : nullptr;
        off += align_up(bytes, 256);
        return p;
    };
    const int64_t sort_tiles = ceil_div(max_edges > 0 ? max_edges : 1, kSortTile);
    s.step_offset = (uint32_t *)take(256);
    s.local_id = (int32_t *)take(sizeof(int32_t) * (size_t)n_nodes);
    s.bitmap = (uint32_t *)take(sizeof(uint32_t) * (size_t)s.n_words);
    s.word_tiles = ceil_div(s.n_words > 0 ? s.n_words : 1, kWordTile);
    s.zero = base ? static_cast<char *>(base) + off : nullptr;
    s.tickets = (unsigned *)take(256);
    for (int h = 0; h < kMaxHops; ++h) s.ghist[h] = (unsigned *)take(sizeof(unsigned) * kSortCountWords);
    s.chain = (unsigned long long *)take(
        8 * (size_t)((kMaxHops + 1) * s.word_tiles + kMaxHops * (ceil_div(max_dst > 0 ? max_dst : 1, kDstTileMin) + 1)));
    for (int h = 0; h < kMaxHops; ++h) {
        SortLane &l = s.lane[h];
        l.edge_row = (int32_t *)take(sizeof(int32_t) * (size_t)(max_edges + 1));
        l.pair = (uint2 *)take(sizeof(uint2) * (size_t)(max_edges + 1));
        l.sort.ghist = s.ghist[h];
        l.sort.tiles = sort_tiles;
        l.sort.state = (unsigned *)take(sort_state_bytes(sort_tiles));
    }
    s.bytes = off;
    return s;
}

// ---------------------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------------------
__global__ void fill_i32_kernel(int32_t *p, int64_t n, int32_t v)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

struct HopCounts { int32_t *of[kMaxHops]; };

// First kernel of a call: clears the tickets, digit counts, chain states and status words of all hops (one launch instead of
// two memsets per hop; a tile of a hop that cleared its status word raced with what other tiles flagged) and, with seeds,
// makes them the first frontier: local id = position in the batch.  counts1 (joint step): a second set of counters to clear.
__global__ void __launch_bounds__(256)
sample_begin_kernel(uint4 *__restrict__ zero, int64_t zero16, const int32_t *__restrict__ seeds, int32_t n_seeds, int64_t n_nodes,
                    int32_t *__restrict__ local_id, HopCounts counts, int n_hops, int32_t *counts1)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, all = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = i; k < zero16; k += all) zero[k] = make_uint4(0, 0, 0, 0);
    if (i == 0) {
        counts.of[0][CNT_DST] = seeds ? n_seeds : 0;
#pragma unroll
        for (int h = 0; h < kMaxHops; ++h)
            if (h < n_hops) counts.of[h][CNT_STATUS] = 0;
        if (counts1) *reinterpret_cast<int4 *>(counts1) = make_int4(0, 0, 0, 0);
    }
    if (!seeds) return;
    for (int64_t k = i; k < n_seeds; k += all) {
        const int32_t u = seeds[k];
        if ((uint32_t)u < (uint64_t)n_nodes) local_id[u] = (int32_t)k;
    }
}

// One hop of sampling in one launch.  A block owns `tile_dst` destinations: |S(u)| = min(deg, fanout) per
// destination, a chained scan for the block's offset into the entry arrays, then one thread per
// (destination, slot).  Slot j of node u at hop h draws with the counter (j/2, u, (1<<8)|h, step) and
// key (seed lo, seed hi); words 2(j%2), 2(j%2)+1 form r and the picked row position is
// floor(r * deg / 2^64); with running sums of integer edge weights (g_cum) it is the first entry of the row
// whose running sum exceeds floor(r * total / 2^64).  deg <= fanout copies the row instead.  Sampled nodes
// that are not yet in the frontier are marked in the bitmap.
//
// Latency is what it costs: a dozen dependent loads per block.  The block's sum is published before the draws and the
// offset asked for after them, so that the chain moves meanwhile; four slots per thread keep their loads in flight together.
// Weighted draws: with up to kQuarterBlocks blocks a draw narrows its row to a quarter per step with the three probes of all
// four slots in flight (kDrawQuarters: 110 registers, two blocks per SM); with more, other blocks hide the latency and what
// counts are probes and registers: one slot after the other by halves, six blocks per SM (kDrawHalves).  B200, us for a
// sample whose table of running sums is not in L2, by quarters / by halves / by halves with four slots' loads behind a common
// look-back as before: seeds by activity (rows of up to a million entries), 64 x 100 33 / 41 / 207, 4096 x 100 57 / 66 / 229,
// 4096 x 15 x 10 68 / 88 / 125, 16 000 x 100 107 / 76 / 231; rows of 130 entries, 8192 x 20 x 10 x 5 416 / 315 / 401,
// 100 000 x 128 647 / 426 / 467.
constexpr int64_t kQuarterBlocks = 148 * 8;
enum { kDrawUniform, kDrawQuarters, kDrawHalves };
template <int kDraw>
__global__ void __launch_bounds__(kDstThreads, kDraw == kDrawUniform ? 5 : kDraw == kDrawHalves ? 6 : 2)
hop_sample_kernel(const int64_t *__restrict__ g_indptr, const int32_t *__restrict__ g_indices,
                  const uint64_t *__restrict__ g_cum, int64_t n_nodes,
                  const int32_t *__restrict__ dst_nodes, const int32_t *n_dst_ptr, int32_t cap_dst, int32_t cap_edges,
                  int32_t fanout, int32_t tile_dst, int32_t hop, uint32_t seed_lo, uint32_t seed_hi, uint32_t step_arg,
                  const uint32_t *__restrict__ step_offset, int32_t *__restrict__ counts,
                  int32_t *__restrict__ blk_indptr, float *__restrict__ inv_cnt, int32_t *__restrict__ src_nodes,
                  int32_t *__restrict__ nbr_global, int32_t *__restrict__ edge_row,
                  const int32_t *__restrict__ local_id, uint32_t *__restrict__ bitmap, unsigned *ticket,
                  unsigned long long *state)
{
    __shared__ int32_t off[kDstTile + 1];
    __shared__ int32_t node[kDstTile];
    __shared__ int64_t gbeg_s[kDstTile];
    __shared__ int64_t deg_s[kDstTile];
    __shared__ int32_t scan_sm[kDstThreads / 32 + 1];
    __shared__ long long bcast;
    __shared__ int tile_s;
    pdl_wait();
    int32_t n_dst = __ldcg(n_dst_ptr);               // on their way while the ticket is
    const uint32_t step = step_arg + __ldcg(step_offset);
    const int tile = chain_ticket(ticket, &tile_s);
    const bool over = n_dst > cap_dst;
    if (over) n_dst = cap_dst;
    if (tile == 0 && threadIdx.x == 0) {
        counts[CNT_DST] = n_dst;
        if (over) atomicOr((unsigned *)&counts[CNT_STATUS], E2EGREC_DEV_CAPACITY);
    }
    const int64_t i0 = (int64_t)tile * tile_dst;
    if (i0 >= n_dst) {
        if (n_dst == 0 && tile == 0 && threadIdx.x == 0) { blk_indptr[0] = 0; counts[CNT_EDGES] = 0; }
        return;
    }
    const int64_t i = i0 + threadIdx.x;
    int32_t c = 0;
    if (threadIdx.x < tile_dst && i < n_dst) {
        int32_t u = __ldcg(dst_nodes + i);
        int64_t gb = 0, deg = 0;
        if ((uint32_t)u < (uint64_t)n_nodes) {
            gb = g_indptr[u];
            deg = g_indptr[u + 1] - gb;
        } else {
            atomicOr((unsigned *)&counts[CNT_STATUS], E2EGREC_DEV_RANGE);
            u = 0;
        }
        c = deg < fanout ? (int32_t)deg : fanout;
        node[threadIdx.x] = u;
        gbeg_s[threadIdx.x] = gb;
        deg_s[threadIdx.x] = deg;
        inv_cnt[i] = c > 0 ? 1.0f / (float)c : 0.0f;
        src_nodes[i] = u;
    }
    int32_t tile_total;
    const int32_t ex = block_exclusive_scan<kDstThreads, int32_t>(c, tile_total, scan_sm);
    if (threadIdx.x < tile_dst) off[threadIdx.x] = ex;
    if (threadIdx.x == 0) {
        off[tile_dst] = tile_total;
        chain_publish(state, tile, tile_total);
    }
    __syncthreads();
    long long base = -1;
    constexpr int S = 4;
    for (int32_t sl0 = threadIdx.x; sl0 - (int32_t)threadIdx.x < tile_total || base < 0; sl0 += kDstThreads * S) {
        int rr[S];
        int64_t src[S], rbeg[S];
        uint64_t target[S];
        int64_t a[S], b[S];
        bool ok[S];
#pragma unroll
        for (int q = 0; q < S; ++q) {
            const int32_t sl = sl0 + q * kDstThreads;
            ok[q] = sl < tile_total;
            rr[q] = 0;
            src[q] = rbeg[q] = 0;
            a[q] = b[q] = 0;
            target[q] = 0;
            if (!ok[q]) continue;
            int lo = 0, hi = tile_dst;               // largest r with off[r] <= sl
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (off[mid] <= sl) lo = mid; else hi = mid;
            }
            rr[q] = lo;
            const int32_t j = sl - off[lo];
            const int64_t deg = deg_s[lo];
            int64_t pos = j;
            rbeg[q] = gbeg_s[lo];
            if (deg > fanout) {
                const uint4 r4 = philox4x32_10(make_uint4((uint32_t)(j >> 1), (uint32_t)node[lo], (1u << 8) | (uint32_t)hop, step),
                                               make_uint2(seed_lo, seed_hi));
                const uint64_t rnd = (j & 1) ? (((uint64_t)r4.w << 32) | r4.z) : (((uint64_t)r4.y << 32) | r4.x);
                const uint64_t total = kDraw != kDrawUniform ? g_cum[rbeg[q] + deg - 1] : 0;
                if (kDraw == kDrawQuarters && total > 0) {
                    target[q] = __umul64hi(rnd, total);
                    b[q] = deg - 1;                  // its running sum is `total`, above every target
                } else if (kDraw == kDrawHalves && total > 0) {
                    const uint64_t *cum = g_cum + rbeg[q];
                    const uint64_t t = __umul64hi(rnd, total);
                    int64_t hi_pos = deg - 1;        // its running sum is `total`, above every target
                    pos = 0;
                    while (pos < hi_pos) {
                        const int64_t mid = (pos + hi_pos) >> 1;
                        if (__ldg(cum + mid) > t) hi_pos = mid; else pos = mid + 1;
                    }
                } else {
                    pos = (int64_t)__umul64hi(rnd, (uint64_t)deg);
                }
            }
            src[q] = rbeg[q] + pos;
        }
        if constexpr (kDraw == kDrawQuarters) {
            // the first entry in [a, b] whose running sum exceeds the target
            while (true) {
                uint64_t c1[S], c2[S], c3[S];
                bool any = false;
#pragma unroll
                for (int q = 0; q < S; ++q) {
                    if (a[q] >= b[q]) continue;
                    any = true;
                    const uint64_t *cum = g_cum + rbeg[q] + a[q];
                    const int64_t w = b[q] - a[q];
                    c1[q] = __ldg(cum + w / 4);
                    c2[q] = __ldg(cum + w / 2);
                    c3[q] = __ldg(cum + w / 2 + (w - w / 2) / 2);
                }
                if (!any) break;
#pragma unroll
                for (int q = 0; q < S; ++q) {
                    if (a[q] >= b[q]) continue;
                    const int64_t w = b[q] - a[q], m1 = a[q] + w / 4, m2 = a[q] + w / 2, m3 = m2 + (w - w / 2) / 2;
                    if (c1[q] > target[q]) b[q] = m1;
                    else if (c2[q] > target[q]) { a[q] = m1 + 1; b[q] = m2; }
                    else if (c3[q] > target[q]) { a[q] = m2 + 1; b[q] = m3; }
                    else a[q] = m3 + 1;
                    if (a[q] >= b[q]) src[q] = rbeg[q] + b[q];
                }
            }
        }
        int32_t v[S];
#pragma unroll
        for (int q = 0; q < S; ++q) v[q] = ok[q] ? __ldg(&g_indices[src[q]]) : 0;
        int32_t lid[S];
#pragma unroll
        for (int q = 0; q < S; ++q) {
            if (ok[q] && (uint32_t)v[q] >= (uint64_t)n_nodes) {
                atomicOr((unsigned *)&counts[CNT_STATUS], E2EGREC_DEV_RANGE);
                v[q] = node[rr[q]];
            }
            lid[q] = ok[q] ? __ldcg(local_id + v[q]) : 0;
        }
        uint32_t word[S];
#pragma unroll
        for (int q = 0; q < S; ++q)   // hubs are sampled thousands of times per hop: look before the atomic
            word[q] = (ok[q] && lid[q] < 0) ? *reinterpret_cast<volatile uint32_t *>(&bitmap[v[q] >> 5]) : 0xFFFFFFFFu;
        if (base < 0) {                                  // the same for all threads: after the first round's loads
            base = chain_lookback(state, tile, tile_total, &counts[CNT_STATUS], &bcast);   // syncs the block
            if (threadIdx.x < tile_dst && i < n_dst) blk_indptr[i] = (int32_t)(base + ex);
            if (i0 + tile_dst >= n_dst && threadIdx.x == 0) {
                const long long total = base + tile_total;
                blk_indptr[n_dst] = (int32_t)total;
                counts[CNT_EDGES] = total > cap_edges ? cap_edges : (int32_t)total;
                if (total > cap_edges) atomicOr((unsigned *)&counts[CNT_STATUS], E2EGREC_DEV_CAPACITY);
            }
        }
#pragma unroll
        for (int q = 0; q < S; ++q) {
            const long long e = base + sl0 + q * kDstThreads;
            if (!ok[q] || e >= cap_edges) continue;
            nbr_global[e] = v[q];
            edge_row[e] = (int32_t)(i0 + rr[q]);
            if (lid[q] < 0 && !(word[q] & (1u << (v[q] & 31)))) atomicOr(&bitmap[v[q] >> 5], 1u << (v[q] & 31));
        }
    }
}

// New frontier nodes in one launch: a block owns kWordTile bitmap words, counts their set bits, takes
// its rank offset from a chained scan and hands out local ids n_dst, n_dst+1, ... in ascending id order.
// The bitmap returns to 0.
__global__ void __launch_bounds__(256)
frontier_kernel(uint32_t *__restrict__ bitmap, int64_t n_words, int32_t *__restrict__ counts, int32_t cap_src,
                int32_t *__restrict__ local_id, int32_t *__restrict__ src_nodes, unsigned *ticket,
                unsigned long long *state)
{
    constexpr int WPT = kWordTile / 256;
    __shared__ int32_t scan_sm[256 / 32 + 1];
    __shared__ long long bcast;
    __shared__ int tile_s;
    pdl_wait();
    const int tile = chain_ticket(ticket, &tile_s);
    const int64_t w0 = (int64_t)tile * kWordTile + (int64_t)threadIdx.x * WPT;
    uint32_t bits[WPT];
    int32_t c = 0;
#pragma unroll
    for (int k = 0; k < WPT; ++k) {
        bits[k] = w0 + k < n_words ? __ldcg(bitmap + w0 + k) : 0u;
        c += __popc(bits[k]);
    }
    int32_t tile_total;
    const int32_t ex = block_exclusive_scan<256, int32_t>(c, tile_total, scan_sm);
    if (threadIdx.x == 0) chain_publish(state, tile, tile_total);
    const long long base = chain_lookback(state, tile, tile_total, &counts[CNT_STATUS], &bcast);
    const int32_t n_dst = __ldcg(counts + CNT_DST);
    const bool last_tile = (int64_t)(tile + 1) * kWordTile >= n_words;
    if (last_tile && threadIdx.x == 0) {
        long long n_src = (long long)n_dst + base + tile_total;
        if (n_src > cap_src) { n_src = cap_src; atomicOr((unsigned *)&counts[CNT_STATUS], E2EGREC_DEV_CAPACITY); }
        counts[CNT_SRC] = (int32_t)n_src;
    }
    long long r = (long long)n_dst + base + ex;
#pragma unroll
    for (int k = 0; k < WPT; ++k) {
        uint32_t b = bits[k];
        if (!b) continue;
        bitmap[w0 + k] = 0;
        while (b) {
            const int bit = __ffs(b) - 1;
            b &= b - 1;
            const int32_t id = (int32_t)((w0 + k) * 32 + bit);
            if (r < cap_src) {
                local_id[id] = (int32_t)r;
                src_nodes[r] = id;
            }
            ++r;
        }
    }
}

// Scan state of the tiles that a sort of n keys will use, zeroed by the whole grid.
__device__ inline void zero_sort_state(const SortState &ss, int64_t n, int bits, int passes)
{
    const int64_t words = ((n + kSortTile - 1) / kSortTile) << bits;
    for (int p = 0; p < passes; ++p) {
        uint4 *dst = reinterpret_cast<uint4 *>(ss.state + ((size_t)p * ss.tiles << bits));
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words / 4; i += (int64_t)gridDim.x * blockDim.x)
            dst[i] = make_uint4(0, 0, 0, 0);
    }
}

// col[e] = position of the sampled node in the frontier, the digit counts of the whole col array for every pass of the
// radix sort that follows, and that sort's scan state.
__global__ void __launch_bounds__(256)
relabel_kernel(const int32_t *__restrict__ nbr_global, const int32_t *__restrict__ local_id,
               const int32_t *__restrict__ counts, int32_t *__restrict__ col, int bits, int passes, SortState ss)
{
    __shared__ unsigned h[kMaxPasses * kMaxRadix];
    pdl_wait();
    const int R = 1 << bits;
    for (int d = threadIdx.x; d < passes * R; d += 256) h[d] = 0;
    __syncthreads();
    const int32_t n = __ldcg(counts + CNT_EDGES);
    const int32_t n_src = __ldcg(counts + CNT_SRC);
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < n; e += (int64_t)gridDim.x * 256) {
        int32_t c = __ldcg(local_id + __ldcg(nbr_global + e));
        if (c < 0 || c >= n_src) c = 0;              // only after a capacity overrun, which is flagged
        col[e] = c;
        for (int p = 0; p < passes; ++p) atomicAdd(&h[p * R + ((c >> (p * bits)) & (R - 1))], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < passes * R; d += 256)
        if (h[d]) atomicAdd(&ss.ghist[(d / R) * kMaxRadix + (d % R)], h[d]);
    zero_sort_state(ss, n, bits, passes);
}

__global__ void frontier_release_kernel(const int32_t *__restrict__ src_nodes, const int32_t *__restrict__ counts,
                                        int32_t *__restrict__ local_id)
{
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < __ldcg(counts + CNT_SRC)) local_id[__ldcg(src_nodes + i)] = -1;
}

// csc_ptr[s] = first position whose column is >= s, from the steps of the sorted column array (a search per column cost 20
// scattered reads each).  Leaves the sort's tickets and scan state zero again, so that a block can be transposed any number
// of times.  After a wait of the sort that ran out all columns are left empty.
__global__ void csc_finalize_kernel(const int32_t *__restrict__ csc_col, const int32_t *__restrict__ counts,
                                    int32_t *__restrict__ csc_ptr, SortState ss, int bits, int passes,
                                    const int32_t *__restrict__ release_nodes, int32_t *__restrict__ local_id)
{
    pdl_wait();
    const int32_t n_all = __ldcg(counts + CNT_EDGES), n_src = __ldcg(counts + CNT_SRC);
    const uint32_t status = (uint32_t)__ldcg(counts + CNT_STATUS);
    if (release_nodes)                               // the last block of a sample also gives the local ids back
        for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_src; k += (int64_t)gridDim.x * blockDim.x)
            local_id[__ldcg(release_nodes + k)] = -1;
    zero_sort_state(ss, n_all, bits, passes);
    if (blockIdx.x == 0 && threadIdx.x < kMaxPasses) ss.tickets()[threadIdx.x] = 0;
    const int32_t n = (status & E2EGREC_DEV_TIMEOUT) ? 0 : n_all;
    const int lane = threadIdx.x & 31;
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; t0 <= n; t0 += (int64_t)gridDim.x * blockDim.x) {
        // position t is the first one whose column is >= s for the columns s in (col[t - 1], col[t]]
        const int32_t t = (int32_t)min(t0 + lane, (int64_t)n + 1);
        int32_t a = n_src, b = n_src;
        if (t <= n) {
            a = t > 0 ? __ldcg(csc_col + t - 1) : -1;
            b = t < n ? __ldcg(csc_col + t) : n_src;
        }
        const bool wide = b - a > 4;                 // columns without entries: the warp fills long stretches together
        if (!wide)
            for (int32_t s = a + 1; s <= b; ++s) csc_ptr[s] = t;
        for (unsigned m = __ballot_sync(0xffffffffu, wide); m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const int32_t wa = __shfl_sync(0xffffffffu, a, l), wb = __shfl_sync(0xffffffffu, b, l), wt = __shfl_sync(0xffffffffu, t, l);
            for (int32_t s = wa + 1 + lane; s <= wb; s += 32) csc_ptr[s] = wt;
        }
    }
}

// Joint step: the endpoints of the training pairs become the seed set.  Every endpoint is marked in the
// bitmap (frontier_kernel then lists the marked ids in ascending order and gives them local ids).
__global__ void pair_mark_kernel(const int32_t *__restrict__ user, const int32_t *__restrict__ item, int32_t n_pairs,
                                 int64_t n_nodes, uint32_t *__restrict__ bitmap, int32_t *__restrict__ counts)
{
    pdl_wait();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_pairs) return;
    const int32_t ids[2] = {user[p], item[p]};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if ((uint32_t)ids[k] < (uint64_t)n_nodes) atomicOr(&bitmap[ids[k] >> 5], 1u << (ids[k] & 31));
        else atomicOr((unsigned *)&counts[CNT_STATUS], E2EGREC_DEV_RANGE);
    }
}

// pair_local[e] = seed position of entry e (e < P: the user of pair e, else the item of pair e - P),
// entry_unit[e] = where that entry's gradient row starts inside the tower's input-gradient matrix, in
// 16-byte units, and the digit counts of pair_local for the sort that groups the entries by seed.
__global__ void __launch_bounds__(256)
pair_local_kernel(const int32_t *__restrict__ user, const int32_t *__restrict__ item, int32_t n_pairs, int64_t n_nodes,
                  const int32_t *__restrict__ local_id, int32_t *__restrict__ pair_local,
                  int32_t *__restrict__ entry_unit, int units_per_row, int item_unit_off, int32_t *__restrict__ pcounts,
                  int bits, int passes, SortState ss)
{
    __shared__ unsigned h[kMaxPasses * kMaxRadix];
    pdl_wait();
    const int R = 1 << bits;
    for (int d = threadIdx.x; d < passes * R; d += 256) h[d] = 0;
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) pcounts[CNT_EDGES] = 2 * n_pairs;
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < 2 * (int64_t)n_pairs; e += (int64_t)gridDim.x * 256) {
        const bool is_item = e >= n_pairs;
        const int32_t pr = (int32_t)(is_item ? e - n_pairs : e);
        const int32_t id = is_item ? item[pr] : user[pr];
        int32_t c = (uint32_t)id < (uint64_t)n_nodes ? __ldcg(local_id + id) : 0;
        if (c < 0) c = 0;
        pair_local[e] = c;
        entry_unit[e] = pr * units_per_row + (is_item ? item_unit_off : 0);
        for (int p = 0; p < passes; ++p) atomicAdd(&h[p * R + ((c >> (p * bits)) & (R - 1))], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < passes * R; d += 256)
        if (h[d]) atomicAdd(&ss.ghist[(d / R) * kMaxRadix + (d % R)], h[d]);
    zero_sort_state(ss, 2 * (int64_t)n_pairs, bits, passes);
}

// The transposed block: entries ordered by (column, position), the last pass looking up every entry's row, and the offsets.
static void transpose_block(const int32_t *col, int32_t *counts, int32_t cap_edges, const int32_t *row_of,
                            int32_t *csc_col, int32_t *csc_eid, int32_t *csc_row, int32_t *csc_ptr, const SortPlan &sp,
                            const SortLane &l, bool chain, cudaStream_t st, const int32_t *release_nodes = nullptr,
                            int32_t *local_id = nullptr)
{
    SortIn in{col, nullptr, nullptr, false, kRankSpread};
    for (int p = 0; p < sp.passes; ++p) {
        const bool last = p == sp.passes - 1, own = (sp.passes - 1 - p) % 2 == 0;       // the last pass ends in the block's arrays
        SortOut<int32_t> out{};
        if (own) {
            out.keys = csc_col;
            out.vals = csc_eid;
        } else {
            out.pairs = l.pair;
        }
        if (last) {
            out.row_of = row_of;
            out.row_out = csc_row;
        }
        sort_pass<int32_t>(sp, in, &counts[CNT_EDGES], cap_edges, 0, cap_edges, p, l.sort, chain, out, &counts[CNT_STATUS], st);
        in = own ? SortIn{csc_col, csc_eid, nullptr, false, kRankMatch} : SortIn{nullptr, nullptr, l.pair, false, kRankMatch};
    }
    note_launch();
    launch_pdl(chain, csc_finalize_kernel, dim3((unsigned)std::min<int64_t>(ceil_div((int64_t)cap_edges + 1, 256), 148 * 8)), dim3(256),
               0, st, csc_col, counts, csc_ptr, l.sort, sp.bits, sp.passes, release_nodes, local_id);
}

static inline unsigned grid_for(int64_t n, int threads) { return (unsigned)ceil_div(n > 0 ? n : 1, threads); }

size_t sampler_scratch_bytes(int64_t n_nodes, int64_t max_dst, int64_t max_src, int64_t max_edges)
{
    return carve(n_nodes, max_dst, max_src, max_edges, nullptr).bytes;
}

}  // namespace e2egrec

using namespace e2egrec;

// ---------------------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------------------
int32_t e2egrec::khop_caps(int64_t n_nodes, int32_t n_seeds, int32_t n_hops, const int32_t *fanouts,
                         int32_t *cap_dst, int32_t *cap_src, int32_t *cap_edges)
{
    if (!fanouts || !cap_dst || !cap_src || !cap_edges) return E2EGREC_ERR_NULL;
    if (n_nodes < 0 || n_seeds < 0) return E2EGREC_ERR_ARG;
    if (n_nodes >= (1ll << 31) || n_hops > kMaxHops) return E2EGREC_ERR_UNSUPPORTED;
    if (n_hops < 1) return E2EGREC_ERR_ARG;
    int64_t dst = n_seeds;
    for (int h = 0; h < n_hops; ++h) {
        if (fanouts[h] < 1) return E2EGREC_ERR_ARG;
        if (fanouts[h] > kMaxFanout) return E2EGREC_ERR_UNSUPPORTED;
        int64_t edges = dst * fanouts[h];
        int64_t src = dst + edges;
        if (src > n_nodes) src = n_nodes;
        if (src < dst) src = dst;
        if (edges >= (1ll << 31) - 1) return E2EGREC_ERR_UNSUPPORTED;
        cap_dst[h] = (int32_t)dst;
        cap_edges[h] = (int32_t)edges;
        cap_src[h] = (int32_t)src;
        dst = src;
    }
    return E2EGREC_OK;
}

extern "C" int32_t e2egrec_sample_khop_workspace(int64_t n_nodes, int32_t n_seeds, int32_t n_hops,
                                                 const int32_t *fanouts, int32_t *cap_dst, int32_t *cap_src,
                                                 int32_t *cap_edges, size_t *scratch_bytes)
{
    if (!scratch_bytes) return E2EGREC_ERR_NULL;
    int32_t rc = khop_caps(n_nodes, n_seeds, n_hops, fanouts, cap_dst, cap_src, cap_edges);
    if (rc != E2EGREC_OK) return rc;
    int64_t md = 0, ms = 0, me = 0;
    for (int h = 0; h < n_hops; ++h) {
        if (cap_dst[h] > md) md = cap_dst[h];
        if (cap_src[h] > ms) ms = cap_src[h];
        if (cap_edges[h] > me) me = cap_edges[h];
    }
    *scratch_bytes = carve(n_nodes, md, ms, me, nullptr).bytes;
    return E2EGREC_OK;
}

extern "C" int32_t e2egrec_sampler_scratch_init(int64_t n_nodes, void *scratch, size_t scratch_bytes, void *stream)
{
    if (!scratch) return E2EGREC_ERR_NULL;
    if (n_nodes < 0) return E2EGREC_ERR_ARG;
    if (n_nodes >= (1ll << 31)) return E2EGREC_ERR_UNSUPPORTED;
    if (reinterpret_cast<uintptr_t>(scratch) % 256) return E2EGREC_ERR_ALIGN;
    SamplerScratch s = carve(n_nodes, 0, 0, 0, scratch);
    if (scratch_bytes < s.bytes) return E2EGREC_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    note_launch();
    fill_i32_kernel<<<(unsigned)std::min<int64_t>(ceil_div(n_nodes > 0 ? n_nodes : 1, 256), 148 * 16), 256, 0, st>>>(
        s.local_id, n_nodes, -1);
    cudaMemsetAsync(s.step_offset, 0, 256, st);
    cudaMemsetAsync(s.bitmap, 0, sizeof(uint32_t) * (size_t)s.n_words, st);
    return check_launch("sampler_scratch_init");
}

__global__ void set_u32_kernel(uint32_t *p, uint32_t v) { *p = v; }

extern "C" int32_t e2egrec_sampler_set_step(void *scratch, uint32_t step_offset, void *stream)
{
    if (!scratch) return E2EGREC_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(scratch) % 256) return E2EGREC_ERR_ALIGN;
    SamplerScratch s = carve(0, 0, 0, 0, scratch);
    note_launch();
    set_u32_kernel<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(s.step_offset, step_offset);
    return check_launch("sampler_set_step");
}

// Running sums of the integer edge weights of every row, one warp per row at a time: 32 entries per round, a
// 64-bit warp scan, the carry kept in a register.
__global__ void __launch_bounds__(256)
edge_cumulate_kernel(int64_t n_nodes, const int64_t *__restrict__ indptr, const uint32_t *__restrict__ q,
                     uint64_t *__restrict__ cum)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n_nodes; u += warps) {
        const int64_t beg = indptr[u], end = indptr[u + 1];
        uint64_t carry = 0;
        for (int64_t e0 = beg; e0 < end; e0 += 32) {
            const int64_t e = e0 + lane;
            uint64_t v = e < end ? (uint64_t)q[e] : 0;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint64_t up = __shfl_up_sync(0xffffffffu, v, off);
                if (lane >= off) v += up;
            }
            if (e < end) cum[e] = carry + v;
            carry += __shfl_sync(0xffffffffu, v, 31);
        }
    }
}

extern "C" int32_t e2egrec_edge_cumulate(int64_t n_nodes, int64_t n_edges, const int64_t *indptr, const uint32_t *q,
                                         uint64_t *cum, void *stream)
{
    if (n_nodes < 0 || n_edges < 0) return E2EGREC_ERR_ARG;
    if (!indptr || (n_edges > 0 && (!q || !cum))) return E2EGREC_ERR_NULL;
    if (n_nodes == 0 || n_edges == 0) return E2EGREC_OK;
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(n_nodes * 32, 256), 148 * 16);
    note_launch();
    edge_cumulate_kernel<<<grid, 256, 0, static_cast<cudaStream_t>(stream)>>>(n_nodes, indptr, q, cum);
    return check_launch("edge_cumulate");
}

extern "C" int32_t e2egrec_sample_khop(const e2egrec_csr *graph, const int32_t *seeds, int32_t n_seeds,
                                       int32_t n_hops, const int32_t *fanouts, uint64_t seed, uint32_t step,
                                       uint32_t flags, const e2egrec_block *blocks,
                                       void *scratch, size_t scratch_bytes, void *stream)
{
    if (n_seeds > 0 && !seeds) return E2EGREC_ERR_NULL;
    return sample_khop_impl(graph, seeds, n_seeds, nullptr, n_hops, fanouts, seed, step, flags, blocks, scratch, scratch_bytes,
                            static_cast<cudaStream_t>(stream));
}

int32_t e2egrec::sample_khop_impl(const e2egrec_csr *graph, const int32_t *seeds, int32_t n_seeds, const PairInput *pairs,
                                  int32_t n_hops, const int32_t *fanouts, uint64_t seed, uint32_t step, uint32_t flags,
                                  const e2egrec_block *blocks, void *scratch, size_t scratch_bytes, cudaStream_t st)
{
    if (!graph || !fanouts || !blocks || !scratch || !graph->indptr) return E2EGREC_ERR_NULL;
    if (graph->n_edges > 0 && !graph->indices) return E2EGREC_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(scratch) % 256) return E2EGREC_ERR_ALIGN;
    int32_t cd[kMaxHops], cs[kMaxHops], ce[kMaxHops];
    int32_t rc = khop_caps(graph->n_nodes, n_seeds, n_hops, fanouts, cd, cs, ce);
    if (rc != E2EGREC_OK) return rc;
    int64_t md = 0, ms = 0, me = 0;
    for (int h = 0; h < n_hops; ++h) {
        const e2egrec_block &b = blocks[h];
        if (!b.counts || !b.indptr || !b.col || !b.nbr_global || !b.src_nodes || !b.csc_ptr || !b.csc_row ||
            !b.csc_eid || !b.csc_col || !b.inv_cnt)
            return E2EGREC_ERR_NULL;
        if (b.cap_dst < cd[h] || b.cap_src < cs[h] || b.cap_edges < ce[h]) return E2EGREC_ERR_WORKSPACE;
        if (b.cap_dst > md) md = b.cap_dst;
        if (b.cap_src > ms) ms = b.cap_src;
        if (b.cap_edges > me) me = b.cap_edges;
    }
    SamplerScratch s = carve(graph->n_nodes, md, ms, me, scratch);
    if (scratch_bytes < s.bytes) return E2EGREC_ERR_WORKSPACE;

    const int T = 256;
    const int64_t n = graph->n_nodes;
    // The transposition of a hop (sort + offsets) is only needed by the backward pass, so it runs on the
    // helper stream beside the sampling of the next hop; everything is joined before this call returns.
    SideStream *side = SideStream::get(st);
    if (side) side->join_pending();               // a transposition deferred by an earlier call still uses the lanes
    tap_begin(TAP_SAMPLE, st);
    const int32_t *dst_nodes = seeds;
    const int32_t *n_dst_ptr = &blocks[0].counts[CNT_DST];
    // chain states of this call: one run of word tiles per frontier, then the destination tiles of every hop
    unsigned long long *words[kMaxHops + 1], *tiles[kMaxHops], *chain = s.chain;
    for (int f = 0; f <= n_hops; ++f, chain += s.word_tiles) words[f] = chain;
    for (int h = 0; h < n_hops; ++h) {
        tiles[h] = chain;
        chain += ceil_div(blocks[h].cap_dst > 0 ? blocks[h].cap_dst : 1, dst_tile(blocks[h].cap_dst, fanouts[h]));
    }
    const int64_t zero16 = ceil_div(reinterpret_cast<char *>(chain) - s.zero, 16);
    HopCounts counts{};
    for (int h = 0; h < n_hops; ++h) counts.of[h] = blocks[h].counts;
    const int64_t begin_blocks = std::max<int64_t>(ceil_div(zero16, T * 2), grid_for(pairs ? 0 : n_seeds, T));
    note_launch();
    sample_begin_kernel<<<(unsigned)std::min<int64_t>(begin_blocks, 148 * 8), T, 0, st>>>(
        reinterpret_cast<uint4 *>(s.zero), zero16, pairs ? nullptr : seeds, n_seeds, n, s.local_id, counts, n_hops,
        pairs ? pairs->pcounts : nullptr);
    cudaStream_t ts = side ? side->stream : st;          // stream of the transpositions
    const bool chained = me < kChainEdges;
    if (pairs) {
        // seeds = ascending distinct endpoints of the pairs; entries (pair, side) grouped by seed.  Nobody reads the groups
        // before the backward pass: they are sorted on the helper stream, in a lane that no hop uses if there is one.
        const PairInput &pi = *pairs;
        const int32_t P2 = 2 * pi.n_pairs;
        note_launch();
        launch_pdl(chained, pair_mark_kernel, dim3(grid_for(pi.n_pairs, T)), dim3(T), 0, st, pi.user, pi.item, pi.n_pairs, n, s.bitmap,
                   blocks[0].counts);
        note_launch();
        launch_pdl(chained, frontier_kernel, dim3((unsigned)s.word_tiles), dim3(256), 0, st, s.bitmap, s.n_words, pi.pcounts, P2,
                   s.local_id, pi.seeds_out, s.tickets + 2 * kMaxHops, words[n_hops]);
        const SortPlan sp = sort_plan(P2 > 1 ? P2 : 2);
        const bool own_lane = n_hops < kMaxHops;
        const SortLane &l = s.lane[own_lane ? kMaxHops - 1 : 0];
        note_launch();
        launch_pdl(chained, pair_local_kernel, dim3((unsigned)std::min<int64_t>(grid_for(P2, T), 148 * 4)), dim3(T), 0, st, pi.user,
                   pi.item, pi.n_pairs, n, s.local_id, pi.pair_local, pi.entry_unit, pi.units_per_row, pi.item_unit_off, pi.pcounts,
                   sp.bits, sp.passes, l.sort);
        if (side && own_lane) side->fork(st);
        transpose_block(pi.pair_local, pi.pcounts, P2, pi.entry_unit, pi.pcsc_col, pi.pcsc_eid, pi.pcsc_idx, pi.pcsc_ptr, sp, l, chained,
                        own_lane ? ts : st);
        if (!own_lane) cudaMemsetAsync(l.sort.ghist, 0, sizeof(unsigned) * kSortCountWords, st);
        dst_nodes = pi.seeds_out;
        n_dst_ptr = &pi.pcounts[CNT_SRC];
    }
    const bool transpose = !(flags & E2EGREC_SAMPLE_NO_TRANSPOSE);
    const e2egrec_block &last = blocks[n_hops - 1];
    for (int h = 0; h < n_hops; ++h) {
        const e2egrec_block &b = blocks[h];
        const SortPlan sp = sort_plan(b.cap_src);
        const SortLane &l = s.lane[h];
        const int tile = dst_tile(b.cap_dst, fanouts[h]);
        const unsigned grid = grid_for(b.cap_dst, tile);
        auto sample = !graph->edge_cum ? hop_sample_kernel<kDrawUniform>
                      : grid <= kQuarterBlocks ? hop_sample_kernel<kDrawQuarters> : hop_sample_kernel<kDrawHalves>;
        note_launch();
        launch_pdl(chained, sample, dim3(grid), dim3(kDstThreads), 0, st, graph->indptr, graph->indices, graph->edge_cum, n, dst_nodes,
                   n_dst_ptr, b.cap_dst, b.cap_edges, fanouts[h], tile, h + 1, (uint32_t)(seed & 0xFFFFFFFFu), (uint32_t)(seed >> 32),
                   step, s.step_offset, b.counts, b.indptr, b.inv_cnt, b.src_nodes, b.nbr_global, l.edge_row, s.local_id, s.bitmap,
                   s.tickets + 2 * h, tiles[h]);
        note_launch();
        launch_pdl(chained, frontier_kernel, dim3((unsigned)s.word_tiles), dim3(256), 0, st, s.bitmap, s.n_words, b.counts, b.cap_src,
                   s.local_id, b.src_nodes, s.tickets + 2 * h + 1, words[h]);
        note_launch();
        launch_pdl(chained, relabel_kernel, dim3((unsigned)std::min<int64_t>(grid_for(b.cap_edges, T), 148 * 4)), dim3(T), 0, st,
                   b.nbr_global, s.local_id, b.counts, b.col, sp.bits, sp.passes, l.sort);
        if (transpose) {
            if (side) side->fork(st);
            const bool release = h == n_hops - 1;        // every relabelling is done: the last block's offsets release the ids
            transpose_block(b.col, b.counts, b.cap_edges, l.edge_row, b.csc_col, b.csc_eid, b.csc_row, b.csc_ptr, sp, l, chained, ts,
                            release ? last.src_nodes : nullptr, s.local_id);
        }
        dst_nodes = b.src_nodes;
        n_dst_ptr = &b.counts[CNT_SRC];
    }
    if (!transpose) {
        note_launch();
        launch_pdl(chained, frontier_release_kernel, dim3(grid_for(last.cap_src, T)), dim3(T), 0, st, last.src_nodes, last.counts,
                   s.local_id);
    }
    if (side && (transpose || (pairs && n_hops < kMaxHops))) {
        if (flags & E2EGREC_SAMPLE_DEFER_TRANSPOSE) side->defer();
        else side->join(st);
    }
    tap_end(TAP_SAMPLE, st);
    return check_launch("sample_khop");
}

// The transposed form of blocks sampled with E2EGREC_SAMPLE_NO_TRANSPOSE: the sort of every block by source and
// its offsets, from what the sampling left in the blocks and in the scratch (entry rows, digit counts of the
// columns).  Blocks are independent, so every other one runs on the helper stream.
extern "C" int32_t e2egrec_blocks_transpose(int64_t n_nodes, int32_t n_hops, const e2egrec_block *blocks, void *scratch,
                                            size_t scratch_bytes, void *stream)
{
    using namespace e2egrec;
    if (!blocks || !scratch) return E2EGREC_ERR_NULL;
    if (n_hops < 1 || n_hops > kMaxHops || n_nodes < 1) return E2EGREC_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(scratch) % 256) return E2EGREC_ERR_ALIGN;
    int64_t md = 0, ms = 0, me = 0;
    for (int h = 0; h < n_hops; ++h) {
        const e2egrec_block &b = blocks[h];
        if (!b.counts || !b.col || !b.csc_ptr || !b.csc_row || !b.csc_eid || !b.csc_col) return E2EGREC_ERR_NULL;
        if (b.cap_dst > md) md = b.cap_dst;
        if (b.cap_src > ms) ms = b.cap_src;
        if (b.cap_edges > me) me = b.cap_edges;
    }
    SamplerScratch s = carve(n_nodes, md, ms, me, scratch);
    if (scratch_bytes < s.bytes) return E2EGREC_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    SideStream *side = SideStream::get(st);
    if (side) side->join_pending();
    const bool forked = side && n_hops > 1;
    if (forked) side->fork(st);
    for (int h = n_hops - 1; h >= 0; --h) {          // the largest block first, on the caller's stream
        const e2egrec_block &b = blocks[h];
        const SortPlan sp = sort_plan(b.cap_src);
        const SortLane &l = s.lane[h];
        cudaStream_t ts = st;
        if (forked && ((n_hops - 1 - h) & 1)) ts = side->stream;
        transpose_block(b.col, b.counts, b.cap_edges, l.edge_row, b.csc_col, b.csc_eid, b.csc_row, b.csc_ptr, sp, l, me < kChainEdges,
                        ts);
    }
    if (forked) side->join(st);
    return check_launch("blocks_transpose");
}

