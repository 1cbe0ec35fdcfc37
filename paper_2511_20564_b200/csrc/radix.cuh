// Building blocks shared by the sampler and the graph ingest: single-pass prefix sums across thread
// blocks, and a stable least-significant-digit radix sort of (int32 key, value) pairs, one launch per digit.
#pragma once

#include <algorithm>

#include "common.cuh"
#include "scan.cuh"

namespace e2egrec {

constexpr int kSortThreads = 512;
constexpr int kSortItems = 16;          // elements per thread of a large tile
constexpr int kSortTile = kSortThreads * 8;      // the smaller of the two tile sizes: what scratch is sized for
constexpr int kMaxRadix = 1024;
constexpr int kMaxPasses = 4;
constexpr int kPassWords = 2048;        // words of scan state per tile for all passes of a sort: two of 1024 digits or more of 256

// ---------------------------------------------------------------------------------------
// Single-pass prefix sums across thread blocks ("chained scan"): every tile publishes its own sum,
// then looks back over the tiles before it until it meets one whose full prefix is known.  Tiles
// are handed out by an atomic ticket, so a tile only ever waits for tiles that already run.  Every
// wait is bounded; when the bound is hit the status word gets E2EGREC_DEV_TIMEOUT and the tile goes
// on with what it has.
// ---------------------------------------------------------------------------------------
constexpr unsigned long long kChainAgg = 1ull << 62, kChainPrefix = 2ull << 62, kChainMask = (1ull << 62) - 1;
constexpr int kChainSpinLimit = 1 << 22;

__device__ inline unsigned long long chain_read(const unsigned long long *slot)
{
    return *reinterpret_cast<const volatile unsigned long long *>(slot);
}

// One thread of the block publishes the tile's own sum as soon as it is known ...
__device__ inline void chain_publish(unsigned long long *state, int tile, long long aggregate)
{
    atomicExch(&state[tile], (tile == 0 ? kChainPrefix : kChainAgg) | (unsigned long long)aggregate);
}

// ... and later all threads of the block ask for the sum of the tiles before it.  A round of the first warp reads
// 4 x 32 tiles: where all tiles of a launch start together none has its prefix yet, and rounds are what the far ones pay.
__device__ inline long long chain_lookback(unsigned long long *state, int tile, long long aggregate, int32_t *status,
                                           long long *bcast)
{
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        long long excl = 0;
        if (tile > 0) {
            bool done = false;
            for (int p = tile - 1; !done; p -= 128) {
                unsigned long long v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int idx = p - 32 * j - lane;
                    v[j] = idx >= 0 ? chain_read(&state[idx]) : kChainPrefix;    // before tile 0: an empty prefix
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (done) break;
                    const int idx = p - 32 * j - lane;
                    bool timed_out = false;
                    for (int spin = 0; !__all_sync(0xffffffffu, (v[j] >> 62) != 0); ++spin) {
                        if (spin >= kChainSpinLimit) { timed_out = true; break; }
                        if (idx >= 0) v[j] = chain_read(&state[idx]);
                    }
                    const unsigned pref = __ballot_sync(0xffffffffu, (v[j] >> 62) == 2);
                    const int first = pref ? __ffs(pref) - 1 : 31;
                    long long c = lane <= first ? (long long)(v[j] & kChainMask) : 0;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
                    excl += c;
                    if (timed_out && lane == 0) atomicOr(reinterpret_cast<unsigned *>(status), E2EGREC_DEV_TIMEOUT);
                    done = timed_out || pref != 0;
                }
            }
            if (lane == 0) atomicExch(&state[tile], kChainPrefix | (unsigned long long)(excl + aggregate));
        }
        if (lane == 0) *bcast = excl;
    }
    __syncthreads();
    return *bcast;
}

__device__ inline int chain_ticket(unsigned *ticket, int *bcast)
{
    if (threadIdx.x == 0) *bcast = (int)atomicAdd(ticket, 1u);
    __syncthreads();
    return *bcast;
}


// ---------------------------------------------------------------------------------------
// Stable LSD radix sort, one launch per digit (the published method of single-pass scans with decoupled look-back, Merrill and
// Garland, applied to a pass's digits, Adinets and Merrill; the code is this file's own).  A block takes a tile of consecutive elements, ranks the equal digits in
// element order (per warp, see kRank..., then across warps), publishes its digit counts and looks back over the tiles
// before it, digit by digit, until it meets one whose full prefix is known -- the chained scan above with one chain per
// digit.  The words of a chain tell their kind by themselves: 0 not there yet, count + 1 a tile's own count, top bit set
// the position behind the tile's last element of that digit in the output.  Tile 0 begins the chains with the digits' bins
// (digit counts of the whole array, known beforehand).  While the chains move, the tile is put into digit order in shared
// memory, so that the elements leave in runs: with 1024 digits a warp's 32 scattered 4-byte stores touched 32 sectors and
// the sectors, not the bytes, set the pace.
//
// B200, 2 * 10^7 pairs, 1024 digits, us for the six passes of an ingest: 240 167 236 167 183 175 -> 140 146 160 150 153 155.
// What it spent them on: loads under a test each, which waited for one another (12 of 27 us a tile); matches of up to 32
// different digits (5 of 27); 170 warp instructions per 32 elements, most of them tests for the last, incomplete tile (now a copy
// of the code), shared-memory accesses per digit and warp (two digits a word now) and per array (pairs).  Tiles of 6144 and
// 4096 elements are slower (206 and 228 for the first pass where 16 per thread took 197), and so is one ballot per bit of the digit
// (196 188 196 184 190 193 with match's 205 142 199 140 160 146).  4096 elements by 512 threads of eight, where the array
// does not fill the machine: a transposition of 2.8 * 10^5 entries 39 -> 29 us, 256 threads of 16 by match 43.  What bounds it
// now is latency at 32 warps per SM (issue slots 50 %, L2 and DRAM at a quarter of their rates).
// ---------------------------------------------------------------------------------------
constexpr unsigned kPosFlag = 0x80000000u;

// Rounds without progress after which a look-back of the sort ends.  Such a sort leaves positions of its output unwritten and
// flags E2EGREC_DEV_TIMEOUT.  Its later passes clamp the values they read, so that none is used as an index out of range,
// and who takes the result makes the offsets over it all zero, so that nothing behind them is reached.  (A tile that counts the
// elements before it itself instead keeps the result whole, but any code there cost the kernel 3 to 7 %.)
#ifndef E2EGREC_SORT_SPIN_LIMIT
#define E2EGREC_SORT_SPIN_LIMIT kChainSpinLimit
#endif

// How the warp ranks equal digits.  kRankMatch: by match_any, whose time goes with the number of different digits in the
// warp.  kRankSpread, for passes whose neighbouring elements mostly differ in their digits: counts by shared-memory atomics, and
// a match only among the lanes whose digit was counted more than once.  kRankAny: elements of a digit may leave in any order, the
// atomics' result is the rank.  Counters are words of two halves: the atomics work on words, which cannot carry (a tile has fewer
// than 2^16 elements), everything else on halves, and between the two there is always a __syncwarp or a barrier.  B200, 2 * 10^7 pairs, 1024 digits, us a pass by match / spread / any: ids of random order 203 /
// 158 / 137, the second digits of such a sort (hubs in runs: lanes that count the same digit wait for one another) 145 / 172.
enum { kRankMatch, kRankSpread, kRankAny };

// What a pass reads and writes.  Between passes keys and values travel as pairs: half the memory instructions, and a run of
// eight elements of a digit fills two sectors where it touched four.
struct SortIn {
    const int32_t *keys, *vals;          // vals may be null: the element's number
    const uint2 *pairs;                  // if set, instead of the two: {key, value}, or with `swap` {value, key}
    bool swap;
    int rank;                            // kRank...
};
template <typename ValT> struct SortOut {
    int32_t *keys;
    ValT *vals;
    uint2 *pairs;                        // if set, instead of the two
    // a sort's last launch may also look up where its values belong: row_out[pos] = row_of[value]
    const int32_t *row_of;
    int32_t *row_out;
};

template <int BITS, int THREADS, int ITEMS>
constexpr size_t sort_smem_bytes()
{
    return (size_t)THREADS * ITEMS * 8 + (size_t)(1 << BITS) * 4 + (size_t)(THREADS / 32) * (1 << BITS) * 2;
}

// One tile of a pass.  FULL: every thread has all its elements.
template <int BITS, int THREADS, int ITEMS, bool FULL, typename ValT>
__device__ __forceinline__ void sort_tile(const SortIn &in, const int32_t n, const int tile, int32_t clamp_keys, int32_t clamp_vals,
                                          int shift, const unsigned *__restrict__ ghist, unsigned *state, const SortOut<ValT> &out,
                                          int32_t *status)
{
    constexpr int R = 1 << BITS;
    constexpr int W = THREADS / 32;
    constexpr int TILE = THREADS * ITEMS;
    constexpr int P = R / 2;                                     // a thread owns two neighbouring digits
    constexpr int K = 4;
    static_assert(P <= THREADS && TILE <= 32768 && ITEMS % K == 0 && K % 2 == 0, "digits fit the block, places 16 bits");
    extern __shared__ uint4 sort_smem[];
    uint2 *skv = reinterpret_cast<uint2 *>(sort_smem);           // the tile in digit order
    int32_t *gbase = reinterpret_cast<int32_t *>(skv + TILE);    // per digit: output position minus place in the tile
    uint32_t *wc = reinterpret_cast<uint32_t *>(gbase + R);      // [W][P] two digits a word: counts of a warp, then its first places
    __shared__ int32_t scan_sm[W + 1];
    for (int d = threadIdx.x; d < W * P / 4; d += THREADS) reinterpret_cast<uint4 *>(wc)[d] = make_uint4(0, 0, 0, 0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tile_n = (int)min((int64_t)TILE, n - (int64_t)tile * TILE);
    const int w0 = warp * (32 * ITEMS);                          // the warp's first element of the tile
    const int64_t i0 = (int64_t)tile * TILE + w0 + lane;
    const int own = tile_n - w0 - lane;                          // the thread's elements are the k with 32 k < own
    uint32_t key[ITEMS], val[ITEMS], rank[ITEMS / 2];            // rank: two a word
    // Every load of the tile is requested before the ranking, which then hides the values'.  Elements beyond the tile repeat
    // its last one: under a test each, the loads waited for one another.
    auto at = [&](int k) -> int64_t { return i0 + (FULL ? k * 32 : min(k * 32, own - 1)); };
    if (in.pairs) {
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const uint2 p = __ldcg(in.pairs + at(k));
            key[k] = p.x;
            val[k] = p.y;
        }
        if (in.swap) {
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                const uint32_t t = key[k];
                key[k] = val[k];
                val[k] = t;
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) key[k] = (uint32_t)__ldcg(in.keys + at(k));
        if (in.vals) {
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) val[k] = (uint32_t)__ldcg(in.vals + at(k));
        } else {
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) val[k] = (uint32_t)(i0 + k * 32);
        }
    }
    if (clamp_keys) {
#pragma unroll
        for (int k = 0; k < ITEMS; ++k)
            if (key[k] >= (uint32_t)clamp_keys) key[k] = 0;
    }
    __syncthreads();
    uint16_t *wcw = reinterpret_cast<uint16_t *>(wc + warp * P);
    const uint32_t below = (1u << lane) - 1u;
    if (in.rank == kRankAny) {
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const uint32_t digit = (key[k] >> shift) & (R - 1), half = (digit & 1) * 16;
            uint32_t r = 0;
            if (FULL || k * 32 < own) r = (atomicAdd(&wc[warp * P + (digit >> 1)], 1u << half) >> half) & 0xFFFFu;
            if (k & 1) rank[k / 2] |= r << 16;
            else rank[k / 2] = r;
        }
    } else if (in.rank == kRankSpread) {
#pragma unroll
        for (int k0 = 0; k0 < ITEMS; k0 += K) {
            uint32_t before[K], after[K];
            volatile const uint16_t *seen = wcw;
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const uint32_t digit = (key[k0 + j] >> shift) & (R - 1);
                before[j] = seen[digit];
                __syncwarp();
                if (FULL || (k0 + j) * 32 < own) atomicAdd(&wc[warp * P + (digit >> 1)], 1u << (16 * (digit & 1)));
                __syncwarp();
                after[j] = seen[digit];
                __syncwarp();
            }
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const bool shared_digit = (FULL || (k0 + j) * 32 < own) && after[j] - before[j] > 1;
                if (__any_sync(0xffffffffu, shared_digit)) {
                    const uint32_t peers = __match_any_sync(0xffffffffu, shared_digit ? (key[k0 + j] >> shift) & (R - 1) : 0xFFFFFFFFu);
                    if (shared_digit) before[j] += __popc(peers & below);
                }
                if (j & 1) rank[(k0 + j) / 2] |= before[j] << 16;
                else rank[(k0 + j) / 2] = before[j];
            }
        }
    } else {
#pragma unroll
        for (int k0 = 0; k0 < ITEMS; k0 += K) {
            uint32_t peers[K];
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const bool ok = FULL || (k0 + j) * 32 < own;
                const uint32_t digit = (key[k0 + j] >> shift) & (R - 1);
                peers[j] = __match_any_sync(0xffffffffu, ok ? digit : 0xFFFFFFFFu);
            }
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const bool ok = FULL || (k0 + j) * 32 < own;
                const uint32_t digit = (key[k0 + j] >> shift) & (R - 1);
                const uint32_t lower = __popc(peers[j] & below), base = wcw[digit];
                __syncwarp();
                if (ok && lower == 0) wcw[digit] = (uint16_t)(base + __popc(peers[j]));
                __syncwarp();
                const uint32_t r = base + lower;
                if (j & 1) rank[(k0 + j) / 2] |= r << 16;
                else rank[(k0 + j) / 2] = r;
            }
        }
    }
    __syncthreads();
    // the thread's digits: counts of the warps -> first places of the warps, in halves of a word
    const int d0 = threadIdx.x * 2;
    const bool owner = threadIdx.x < P;
    uint32_t sum2 = 0;
    if (owner) {
#pragma unroll
        for (int w = 0; w < W; ++w) sum2 += wc[w * P + threadIdx.x];
    }
    const int32_t cnt[2] = {(int32_t)(sum2 & 0xFFFFu), (int32_t)(sum2 >> 16)};
    if (owner && tile > 0)
        __stcg(reinterpret_cast<uint2 *>(state + (int64_t)tile * R + d0), make_uint2((unsigned)cnt[0] + 1u, (unsigned)cnt[1] + 1u));
    int32_t total;
    const int32_t place = block_exclusive_scan<THREADS, int32_t>(cnt[0] + cnt[1], total, scan_sm);
    int32_t first[2] = {0, 0};                                   // output position of the tile's first element of a digit
    if (tile == 0) {
        const uint2 g = owner ? __ldcg(reinterpret_cast<const uint2 *>(ghist + d0)) : make_uint2(0, 0);
        first[0] = block_exclusive_scan<THREADS, int32_t>((int32_t)(g.x + g.y), total, scan_sm);
        first[1] = first[0] + (int32_t)g.x;
    }
    if (owner) {
        uint32_t p2 = (uint32_t)place | (uint32_t)(place + cnt[0]) << 16;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const uint32_t c2 = wc[w * P + threadIdx.x];
            wc[w * P + threadIdx.x] = p2;
            p2 += c2;
        }
    }
    __syncthreads();
    // ---- the tile in digit order
    const uint16_t *first_place = wcw;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        if (clamp_vals && val[k] >= (uint32_t)clamp_vals) val[k] = 0;       // not before: the value's load is still on its way
        const uint32_t pos = first_place[(key[k] >> shift) & (R - 1)] + ((rank[k / 2] >> (16 * (k & 1))) & 0xFFFFu);
        if (FULL || k * 32 < own) skv[pos] = make_uint2(key[k], val[k]);
    }
    // ---- the chains of the thread's digits, the nearest tiles first
    if (owner) {
        if (tile > 0) {
            unsigned open = 3;
            constexpr int B = 8;                                 // tiles per round (16 and 32: no faster)
            int spin = 0;
            for (int p = tile - 1; open && p >= 0;) {
                uint2 v[B];
#pragma unroll
                for (int b = 0; b < B; ++b) v[b] = __ldcv(reinterpret_cast<const uint2 *>(state + (int64_t)max(p - b, 0) * R + d0));
                int went = 0;                                    // tiles of the batch that are behind us
                bool ready = true;
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const unsigned x[2] = {v[b].x, v[b].y};
                    ready = ready && (x[0] != 0 || !(open & 1u)) && (x[1] != 0 || !(open & 2u));
                    if (ready && open) {
                        ++went;
#pragma unroll
                        for (int q = 0; q < 2; ++q)
                            if ((open >> q) & 1u) {
                                if (x[q] & kPosFlag) {
                                    first[q] += (int32_t)(x[q] & ~kPosFlag);
                                    open &= ~(1u << q);
                                } else {
                                    first[q] += (int32_t)x[q] - 1;
                                }
                            }
                    }
                }
                p -= went;
                if (went) spin = 0;
                else if (++spin > E2EGREC_SORT_SPIN_LIMIT) {
                    if (status) atomicOr(reinterpret_cast<unsigned *>(status), E2EGREC_DEV_TIMEOUT);
                    break;
                }
            }
        }
        __stcg(reinterpret_cast<uint2 *>(state + (int64_t)tile * R + d0),
               make_uint2(kPosFlag | (unsigned)(first[0] + cnt[0]), kPosFlag | (unsigned)(first[1] + cnt[1])));
        *reinterpret_cast<int2 *>(gbase + d0) = make_int2(first[0] - place, first[1] - place - cnt[0]);
    }
    __syncthreads();
    constexpr int O = 8;                                         // elements per round: the look-ups of all are in flight
    static_assert(ITEMS % O == 0, "whole rounds");
#pragma unroll
    for (int r = 0; r < ITEMS / O; ++r) {
        const int p0 = threadIdx.x + r * O * THREADS;
        if (!FULL && p0 >= tile_n) break;
        uint2 kv[O];
        int32_t pos[O], row[O];
#pragma unroll
        for (int q = 0; q < O; ++q) kv[q] = skv[FULL ? p0 + q * THREADS : min(p0 + q * THREADS, tile_n - 1)];
        if (out.row_out) {
#pragma unroll
            for (int q = 0; q < O; ++q) row[q] = __ldcg(out.row_of + kv[q].y);
        }
#pragma unroll
        for (int q = 0; q < O; ++q) {
            pos[q] = gbase[(kv[q].x >> shift) & (R - 1)] + p0 + q * THREADS;
            // nowhere: beyond the tile, or after a wait that ran out (flagged)
            if ((!FULL && p0 + q * THREADS >= tile_n) || (uint32_t)pos[q] >= (uint32_t)n) pos[q] = -1;
        }
        if (out.pairs) {
#pragma unroll
            for (int q = 0; q < O; ++q)
                if (pos[q] >= 0) out.pairs[pos[q]] = kv[q];
        } else {
#pragma unroll
            for (int q = 0; q < O; ++q)
                if (pos[q] >= 0) {
                    out.keys[pos[q]] = (int32_t)kv[q].x;
                    out.vals[pos[q]] = (ValT)kv[q].y;
                }
        }
        if (out.row_out) {
#pragma unroll
            for (int q = 0; q < O; ++q)
                if (pos[q] >= 0) out.row_out[pos[q]] = row[q];
        }
    }
}

template <int BITS, int THREADS, int ITEMS, typename ValT>
__global__ void __launch_bounds__(THREADS, 2)
sort_pass_kernel(SortIn in, const int32_t *n_dev, int32_t n_host, int32_t clamp_keys, int32_t clamp_vals, int shift,
                 const unsigned *__restrict__ ghist, unsigned *ticket, unsigned *state, SortOut<ValT> out, int32_t *status)
{
    __shared__ int tile_s;
    pdl_wait();
    const int32_t n = n_dev ? __ldcg(n_dev) : n_host;
    const int tile = chain_ticket(ticket, &tile_s);
    const int64_t left = n - (int64_t)tile * THREADS * ITEMS;
    if (left >= THREADS * ITEMS)
        sort_tile<BITS, THREADS, ITEMS, true>(in, n, tile, clamp_keys, clamp_vals, shift, ghist, state, out, status);
    else if (left > 0)
        sort_tile<BITS, THREADS, ITEMS, false>(in, n, tile, clamp_keys, clamp_vals, shift, ghist, state, out, status);
}


struct SortPlan { int bits, passes; };

static inline SortPlan sort_plan(int32_t cap_src)
{
    int key_bits = 1;
    while (key_bits < 31 && (1ll << key_bits) < (int64_t)cap_src) ++key_bits;
    if (key_bits <= 8) return {8, 1};
    if (key_bits <= 10) return {10, 1};
    if (key_bits <= 16) return {8, 2};
    if (key_bits <= 20) return {10, 2};
    if (key_bits <= 24) return {8, 3};
    // (the scan state of a sort is kPassWords words per tile, which three digits of 10 bits would exceed; CSR and CSC of 2 * 10^7
    // entries over 2^25 nodes: 8.95 ms with three passes of 10 bits in three launches each, 5.09 with these)
    return {8, 4};
}

// 16 elements per thread where the array can fill the machine with such tiles (longer runs per digit on the way out),
// eight below.  The line: 2 * 148 tiles of 8192.
constexpr int64_t kSortWideTile = kSortThreads * (int64_t)kSortItems, kSortWide = 2 * 148 * kSortWideTile;

// One sort's scratch in device memory: digit counts of the whole array per pass, one ticket per pass and the scan state
// of every pass.  The counts and tickets must be zero before the kernel that fills the counts, the state of the live tiles
// before the first pass.
struct SortState {
    unsigned *ghist;                   // [kMaxPasses x kMaxRadix], then kMaxPasses tickets
    unsigned *state;                   // [passes][tiles][radix]
    int64_t tiles;                     // tiles of kSortTile elements that the state was sized for
    __host__ __device__ unsigned *tickets() const { return ghist + kMaxPasses * kMaxRadix; }
};
constexpr size_t kSortCountWords = kMaxPasses * kMaxRadix + 64;
constexpr size_t sort_state_bytes(int64_t tiles) { return sizeof(unsigned) * (size_t)kPassWords * (size_t)tiles; }

template <int BITS, int THREADS, int ITEMS, typename ValT>
static inline void launch_sort_pass(const SortIn &in, const int32_t *n_dev, int64_t cap, int32_t clamp_keys, int32_t clamp_vals, int pass,
                                    const SortState &ss, bool chain, const SortOut<ValT> &out, int32_t *status, cudaStream_t st)
{
    constexpr size_t smem = sort_smem_bytes<BITS, THREADS, ITEMS>();
    auto kern = sort_pass_kernel<BITS, THREADS, ITEMS, ValT>;
    if (smem > 48 * 1024) {
        static bool set[64] = {};                                // per device; the attribute may be set twice by two threads
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev < 0 || dev >= 64 || !set[dev]) {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (dev >= 0 && dev < 64) set[dev] = true;
        }
    }
    const unsigned grid = (unsigned)ceil_div(cap > 0 ? cap : 1, (int64_t)THREADS * ITEMS);
    note_launch();
    launch_pdl(chain, kern, dim3(grid), dim3(THREADS), smem, st, in, n_dev, (int32_t)cap, clamp_keys, clamp_vals, pass * BITS,
               ss.ghist + pass * kMaxRadix, ss.tickets() + pass, ss.state + (size_t)pass * ss.tiles * (1 << BITS), out, status);
}

template <typename ValT>
static inline void sort_pass(const SortPlan &sp, const SortIn &in, const int32_t *n_dev, int64_t cap, int32_t clamp_keys,
                             int32_t clamp_vals, int pass, const SortState &ss, bool chain, const SortOut<ValT> &out, int32_t *status,
                             cudaStream_t st)
{
    const bool wide = cap >= kSortWide;
    auto launch = sp.bits == 8 ? (wide ? launch_sort_pass<8, kSortThreads, kSortItems, ValT> : launch_sort_pass<8, kSortThreads, 8, ValT>)
                               : (wide ? launch_sort_pass<10, kSortThreads, kSortItems, ValT> : launch_sort_pass<10, kSortThreads, 8, ValT>);
    launch(in, n_dev, cap, clamp_keys, clamp_vals, pass, ss, chain, out, status, st);
}

}  // namespace e2egrec
