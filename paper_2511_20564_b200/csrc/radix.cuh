// Building blocks shared by the sampler and the graph ingest: single-pass prefix sums across thread
// blocks, and a stable least-significant-digit radix sort of (int32 key, value) pairs, one launch per digit.
#pragma once

#include "common.cuh"
#include "scan.cuh"

namespace e2egrec {

constexpr int kSortItems = 16;          // elements per thread of a tile
constexpr int kSortTile = 256 * kSortItems;        // the smaller of the two tile sizes: what scratch is sized for
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
// Stable LSD radix sort, one launch per digit.  A block takes a tile of consecutive elements, ranks the equal digits in
// element order (per warp by match_any, then across warps), publishes its digit counts and looks back over the tiles
// before it, digit by digit, until it meets one whose full prefix is known -- the chained scan above with one chain per
// digit.  The words of a chain tell their kind by themselves: 0 not there yet, count + 1 a tile's own count, top bit set
// the position behind the tile's last element of that digit in the output.  Tile 0 begins the chains with the digits' bins
// (digit counts of the whole array, known beforehand).  While the chains move, the tile is put into digit order in shared
// memory, so that the elements leave in runs: with 1024 digits a warp's 32 scattered 4-byte stores touched 32 sectors and
// the sectors, not the bytes, set the pace.
//
// The form before this one took three launches per digit (counts per tile, scan over the tiles, scatter straight from
// registers).  B200, 2 * 10^7 pairs, 1024 digits, a pass: 500 and 345 us (random and half-sorted digits), now 238 and 169;
// 2.9 * 10^5 entries of a sampled block: 24 us in three launches, now 16.  What bounds it now is the ranking's shared-memory
// and match latency at 32 warps per SM; L2 and DRAM are at a quarter of their rates.
// ---------------------------------------------------------------------------------------
constexpr unsigned kPosFlag = 0x80000000u;

// Rounds without progress after which a look-back of the sort ends.  Such a sort leaves positions of its output unwritten and
// flags E2EGREC_DEV_TIMEOUT.  Its later passes clamp the values they read, so that none is used as an index out of range,
// and who takes the result makes the offsets over it all zero, so that nothing behind them is reached.  (A tile that counts the
// elements before it itself instead keeps the result whole, but any code there cost the kernel 3 to 7 %.)
#ifndef E2EGREC_SORT_SPIN_LIMIT
#define E2EGREC_SORT_SPIN_LIMIT kChainSpinLimit
#endif

// A sort's last launch may also look up where its values belong: row_out[pos] = row_of[value].
struct SortMap { const int32_t *row_of; int32_t *row_out; };

template <int BITS, int THREADS>
constexpr size_t sort_smem_bytes()
{
    return (size_t)(THREADS / 32) * (1 << BITS) * 2 + (size_t)2 * (1 << BITS) * 4 + (size_t)2 * THREADS * kSortItems * 4;
}

template <int BITS, int THREADS, typename ValT>
__global__ void __launch_bounds__(THREADS, 2)
sort_pass_kernel(const int32_t *__restrict__ keys_in, const int32_t *__restrict__ vals_in, const int32_t *n_dev, int32_t n_host,
                 int32_t clamp_keys, int32_t clamp_vals, int shift, const unsigned *__restrict__ ghist, unsigned *ticket,
                 unsigned *state, int32_t *__restrict__ keys_out, ValT *__restrict__ vals_out, SortMap map, int32_t *status)
{
    constexpr int R = 1 << BITS;
    constexpr int W = THREADS / 32;
    constexpr int TILE = THREADS * kSortItems;
    constexpr int D = R >= THREADS ? R / THREADS : 1;            // consecutive digits per thread
    extern __shared__ uint4 sort_smem[];
    uint32_t *skey = reinterpret_cast<uint32_t *>(sort_smem);
    uint32_t *sval = skey + TILE;
    int32_t *start = reinterpret_cast<int32_t *>(sval + TILE);   // per digit: its first place in the tile's digit order
    int32_t *gbase = start + R;                                  // per digit: output position minus place in the tile
    uint16_t *wc = reinterpret_cast<uint16_t *>(gbase + R);      // [W][R] per warp: counts, then offsets within the digit
    __shared__ int32_t scan_sm[W + 1];
    __shared__ int tile_s;
    pdl_wait();
    const int32_t n = n_dev ? __ldcg(n_dev) : n_host;
    const int tile = chain_ticket(ticket, &tile_s);
    if ((int64_t)tile * TILE >= n) return;
    for (int d = threadIdx.x; d < W * R / 2; d += THREADS) reinterpret_cast<uint32_t *>(wc)[d] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tile_n = (int)min((int64_t)TILE, n - (int64_t)tile * TILE);
    const int w0 = warp * (32 * kSortItems);                     // the warp's first element of the tile
    const int32_t *kin = keys_in + (int64_t)tile * TILE;
    // every load of the tile is requested before the ranking, which then hides it
    const int32_t *vin = vals_in ? vals_in + (int64_t)tile * TILE : nullptr;
    uint32_t key[kSortItems], val[kSortItems];
    int rank[kSortItems];
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
        const int i = w0 + k * 32 + lane;
        key[k] = i < tile_n ? (uint32_t)__ldcg(kin + i) : 0u;
        if (clamp_keys && key[k] >= (uint32_t)clamp_keys) key[k] = 0;
    }
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
        const int i = w0 + k * 32 + lane;
        val[k] = !vin ? (uint32_t)(tile * TILE + i) : i < tile_n ? (uint32_t)__ldcg(vin + i) : 0u;
    }
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
        const bool ok = w0 + k * 32 + lane < tile_n;
        // (one ballot per bit instead: 240 and 231 us for the two passes over 2 * 10^7 pairs, against 238 and 169)
        const uint32_t digit = ok ? (key[k] >> shift) & (R - 1) : 0xFFFFFFFFu;
        const uint32_t peers = __match_any_sync(0xffffffffu, digit);
        const int leader = __ffs(peers) - 1;
        int base = 0;
        if (ok && lane == leader) {
            base = wc[warp * R + digit];
            wc[warp * R + digit] = (uint16_t)(base + __popc(peers));
        }
        base = __shfl_sync(0xffffffffu, base, leader);
        rank[k] = base + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
    }
    __syncthreads();
    // the thread's digits: counts of the warps -> offsets, the tile's count, its place in the tile's digit order
    const int d0 = threadIdx.x * D;
    const bool owner = d0 < R;
    int32_t cnt[D], sum = 0;
#pragma unroll
    for (int q = 0; q < D; ++q) {
        cnt[q] = 0;
        if (owner) {
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const int c = wc[w * R + d0 + q];
                wc[w * R + d0 + q] = (uint16_t)cnt[q];
                cnt[q] += c;
            }
            if (tile > 0) *reinterpret_cast<volatile unsigned *>(&state[(int64_t)tile * R + d0 + q]) = (unsigned)cnt[q] + 1u;
        }
        sum += cnt[q];
    }
    int32_t total;
    int32_t place = block_exclusive_scan<THREADS, int32_t>(sum, total, scan_sm);
    int32_t first[D];                                            // output position of the tile's first element of a digit
    if (tile == 0) {
        int32_t g = 0, gs[D];
#pragma unroll
        for (int q = 0; q < D; ++q) {
            gs[q] = g;
            g += owner ? (int32_t)__ldcg(ghist + d0 + q) : 0;
        }
        const int32_t bin = block_exclusive_scan<THREADS, int32_t>(g, total, scan_sm);
#pragma unroll
        for (int q = 0; q < D; ++q) first[q] = bin + gs[q];
    }
    if (owner) {
        int32_t pl = place;
#pragma unroll
        for (int q = 0; q < D; ++q) {
            start[d0 + q] = pl;
            pl += cnt[q];
        }
    }
    __syncthreads();
    // ---- the tile in digit order
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
        const int i = w0 + k * 32 + lane;
        if (i < tile_n) {
            const uint32_t digit = (key[k] >> shift) & (R - 1);
            const int pos = start[digit] + wc[warp * R + digit] + rank[k];
            skey[pos] = key[k];
            sval[pos] = clamp_vals && val[k] >= (uint32_t)clamp_vals ? 0u : val[k];     // not before: the value's load is still on its way
        }
    }
    // ---- the chains of the thread's digits, the nearest tiles first
    if (owner) {
        if (tile > 0) {
            int32_t before[D];
            unsigned open = (1u << D) - 1;
#pragma unroll
            for (int q = 0; q < D; ++q) before[q] = 0;
            constexpr int B = 8;                                 // tiles per round (16 and 32: no faster)
            int spin = 0;
            for (int p = tile - 1; open && p >= 0;) {
                unsigned v[B][D];
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const unsigned *src = state + (int64_t)max(p - b, 0) * R + d0;
                    if constexpr (D == 4) {
                        const uint4 x = __ldcv(reinterpret_cast<const uint4 *>(src));
                        v[b][0] = x.x; v[b][1] = x.y; v[b][2] = x.z; v[b][3] = x.w;
                    } else if constexpr (D == 2) {
                        const uint2 x = __ldcv(reinterpret_cast<const uint2 *>(src));
                        v[b][0] = x.x; v[b][1] = x.y;
                    } else {
                        v[b][0] = __ldcv(src);
                    }
                }
                int went = 0;                                    // tiles of the batch that are behind us
                bool ready = true;
#pragma unroll
                for (int b = 0; b < B; ++b) {
#pragma unroll
                    for (int q = 0; q < D; ++q) ready = ready && (v[b][q] != 0 || !((open >> q) & 1u));
                    if (ready && open) {
                        ++went;
#pragma unroll
                        for (int q = 0; q < D; ++q)
                            if ((open >> q) & 1u) {
                                if (v[b][q] & kPosFlag) {
                                    before[q] += (int32_t)(v[b][q] & ~kPosFlag);
                                    open &= ~(1u << q);
                                } else {
                                    before[q] += (int32_t)v[b][q] - 1;
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
#pragma unroll
            for (int q = 0; q < D; ++q) first[q] = before[q];
        }
#pragma unroll
        for (int q = 0; q < D; ++q)
            *reinterpret_cast<volatile unsigned *>(&state[(int64_t)tile * R + d0 + q]) = kPosFlag | (unsigned)(first[q] + cnt[q]);
        int32_t pl = place;
#pragma unroll
        for (int q = 0; q < D; ++q) {
            gbase[d0 + q] = first[q] - pl;
            pl += cnt[q];
        }
    }
    __syncthreads();
    constexpr int O = 8;                                         // elements per round: the look-ups of all are in flight
    for (int i0 = threadIdx.x; i0 < tile_n; i0 += O * THREADS) {
        uint32_t ky[O], v[O];
        int32_t pos[O], row[O];
#pragma unroll
        for (int q = 0; q < O; ++q) {
            const int i = i0 + q * THREADS;
            pos[q] = -1;
            row[q] = 0;
            if (i < tile_n) {
                ky[q] = skey[i];
                v[q] = sval[i];
                if (map.row_out) row[q] = __ldcg(map.row_of + v[q]);
                pos[q] = gbase[(ky[q] >> shift) & (R - 1)] + i;
            }
        }
#pragma unroll
        for (int q = 0; q < O; ++q) {
            if ((uint32_t)pos[q] >= (uint32_t)n) continue;       // beyond the tile, or after a wait that ran out (flagged)
            keys_out[pos[q]] = (int32_t)ky[q];
            vals_out[pos[q]] = (ValT)v[q];
            if (map.row_out) map.row_out[pos[q]] = row[q];
        }
    }
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

// Blocks of 512 threads where the array can fill the machine with their tiles (longer runs per digit on the way out),
// of 256 below.  The line: 2 * 148 tiles of 8192.
constexpr int64_t kSortWide = 2 * 148 * 512 * (int64_t)kSortItems;

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

template <int BITS, int THREADS, typename ValT>
static inline void launch_sort_pass(const int32_t *kin, const int32_t *vin, const int32_t *n_dev, int64_t cap, int32_t clamp_keys,
                                    int32_t clamp_vals, int pass, const SortState &ss, bool chain, int32_t *kout, ValT *vout, const SortMap &map,
                                    int32_t *status, cudaStream_t st)
{
    constexpr size_t smem = sort_smem_bytes<BITS, THREADS>();
    auto kern = sort_pass_kernel<BITS, THREADS, ValT>;
    if (smem > 48 * 1024) {
        static bool set[64] = {};                                // per device; the attribute may be set twice by two threads
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev < 0 || dev >= 64 || !set[dev]) {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (dev >= 0 && dev < 64) set[dev] = true;
        }
    }
    const unsigned grid = (unsigned)ceil_div(cap > 0 ? cap : 1, (int64_t)THREADS * kSortItems);
    note_launch();
    launch_pdl(chain, kern, dim3(grid), dim3(THREADS), smem, st, kin, vin, n_dev, (int32_t)cap, clamp_keys, clamp_vals, pass * BITS,
               ss.ghist + pass * kMaxRadix, ss.tickets() + pass, ss.state + (size_t)pass * ss.tiles * (1 << BITS), kout, vout, map, status);
}

template <typename ValT>
static inline void sort_pass(const SortPlan &sp, const int32_t *kin, const int32_t *vin, const int32_t *n_dev, int64_t cap,
                             int32_t clamp_keys, int32_t clamp_vals, int pass, const SortState &ss, bool chain, int32_t *kout, ValT *vout,
                             const SortMap &map, int32_t *status, cudaStream_t st)
{
    const bool wide = cap >= kSortWide;
    auto launch = sp.bits == 8 ? (wide ? launch_sort_pass<8, 512, ValT> : launch_sort_pass<8, 256, ValT>)
                               : (wide ? launch_sort_pass<10, 512, ValT> : launch_sort_pass<10, 256, ValT>);
    launch(kin, vin, n_dev, cap, clamp_keys, clamp_vals, pass, ss, chain, kout, vout, map, status, st);
}

}  // namespace e2egrec
