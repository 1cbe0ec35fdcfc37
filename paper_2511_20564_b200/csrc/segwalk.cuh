// Segment reduction over a CSR / CSC whose offsets are walked (no entry -> segment array), one warp per stretch:
//
//     out[s] = fin( sum_{k in [ptr[s], ptr[s+1])} w[idx[k]] * in[idx[k]] ),   fin = mean, seg_scale or nothing
//
// Whole-graph aggregation and LightGCN, and the forward propagation over a sampled block.  The windows, their records and
// the kernel that joins them are those of segreduce.cuh; a window is cut into one stretch of consecutive entries per
// warp of the block.
//
// What bounds it: instructions and the latency of the rows (sources that L2 serves: issue slots 57 % busy, 7.6 warps waiting for loads
// per issue) and, on power-law graphs, as much the barrier before the join (issue slots 50 %, 4.6 waiting for loads, 4.2 at the
// barrier; 2 * 10^7 entries of 128-byte rows, B200).
// A bf16 row is added without being widened first and its address is one product, and 32 entries of a long segment take no tests:
// 10^8 entries of 64 bf16 values and the transpose, weighted, 3.75 -> 3.19 ms (with stretches twice as long 3.16 at the time, but
// their longer sums doubled the rounding error).  With one lane group per run, 32 / LPR runs per warp each with its own
// segment ends, a 128-byte row took 22 warp instructions, most of them bookkeeping that the warp executes for all of its groups'
// different positions.  Here the offsets come 32 segments at a time, one lane each, and the segments are handled by their length:
//   - longer ones by the whole warp: 32 entry ids in one coalesced load (the next 32 and the entry weights on their way),
//     steps of 32 / LPR rows with no test per entry, and one sum across the lane groups per segment that halves the row at
//     every exchange, so that every lane stores its own share of the finished row;
//   - short ones (in a power-law graph nine tenths of the segments and a tenth of the entries) by one lane group each,
//     32 / LPR segments side by side, with no exchange; where a row takes the whole warp, as one stream of entries, so that
//     ids and weights come 32 at a time and four rows are in flight whatever the segments' lengths (one after another,
//     2 M segments of two entries on average took 719 and, weighted, 857 us with 256 bf16 values, 824 with 100 fp32 values;
//     now 578, 655 and 577).
// Together 5.6 warp instructions per row where segments are long and 10 on a power-law graph with weights.  Tried and slower:
// rows through a cp.async ring in shared memory (4.57 ms against 3.74 at the time: the copies and the reads of the ring load the L1
// path to 86 %), two groups of rows in registers (5.18), all segments by the whole warp (4.57), a row's registers loaded again as
// soon as it has been added (3.70 against 3.55), the ids of the next short segments loaded before the rows of these (3.48 against
// 3.28: registers spilled), stretches handed out by a counter (3.76 to 3.88: less waiting at the join's barrier, more stretches to
// begin and to join).
#pragma once

#include "segreduce.cuh"
#include "window.h"

namespace e2egrec {

// Segment of entry k by the whole warp: every round splits the range into 33 parts with 32 probes.
// Largest s in [0, n_seg) with ptr[s] <= k   (0 <= k < ptr[n_seg], ptr[0] = 0).
template <typename PtrT>
__device__ inline int64_t warp_seg_containing(const PtrT *__restrict__ ptr, int64_t n_seg, int64_t k)
{
    const int lane = threadIdx.x & 31;
    int64_t lo = 0, hi = n_seg;                    // ptr[lo] <= k < ptr[hi]
    while (hi - lo > 1) {
        const int64_t part = (hi - lo + 32) / 33;  // >= 1
        const int64_t probe = lo + (int64_t)(lane + 1) * part;
        const bool below = probe < hi && (int64_t)__ldg(&ptr[probe]) <= k;
        const int n = __popc(__ballot_sync(0xffffffffu, below));       // the offsets do not decrease: a prefix of the lanes
        const int64_t top = lo + (int64_t)(n + 1) * part;
        lo += (int64_t)n * part;
        if (top < hi) hi = top;
    }
    return lo;
}

// One exchange of the sum across lane groups: lanes that differ in bit `kOff` swap halves of their first kLen values and
// add; a lane ends up with half of them, at offset `off`.  With one value left both lanes keep the sum.
template <int kOff, int kLen, int kStop, int E>
__device__ __forceinline__ void walk_fold(float (&a)[E], int &off)
{
    if constexpr (kOff >= kStop) {
        if constexpr (kLen > 1) {
            const bool up = (threadIdx.x & kOff) != 0;
            constexpr int H = kLen / 2;
#pragma unroll
            for (int e = 0; e < H; ++e) {
                const float send = up ? a[e] : a[e + H], keep = up ? a[e + H] : a[e];
                a[e] = keep + __shfl_xor_sync(0xffffffffu, send, kOff);
            }
            if (up) off += H;
            walk_fold<kOff / 2, H, kStop, E>(a, off);
        } else {
            a[0] += __shfl_xor_sync(0xffffffffu, a[0], kOff);
            walk_fold<kOff / 2, 1, kStop, E>(a, off);
        }
    }
}

// Values of a row chunk that a lane holds after the sum across the lane groups.
template <int LPR, int E> __host__ __device__ constexpr int walk_share()
{
    int n = E;
    for (int o = 16; o >= LPR; o /= 2) n = n > 1 ? n / 2 : 1;
    return n;
}

template <typename T, int N> __device__ __forceinline__ void store_share(T *p, const float *v)
{
    if constexpr (sizeof(T) == 4) {
        if constexpr (N == 4) *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
        else if constexpr (N == 2) *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
        else *p = from_float<T>(v[0]);
    } else if constexpr (N == 1) {
        *p = from_float<T>(v[0]);
    } else {
        uint32_t r[N / 2];
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            r[i] = *reinterpret_cast<uint32_t *>(&h);
        }
        if constexpr (N == 8) *reinterpret_cast<uint4 *>(p) = make_uint4(r[0], r[1], r[2], r[3]);
        else if constexpr (N == 4) *reinterpret_cast<uint2 *>(p) = make_uint2(r[0], r[1]);
        else *reinterpret_cast<uint32_t *>(p) = r[0];
    }
}

// Steps (of 32 / LPR rows) whose loads a warp has in flight, and the longest segment that counts as short.
// Measured on whole_mean / three LightGCN layers (see launch_seg_walk), ms: 4 steps at four blocks per SM 3.74 / 3.03,
// 4 steps at three blocks 4.40 / 3.42, 8 steps at three 4.10 / 3.31; short segments up to 4, 8, 16 entries: 3.89 / 3.10,
// 3.74 / 3.03, 3.74 / 3.04.
constexpr int kWalkSteps = 4;
constexpr int kWalkSmall = 8;
constexpr int kWalkRuns = 8;              // stretches of a window, consecutive ones to a warp of the block
template <int LPR, int CPL> __host__ __device__ constexpr int walk_steps() { return CPL >= kWalkSteps ? 1 : kWalkSteps / CPL; }
template <int LPR, int CPL, int E> __host__ __device__ constexpr size_t walk_smem_bytes()
{
    return (size_t)2 * kWalkRuns * LPR * CPL * E * sizeof(float) + kWalkRuns * sizeof(int4);
}

// win_len: entries of a window (block), a multiple of kWalkRuns; cap: entries that the arrays hold, at least; kWide: rows lie
// 4 GB or more apart.
template <typename T, typename PtrT, int LPR, int CPL, bool kWeight, int kWalkWarps, bool kWide>
__global__ void __launch_bounds__(kWalkWarps * 32, CPL > 4 ? 2 : CPL > 1 ? 1 : 32 / kWalkWarps)
seg_walk_kernel(const T *__restrict__ in, int64_t ld_in, const PtrT *__restrict__ ptr, const int32_t *__restrict__ idx,
                const int32_t *n_seg_dev, int64_t n_seg_host, const float *__restrict__ w, int win_len, int64_t cap, int d,
                float *__restrict__ head2, float *__restrict__ tail2, int4 *__restrict__ win_info, SegOut<T> o)
{
    constexpr int E = Chunk<T>::kElems;
    constexpr int G = 32 / LPR;                                  // rows per step
    constexpr int U = walk_steps<LPR, CPL>();                    // steps per group
    constexpr int C = G * U;                                     // entries per group, a divisor of 32
    constexpr int S = walk_share<LPR, E>();
    constexpr int ROW = LPR * CPL * E;
    // Groups of 32 entries that are written out.  Rows that a lane reads in several parts have enough loads in flight with one: four
    // took 141 instead of 80 registers, one block per SM instead of three (10^7 entries of 256 fp32 values and the transpose 2.68 ms,
    // 1.76 with one; two blocks of the widest rows, up to 128 registers, 0.81 where one took 1.15 for 1.2 M entries of 1024).
    constexpr int kUnrollGroups = CPL > 1 ? 1 : 4 < 32 / C ? 4 : 32 / C;
    constexpr int kFar = 1 << 30;
    static_assert(32 % C == 0, "a group takes its ids from one window of 32");
    extern __shared__ float4 seg_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = lane % LPR, sub = lane / LPR;
    float *sh_head = reinterpret_cast<float *>(seg_smem);
    float *sh_tail = sh_head + kWalkRuns * ROW;
    int4 *sh_info = reinterpret_cast<int4 *>(sh_tail + kWalkRuns * ROW);
    __shared__ int32_t sh_win[4];

    const int n_chunks = d / E;
    pdl_wait();
    const int64_t n_seg = n_seg_dev ? (int64_t)__ldcg(n_seg_dev) : n_seg_host;
    const int64_t total = n_seg > 0 ? min((int64_t)__ldcg(ptr + n_seg), cap) : 0;
    if ((int64_t)blockIdx.x * win_len >= total) return;          // a window beyond the stream leaves no record
    const int stretch = win_len / kWalkRuns;
    if (threadIdx.x < 4) sh_win[threadIdx.x] = threadIdx.x == 1 || threadIdx.x == 3 ? 0 : -1;
    constexpr int kOwn = kWalkRuns / kWalkWarps;                 // the warp's stretches, one after another
    int64_t s_next = 0;                                          // the segment in which the warp's next stretch begins
#pragma unroll 1
    for (int own = 0; own < kOwn; ++own) {
    const int rl = warp * kOwn + own;
    const int64_t k0 = (int64_t)blockIdx.x * win_len + (int64_t)rl * stretch;
    int32_t head_seg = -1, head_ends = 0, tail_seg = -1;

    if (k0 < total) {
        const int len = (int)min((int64_t)stretch, total - k0);  // positions below are relative to k0
        const int32_t *__restrict__ idx0 = idx + k0;
        // lanes beyond the row's chunks load its last one and store nothing
        const uint8_t *in_c[CPL];
#pragma unroll
        for (int q = 0; q < CPL; ++q) in_c[q] = reinterpret_cast<const uint8_t *>(in) + (size_t)min(c + q * LPR, n_chunks - 1) * 16;
        const uint64_t ld_bytes = (uint64_t)ld_in * sizeof(T);
        const uint32_t ld_lo = (uint32_t)ld_bytes, ld_hi = (uint32_t)(ld_bytes >> 32);
        // a row's address: one wide product with the lane's chunk as its addend (a stride of 4 GB and more has an upper half too: in
        // kernels of their own, beside the others it cost registers)
        auto load_row = [&](int32_t id, uint4 (&v)[CPL]) {
#pragma unroll
            for (int q = 0; q < CPL; ++q) {
                uint64_t at = (uint64_t)(uint32_t)id * ld_lo + reinterpret_cast<uint64_t>(in_c[q]);
                if constexpr (kWide) at += (uint64_t)((uint32_t)id * ld_hi) << 32;
                v[q] = __ldg(reinterpret_cast<const uint4 *>(at));
            }
        };
        float acc[CPL][E];
        auto clear = [&]() {
#pragma unroll
            for (int q = 0; q < CPL; ++q)
#pragma unroll
                for (int e = 0; e < E; ++e) acc[q][e] = 0.f;
        };
        auto add_row = [&](const uint4 (&raws)[CPL], float wgt, bool mine) {
            if (kWeight && !mine) wgt = 0.f;
#pragma unroll
            for (int q = 0; q < CPL; ++q) {
                const uint4 raw = mine ? raws[q] : make_uint4(0, 0, 0, 0);
                if constexpr (!kWeight) {
                    add_chunk(acc[q], raw, T());
                } else {
                    float x[E];
                    Chunk<T>::unpack(raw, x);
#pragma unroll
                    for (int e = 0; e < E; e += 2) {
                        const float2 r = __ffma2_rn(make_float2(wgt, wgt), make_float2(x[e], x[e + 1]),
                                                    make_float2(acc[q][e], acc[q][e + 1]));
                        acc[q][e] = r.x;
                        acc[q][e + 1] = r.y;
                    }
                }
            }
        };
        auto scale_of = [&](int32_t seg, int n) -> float {
            return o.mean ? __frcp_rn((float)n) : (o.seg_scale ? o.seg_scale[seg] : 1.0f);
        };

        // Segments come in windows of 32, lane i holding where segment s_base + i begins and ends; the ends of the window
        // after it are on their way.
        auto rel = [&](int64_t p) -> int { return (int)max(min(p - k0, (int64_t)kFar), (int64_t)-kFar); };
        auto load_ends = [&](uint32_t b) -> int { return (int64_t)b + lane < n_seg ? rel((int64_t)__ldg(&ptr[(int64_t)b + lane + 1])) : kFar; };
        // unsigned: windows reach beyond the last segment, 2^31 and on
        uint32_t s_base = own == 0 ? (uint32_t)warp_seg_containing(ptr, n_seg, k0) : (uint32_t)s_next;
        int ends = load_ends(s_base), ends_ahead = load_ends(s_base + 32);
        int carry = rel((int64_t)__ldg(&ptr[s_base]));           // where the window's first segment begins
        int quiet = 0;                                           // windows without an entry in a row
        while (true) {
            int beg = __shfl_up_sync(0xffffffffu, ends, 1);
            if (lane == 0) beg = carry;
            const int n = min(ends, len) - max(beg, 0);          // entries of the segment in this stretch
            const bool small = n > 0 && n <= kWalkSmall && beg >= 0 && ends <= len;
            unsigned small_m = __ballot_sync(0xffffffffu, small), big_m = __ballot_sync(0xffffffffu, n > 0 && !small);

            // ---- short segments: one lane group each
            if constexpr (G >= 2) {
                while (small_m) {
                    // the group's segment: the (sub + 1)-th lane that is set
                    unsigned m = small_m;
#pragma unroll
                    for (int k = 0; k < G - 1; ++k)
                        if (k < sub) m &= m - 1;
                    const bool live = m != 0;
                    const int i = live ? __ffs(m) - 1 : 0;
                    const int sb = __shfl_sync(0xffffffffu, beg, i);
                    int sn = __shfl_sync(0xffffffffu, n, i);
                    if (!live) sn = 0;
#pragma unroll
                    for (int k = 0; k < G; ++k) small_m &= small_m - 1;
                    const int longest = __reduce_max_sync(0xffffffffu, sn);
                    clear();
                    for (int j0 = 0; j0 < longest; j0 += U) {
                        uint4 v[U][CPL];
                        float wt[U];
                        int32_t id[U];
                        bool on[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            on[u] = j0 + u < sn;
                            id[u] = on[u] ? __ldg(idx0 + sb + j0 + u) : 0;
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            wt[u] = 1.f;
#pragma unroll
                            for (int q = 0; q < CPL; ++q) v[u][q] = make_uint4(0, 0, 0, 0);
                            if (on[u]) {
                                if (kWeight) wt[u] = __ldg(w + id[u]);
                                load_row(id[u], v[u]);
                            }
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (j0 + u < longest) add_row(v[u], wt[u], true);
                    }
                    if (live) {
                        const int32_t seg = (int32_t)(s_base + i);
                        const float inv = scale_of(seg, sn);
#pragma unroll
                        for (int q = 0; q < CPL; ++q) {
                            const int ch = c + q * LPR;
#pragma unroll
                            for (int e = 0; e < E; ++e) acc[q][e] *= inv;
                            if (ch < n_chunks) Chunk<T>::store(o.out + (int64_t)seg * o.ld_out + ch * E, acc[q]);
                        }
                    }
                }
            }

            // ---- short segments whose rows take the whole warp: their entries in one stream, 32 ids and weights at a time, a row
            // stored where a segment's last entry has been added
            if constexpr (G == 1) {
                int upto = small ? n : 0;                        // entries of the short segments up to and with the lane's
#pragma unroll
                for (int k = 1; k < 32; k <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, upto, k);
                    if (lane >= k) upto += t;
                }
                const int all = __shfl_sync(0xffffffffu, upto, 31);
                clear();
                for (int e0 = 0; e0 < all; e0 += 32) {
                    const int e = min(e0 + lane, all - 1);
                    int i = 0;                                   // the lane of entry e's segment
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (__shfl_sync(0xffffffffu, upto, i + step - 1) <= e) i += step;
                    const int after = __shfl_sync(0xffffffffu, upto, i) - e;             // entries of the segment from e on
                    const int32_t id = __ldg(idx0 + __shfl_sync(0xffffffffu, ends, i) - after);
                    const float wt = kWeight ? __ldg(w + id) : 1.f;
                    const unsigned last = __ballot_sync(0xffffffffu, after == 1 && e0 + lane < all);
                    const int cnt = min(32, all - e0);
#pragma unroll 1
                    for (int c0 = 0; c0 < cnt; c0 += U) {
                        uint4 v[U][CPL];
#pragma unroll
                        for (int u = 0; u < U; ++u) load_row(__shfl_sync(0xffffffffu, id, c0 + u), v[u]);
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            if (c0 + u >= cnt) break;            // uniform over the warp, as is the next condition
                            add_row(v[u], kWeight ? __shfl_sync(0xffffffffu, wt, c0 + u) : 1.f, true);
                            if (!((last >> (c0 + u)) & 1u)) continue;
                            const int j = __shfl_sync(0xffffffffu, i, c0 + u);
                            const int32_t seg = (int32_t)(s_base + j);
                            const float inv = scale_of(seg, __shfl_sync(0xffffffffu, n, j));
#pragma unroll
                            for (int q = 0; q < CPL; ++q) {
                                const int ch = c + q * LPR;
#pragma unroll
                                for (int k = 0; k < E; ++k) acc[q][k] *= inv;
                                if (ch < n_chunks) Chunk<T>::store(o.out + (int64_t)seg * o.ld_out + ch * E, acc[q]);
                            }
                            clear();
                        }
                    }
                }
            }

            // ---- the others one after another, all lane groups on the same segment
            while (big_m) {
                const int i = __ffs(big_m) - 1;
                big_m &= big_m - 1;
                const int32_t seg = (int32_t)(s_base + i);
                const int sbeg = __shfl_sync(0xffffffffu, beg, i), send = __shfl_sync(0xffffffffu, ends, i);
                const int first = max(sbeg, 0), sn = min(send, len) - first;
                const int32_t *__restrict__ ids = idx0 + first;
                auto load_id = [&](int b) -> int32_t { return __ldg(ids + min(b + lane, sn - 1)); };
                int32_t id_cur = load_id(0), id_1 = load_id(32);
                float w_cur = kWeight ? __ldg(w + id_cur) : 0.f;
                clear();
                for (int b = 0; b < sn; b += 32) {
                    const int32_t id_2 = b + 32 < sn ? load_id(b + 64) : 0;
                    const float w_1 = kWeight && b + 32 < sn ? __ldg(w + id_1) : 0.f;
                    auto load_group = [&](int c0, uint4 (&v)[U][CPL]) {
#pragma unroll
                        for (int u = 0; u < U; ++u) load_row(__shfl_sync(0xffffffffu, id_cur, c0 + u * G + sub), v[u]);
                    };
                    auto weight = [&](int e) -> float { return kWeight ? __shfl_sync(0xffffffffu, w_cur, e) : 1.f; };
                    // 32 entries without tests; fewer, or where 32 are one group, a test per group first: segments of small inputs are
                    // mostly cut within 32 (60 k nodes, 10^6 entries, 32 bf16 values, two layers and back 178 us with tests per
                    // entry there, 172)
                    if (C < 32 && b + 32 <= sn) {
#pragma unroll kUnrollGroups
                        for (int c0 = 0; c0 < 32; c0 += C) {
                            uint4 v[U][CPL];
                            load_group(c0, v);
#pragma unroll
                            for (int u = 0; u < U; ++u) add_row(v[u], weight(c0 + u * G + sub), true);
                        }
                    } else {
#pragma unroll 1
                        for (int c0 = 0; c0 < 32 && b + c0 < sn; c0 += C) {
                            uint4 v[U][CPL];
                            load_group(c0, v);
                            if (b + c0 + C <= sn) {
#pragma unroll
                                for (int u = 0; u < U; ++u) add_row(v[u], weight(c0 + u * G + sub), true);
                            } else {
#pragma unroll
                                for (int u = 0; u < U; ++u)
                                    if (b + c0 + u * G < sn)     // uniform over the warp
                                        add_row(v[u], weight(c0 + u * G + sub), b + c0 + u * G + sub < sn);
                            }
                        }
                    }
                    id_cur = id_1;
                    id_1 = id_2;
                    w_cur = w_1;
                }
                int off = 0;
#pragma unroll
                for (int q = 0; q < CPL; ++q) {
                    off = 0;
                    walk_fold<16, E, LPR, E>(acc[q], off);
                }
                if (sbeg >= 0 && send <= len) {
                    const float inv = scale_of(seg, sn);
                    T *row = o.out + (int64_t)seg * o.ld_out + off;
#pragma unroll
                    for (int q = 0; q < CPL; ++q) {
                        const int ch = c + q * LPR;
                        float r[S];
#pragma unroll
                        for (int e = 0; e < S; ++e) r[e] = acc[q][e] * inv;          // inv = 1 without mean / scale
                        if (ch < n_chunks) store_share<T, S>(row + ch * E, r);
                    }
                } else {                                         // cut by the stretch's ends: a part for the join
                    float *dst = (sbeg >= 0 ? sh_tail : sh_head) + rl * ROW + off;
#pragma unroll
                    for (int q = 0; q < CPL; ++q) {
                        store_share<float, (S > 4 ? 4 : S)>(dst + (c + q * LPR) * E, acc[q]);
                        if constexpr (S == 8) store_share<float, 4>(dst + (c + q * LPR) * E + 4, acc[q] + 4);
                    }
                    if (sbeg >= 0) tail_seg = seg;
                    else { head_seg = seg; head_ends = send <= len ? 1 : 0; }
                }
            }
            carry = __shfl_sync(0xffffffffu, ends, 31);          // the offsets do not decrease: the window's last end
            if (carry >= len) {
                if (own + 1 < kOwn)                              // the segments that end in this stretch lie behind
                    s_next = min((int64_t)s_base + __popc(__ballot_sync(0xffffffffu, ends <= len)), n_seg - 1);
                break;
            }
            quiet = __any_sync(0xffffffffu, n > 0) ? 0 : quiet + 1;
            if (quiet < kQuietWindows) {
                s_base += 32;
                ends = ends_ahead;
            } else {                                             // a long stretch of empty segments
                s_base = window_found(s_base, (uint32_t)warp_seg_containing(ptr, n_seg, k0 + carry));
                ends = load_ends(s_base);
                quiet = 0;
            }
            ends_ahead = load_ends(s_base + 32);
        }
    }
    if (lane == 0) sh_info[rl] = make_int4(head_seg, head_ends, tail_seg, 0);
    }
    __syncthreads();
    if (lane < LPR) {
#pragma unroll 1
        for (int rl = warp * kOwn; rl < (warp + 1) * kOwn; ++rl) {
            const int4 info = sh_info[rl];
            seg_join_run<T, PtrT, LPR, CPL, 0>(sh_head, sh_tail, sh_info, sh_win, rl, kWalkRuns, blockIdx.x, lane, n_chunks, d, info.x, info.y, info.z,
                                               ptr, head2, tail2, o, nullptr, 0);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) win_info[blockIdx.x] = make_int4(sh_win[0], sh_win[1], sh_win[2], 0);
}

// B200: 5 M nodes, 10^8 entries, 64 bf16 values, forward and transposed 3.74 -> 3.18 ms (8.8 TB/s of gathered rows);
// 500 k nodes, 2 * 10^7 entries, 64 fp32 values, weighted, per layer 0.45 -> 0.40 ms (12.7 TB/s).
template <typename T, typename PtrT, int LPR, int CPL, bool kWeight, int kWalkWarps, bool kWide>
inline void launch_seg_walk(const T *in, int64_t ld_in, const PtrT *ptr, const int32_t *idx, const int32_t *n_seg_dev,
                            int64_t n_seg_host, int64_t cap_seg, const float *w, int run_len, int d, const SegScratch &sc,
                            const SegOut<T> &o, cudaStream_t st)
{
    constexpr size_t smem = walk_smem_bytes<LPR, CPL, Chunk<T>::kElems>();
    auto kern = seg_walk_kernel<T, PtrT, LPR, CPL, kWeight, kWalkWarps, kWide>;
    if (smem > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    tap_begin(TAP_SEG_L1, st);
    note_launch();
    launch_pdl(n_seg_dev && sc.cap_runs * run_len < kChainEdges, kern, dim3((unsigned)sc.n_windows), dim3(kWalkWarps * 32), smem, st, in, ld_in,
               ptr, idx, n_seg_dev, n_seg_host, w, run_len * sc.runs_per_window, sc.cap_runs * run_len, d, sc.head2, sc.tail2,
               sc.win_info, o);
    tap_end(TAP_SEG_L1, st);
    launch_seg_final(ptr, n_seg_dev, n_seg_host, cap_seg, run_len, d, sc, o, st);
}

// Four warps with two stretches each, of which fewer wait before the join, or eight with one.  Four pay for rows of 65 to 128 bytes
// once so many windows follow one another that a block's begin and end count less than the wait.  B200, ms with four / eight, mean and
// transpose, 64 bf16 values: 2 * 10^7 entries of 500 k rows 0.70 / 0.65, 2.5 * 10^7 of 2.5 M 1.23 / 1.17, 5 * 10^7 of 1, 2.5 and 5 M
// 1.38 / 1.39, 1.73 / 1.74 and 2.15 / 2.20, 10^8 of 1, 5 and 10 M 2.26 / 2.37, 3.19 / 3.35 and 4.01 / 4.20; 32 fp32 values, 5 * 10^7 1.57 / 1.56,
// 10^8 2.89 / 3.01.  Narrower rows, whose stretches hold fewer loads: 3 * 10^7 of 32 bf16 values 1.20 / 1.06, 10^8 2.44 / 2.43; wider ones,
// three layers of 2 * 10^7 entries of 256 bytes, 2.83 / 2.76.
constexpr int64_t kWalkPaired = 48'000'000;          // entries

// Same contract as dispatch_seg_reduce, without an entry -> segment array, self rows or masks.
template <typename T, typename PtrT, bool kWeight>
inline bool dispatch_seg_walk(const T *in, int64_t ld_in, const PtrT *ptr, const int32_t *idx, const int32_t *n_seg_dev,
                              int64_t n_seg_host, int64_t cap_seg, const float *w, int run_len, int d, int32_t dtype,
                              const SegScratch &sc, const SegOut<T> &o, cudaStream_t st)
{
    const RowShape rs = row_shape(d, dtype);
    const bool wide = (uint64_t)ld_in * sizeof(T) >> 32 != 0;
#define E2E_WALK(L, C, WARPS, WIDE)                                                                                         \
    launch_seg_walk<T, PtrT, L, C, kWeight, WARPS, WIDE>(in, ld_in, ptr, idx, n_seg_dev, n_seg_host, cap_seg, w, run_len, d, sc, o, st)
#define E2E_CASE(L, C)                                                                                                      \
    if (rs.lpr == L && rs.cpl == C) {                                                                                       \
        if (wide) {                                                                                                         \
            E2E_WALK(L, C, 8, true);                                                                                        \
            return true;                                                                                                    \
        }                                                                                                                   \
        if constexpr (L == 8 && sizeof(PtrT) == 8)                                                                          \
            if (sc.cap_runs * run_len >= kWalkPaired) {                                                                     \
                E2E_WALK(L, C, 4, false);                                                                                   \
                return true;                                                                                                \
            }                                                                                                               \
        E2E_WALK(L, C, 8, false);                                                                                           \
        return true;                                                                                                        \
    }
    E2E_CASE(4, 1) E2E_CASE(8, 1) E2E_CASE(16, 1) E2E_CASE(32, 1) E2E_CASE(32, 2) E2E_CASE(32, 4)
    if constexpr (sizeof(T) == 4) {      // rows of 2049 .. 4096 bytes exist only for fp32 (dim <= kMaxDim)
        E2E_CASE(32, 8)
    }
#undef E2E_CASE
#undef E2E_WALK
    return false;
}

}  // namespace e2egrec
