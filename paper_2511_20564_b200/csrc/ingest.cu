// Graph ingest on the device: canonical CSR from an edge list, and the CSC (transpose) of a CSR.
// Both are stable radix sorts plus offset look-ups, so the result depends only on the multiset of edges: rows ordered by
// (row, col), columns by (col, CSR position), parallel edges kept.
//
// The CSR is the (col, row) pairs sorted by column and then, key and value exchanged, by row: the other id travels as the
// value, so nothing is gathered between the sorts (entries equal in both ids need no order).  The transpose sorts
// (col, position) and looks up the row of every position afterwards.  B200, 10^7 interactions (2 * 10^7 entries, 500 k nodes),
// CSR and CSC together: 1.51 -> 1.19 ms.
#include <algorithm>

#include "radix.cuh"
#include "segwalk.cuh"

namespace e2egrec {
namespace {

struct IngestScratch {
    int32_t *counts;                 // int32[4]: CNT_STATUS is the status word of the run
    int32_t *a;                      // [m]
    uint2 *pair[2];                  // [m]
    SortState sort[2];
    char *zero;                      // the part that has to be zero beforehand
    size_t zero_bytes, bytes;
};

SortPlan plan_for(int64_t key_range) { return sort_plan((int32_t)std::min<int64_t>(std::max<int64_t>(key_range, 2), 0x7fffffff)); }

// n_sorts sorts of m entries by `sp`: digit counts and scan state of what these will use lie together, to be zeroed at once
// (zeroing the smaller tiles' state for two sorts, 80 MB, took 14 us at 2 * 10^7 entries).  The size goes by m alone and grows with
// it, so that a workspace serves shorter lists, other id ranges and the other call: two sorts, state for any digits and for the tiles of
// whichever list up to m has most.
IngestScratch carve_ingest(int64_t m, const SortPlan &sp, int n_sorts, void *base)
{
    IngestScratch s{};
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *p = base ? static_cast<char *>(base) + off : nullptr;
        off += align_up(bytes, 256);
        return p;
    };
    const size_t mm = (size_t)(m > 0 ? m : 1);
    s.counts = (int32_t *)take(256);
    s.a = (int32_t *)take(mm * 4);
    for (uint2 *&p : s.pair) p = (uint2 *)take(mm * 8);
    const int64_t tiles = ceil_div((int64_t)mm, (int64_t)mm >= kSortWide ? kSortWideTile : kSortTile);
    const size_t begin = off;
    s.zero = base ? static_cast<char *>(base) + off : nullptr;
    for (int i = 0; i < n_sorts; ++i) {
        SortState &ss = s.sort[i];
        ss.ghist = (unsigned *)take(kSortCountWords * sizeof(unsigned));
        ss.tiles = tiles;
        ss.state = (unsigned *)take(sizeof(unsigned) * (size_t)sp.passes * (size_t)tiles << sp.bits);
    }
    s.zero_bytes = off - begin;
    const int64_t most = std::max(ceil_div(std::min<int64_t>((int64_t)mm, kSortWide - 1), (int64_t)kSortTile), ceil_div((int64_t)mm, kSortWideTile));
    s.bytes = begin + 2 * (align_up(kSortCountWords * sizeof(unsigned), 256) + align_up(sort_state_bytes(most), 256));
    return s;
}

__global__ void ingest_begin_kernel(int32_t *counts, int32_t m)
{
    counts[CNT_DST] = 0;
    counts[CNT_SRC] = 0;
    counts[CNT_EDGES] = m;
    counts[CNT_STATUS] = 0;
}

// Digit counts of one or two id arrays for every pass of their sorts.  Ids outside [0, n) are flagged here and count as
// 0, which the first pass of a sort makes of them.  One block of 1024 threads per SM, and two copies of the counts, for even
// and odd lanes: what the blocks add to the global counts at their ends (4096 each) and the lanes of a warp that meet in a
// hub's digits were what it cost.
constexpr int kHistThreads = 1024;
__global__ void __launch_bounds__(kHistThreads)
id_hist_kernel(const int32_t *__restrict__ ids0, const int32_t *__restrict__ ids1, int64_t m, int64_t n, int bits, int passes,
               unsigned *__restrict__ ghist0, unsigned *__restrict__ ghist1, int32_t *counts)
{
    extern __shared__ unsigned hist_sm[];                        // [2][arrays][passes][1 << bits]
    const int R = 1 << bits, per = passes * R;
    const int all = ids1 ? 2 * per : per;
    for (int d = threadIdx.x; d < 2 * all; d += kHistThreads) hist_sm[d] = 0;
    __syncthreads();
    unsigned *h = hist_sm + (threadIdx.x & 1) * all;
    bool bad = false;
    const int64_t step = (int64_t)gridDim.x * kHistThreads;
    auto count = [&](uint32_t v, unsigned *hh) {
        if (v >= (uint64_t)n) { bad = true; v = 0; }
        for (int p = 0; p < passes; ++p) atomicAdd(&hh[p * R + ((v >> (p * bits)) & (R - 1))], 1u);
    };
    constexpr int U = 4;
    int64_t i = (int64_t)blockIdx.x * kHistThreads + threadIdx.x;
    for (; i + (U - 1) * step < m; i += U * step) {
        uint32_t v0[U], v1[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v0[u] = (uint32_t)__ldg(ids0 + i + u * step);
            v1[u] = ids1 ? (uint32_t)__ldg(ids1 + i + u * step) : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            count(v0[u], h);
            if (ids1) count(v1[u], h + per);
        }
    }
    for (; i < m; i += step) {
        count((uint32_t)ids0[i], h);
        if (ids1) count((uint32_t)ids1[i], h + per);
    }
    if (bad) atomicOr((unsigned *)&counts[CNT_STATUS], E2EGREC_DEV_RANGE);
    __syncthreads();
    for (int d = threadIdx.x; d < all; d += kHistThreads) {
        const unsigned c = hist_sm[d] + hist_sm[all + d];
        if (!c) continue;
        const int e = d % per;
        atomicAdd(&(d < per ? ghist0 : ghist1)[(e / R) * kMaxRadix + e % R], c);
    }
}

// row_of[e] = row of CSR position e.  A warp owns kSpan consecutive positions: it finds its first row by a search over the
// offsets, goes through the rows 32 at a time and notes every row with entries where it begins, in shared memory; a running
// maximum over the span (each lane over 32 positions, then over the lanes) carries the rows on.  (A bisection across the lanes
// for every 32 positions, as before, was 1100 instructions a span where this is 300: 2 * 10^7 positions 52 -> 26 us.)
__global__ void __launch_bounds__(256)
expand_rows_kernel(const int64_t *__restrict__ indptr, int64_t n_rows, int64_t m, int32_t *__restrict__ row_of)
{
    constexpr int kSpan = 1024, kPad = 33;                       // position p lies at (p / 32) * kPad + p % 32
    __shared__ int32_t sm[8][32 * kPad];
    const int lane = threadIdx.x & 31;
    int32_t *mark = sm[threadIdx.x >> 5];
    const int64_t k0 = (((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5) * kSpan;
    if (k0 >= m) return;
    const int len = (int)min((int64_t)kSpan, m - k0);
    int64_t base = warp_seg_containing(indptr, n_rows, k0);
    const int32_t first = (int32_t)max(min(base, n_rows - 1), (int64_t)0);
#pragma unroll
    for (int c = 0; c < 32; ++c) mark[c * kPad + lane] = 0;
    __syncwarp();
    auto load_beg = [&](int64_t b) -> int { return b + lane <= n_rows ? (int)max(min(indptr[b + lane] - k0, (int64_t)kSpan), (int64_t)0) : kSpan; };
    int beg = load_beg(base);
    for (int quiet = 0;;) {
        const int beg_n = load_beg(base + 32);                   // the window after this one, on its way
        const int after = __shfl_sync(0xffffffffu, beg_n, 0);    // where the row behind the window begins
        int end = __shfl_down_sync(0xffffffffu, beg, 1);
        if (lane == 31) end = after;
        const int32_t row = row_to_note(base + lane, n_rows, beg, end, len);
        if (row >= 0) mark[(beg >> 5) * kPad + (beg & 31)] = row;
        if (!more_rows(base, n_rows, after, len)) break;
        quiet = __any_sync(0xffffffffu, beg < end) ? 0 : quiet + 1;
        if (quiet < kQuietWindows) {
            base += 32;
            beg = beg_n;
        } else {                                                 // a long stretch of empty rows
            base = window_found(base, warp_seg_containing(indptr, n_rows, k0 + after));
            beg = load_beg(base);
            quiet = 0;
        }
    }
    __syncwarp();
    int32_t run = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) run = max(run, mark[lane * kPad + j]);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(0xffffffffu, run, o);
        if (lane >= o) run = max(run, t);
    }
    run = __shfl_up_sync(0xffffffffu, run, 1);
    run = lane > 0 ? max(run, first) : first;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        run = max(run, mark[lane * kPad + j]);
        mark[lane * kPad + j] = run;
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 32; ++c)
        if (c * 32 + lane < len) row_of[k0 + c * 32 + lane] = mark[c * kPad + lane];
}

// csc_row[k] = row_of[csc_eid[k]], four scattered reads per thread in flight.  In a launch of its own row_of stays in L2
// (80 MB at 2 * 10^7 entries); looked up by the sort's last pass, between its own 320 MB of output, it cost 160 us
// against 59; the search over the offsets that came before took 360.
__global__ void rows_of_kernel(const int64_t *__restrict__ eid, const int32_t *__restrict__ row_of, int64_t m, int32_t *__restrict__ csc_row)
{
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m; k += 4 * step) {
        int32_t r[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t e = k + q * step < m ? __ldcs(eid + k + q * step) : 0;
            r[q] = __ldg(row_of + ((uint64_t)e < (uint64_t)m ? e : 0));      // beyond: after a wait of the sort that ran out
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (k + q * step < m) __stcs(csc_row + k + q * step, r[q]);
    }
}

// ptr[s] = first position of the sorted key array whose key is >= s, for s = 0 .. n; all zero after a wait of the sort that
// ran out
__global__ void offsets_kernel(const int32_t *__restrict__ sorted, int64_t m, int64_t n, const int32_t *__restrict__ counts,
                               int64_t *__restrict__ ptr)
{
    if ((uint32_t)counts[CNT_STATUS] & E2EGREC_DEV_TIMEOUT) m = 0;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s <= n; s += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = m;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if ((int64_t)sorted[mid] < s) lo = mid + 1; else hi = mid;
        }
        ptr[s] = lo;
    }
}

unsigned wide_grid(int64_t n) { return (unsigned)std::min<int64_t>(ceil_div(n > 0 ? n : 1, 256), 148 * 16); }

void id_hist(const int32_t *ids0, const int32_t *ids1, int64_t m, int64_t n, const SortPlan &sp, IngestScratch &s, cudaStream_t st)
{
    cudaMemsetAsync(s.zero, 0, s.zero_bytes, st);
    const size_t smem = (size_t)(ids1 ? 4 : 2) * sp.passes * (1 << sp.bits) * sizeof(unsigned);      // at most 32 KB
    note_launch();
    id_hist_kernel<<<(unsigned)std::min<int64_t>(ceil_div(m, 4 * kHistThreads), 148), kHistThreads, smem, st>>>(
        ids0, ids1, m, n, sp.bits, sp.passes, s.sort[0].ghist, s.sort[1].ghist, s.counts);
}

}  // namespace
}  // namespace e2egrec

using namespace e2egrec;

extern "C" int32_t e2egrec_graph_from_coo(int64_t n_nodes, int64_t n_edges, const int32_t *row, const int32_t *col,
                                          int64_t *indptr, int32_t *indices, int32_t *status, void *ws,
                                          size_t *ws_bytes, void *stream)
{
    if (!ws_bytes) return E2EGREC_ERR_NULL;
    if (n_nodes < 0 || n_edges < 0) return E2EGREC_ERR_ARG;
    if (n_nodes >= (1ll << 31) || n_edges >= (1ll << 31) - 1) return E2EGREC_ERR_UNSUPPORTED;
    const SortPlan sp = plan_for(n_nodes);
    IngestScratch s = carve_ingest(n_edges, sp, 2, ws);
    if (!ws) { *ws_bytes = s.bytes; return E2EGREC_OK; }
    if (*ws_bytes < s.bytes) { *ws_bytes = s.bytes; return E2EGREC_ERR_WORKSPACE; }
    if (reinterpret_cast<uintptr_t>(ws) % 256) return E2EGREC_ERR_ALIGN;
    if (!indptr || (n_edges > 0 && (!row || !col || !indices))) return E2EGREC_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t m = n_edges;
    note_launch();
    ingest_begin_kernel<<<1, 1, 0, st>>>(s.counts, (int32_t)m);
    if (m > 0) {
        const int32_t clamp = (int32_t)std::max<int64_t>(n_nodes, 1);
        id_hist(col, row, m, n_nodes, sp, s, st);
        // (col, row) by column, then (row, col) by row
        SortIn in{col, row, nullptr, false, kRankAny};           // equal pairs are alike: the first pass needs no order
        for (int q = 0; q < 2 * sp.passes; ++q) {
            const int sort = q / sp.passes, pass = q % sp.passes;
            const bool last = q == 2 * sp.passes - 1;
            if (q == sp.passes) {
                in.swap = true;
                in.rank = kRankSpread;
            }
            SortOut<int32_t> out{};
            if (last) {
                out.keys = s.a;                                  // the rows in order
                out.vals = indices;
            } else {
                out.pairs = s.pair[q & 1];
            }
            sort_pass<int32_t>(sp, in, nullptr, m, q == 0 ? clamp : 0, q == 0 ? clamp : 0, pass, s.sort[sort], false, out,
                               &s.counts[CNT_STATUS], st);
            in = SortIn{nullptr, nullptr, s.pair[q & 1], false, kRankMatch};
        }
    }
    note_launch();
    offsets_kernel<<<wide_grid(n_nodes + 1), 256, 0, st>>>(s.a, m, n_nodes, s.counts, indptr);
    if (status) cudaMemcpyAsync(status, &s.counts[CNT_STATUS], sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
    return check_launch("graph_from_coo");
}

extern "C" int32_t e2egrec_csr_transpose(const e2egrec_csr *csr, int64_t n_cols, int64_t *csc_ptr, int32_t *csc_row,
                                         int64_t *csc_eid, int32_t *status, void *ws, size_t *ws_bytes, void *stream)
{
    if (!ws_bytes || !csr) return E2EGREC_ERR_NULL;
    if (csr->n_nodes < 0 || csr->n_edges < 0 || n_cols < 0) return E2EGREC_ERR_ARG;
    if (csr->n_nodes >= (1ll << 31) || n_cols >= (1ll << 31) || csr->n_edges >= (1ll << 31) - 1) return E2EGREC_ERR_UNSUPPORTED;
    const SortPlan sp = plan_for(n_cols);
    IngestScratch s = carve_ingest(csr->n_edges, sp, 1, ws);
    if (!ws) { *ws_bytes = s.bytes; return E2EGREC_OK; }
    if (*ws_bytes < s.bytes) { *ws_bytes = s.bytes; return E2EGREC_ERR_WORKSPACE; }
    if (reinterpret_cast<uintptr_t>(ws) % 256) return E2EGREC_ERR_ALIGN;
    if (!csr->indptr || !csc_ptr || (csr->n_edges > 0 && (!csr->indices || !csc_row || !csc_eid))) return E2EGREC_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t m = csr->n_edges;
    const int32_t *sorted = s.a;
    note_launch();
    ingest_begin_kernel<<<1, 1, 0, st>>>(s.counts, (int32_t)m);
    if (m > 0) {
        id_hist(csr->indices, nullptr, m, n_cols, sp, s, st);
        note_launch();
        expand_rows_kernel<<<(unsigned)ceil_div(m, 8 * 1024), 256, 0, st>>>(csr->indptr, csr->n_nodes, m, s.a);
        SortIn in{csr->indices, nullptr, nullptr, false, kRankMatch};        // value = CSR position
        for (int q = 0; q < sp.passes; ++q) {
            const int32_t clamp = q == 0 ? (int32_t)std::max<int64_t>(n_cols, 1) : 0;
            if (q == sp.passes - 1) {
                SortOut<int64_t> out{};
                sorted = out.keys = reinterpret_cast<int32_t *>(s.pair[q & 1]);          // the columns in order
                out.vals = csc_eid;
                sort_pass<int64_t>(sp, in, nullptr, m, clamp, (int32_t)m, q, s.sort[0], false, out, &s.counts[CNT_STATUS], st);
            } else {
                SortOut<int32_t> out{};
                out.pairs = s.pair[q & 1];
                sort_pass<int32_t>(sp, in, nullptr, m, clamp, (int32_t)m, q, s.sort[0], false, out, &s.counts[CNT_STATUS], st);
                in = SortIn{nullptr, nullptr, s.pair[q & 1], false, kRankMatch};
            }
        }
        note_launch();
        rows_of_kernel<<<(unsigned)std::min<int64_t>(ceil_div(m, 1024), 148 * 16), 256, 0, st>>>(csc_eid, s.a, m, csc_row);
    }
    note_launch();
    offsets_kernel<<<wide_grid(n_cols + 1), 256, 0, st>>>(sorted, m, n_cols, s.counts, csc_ptr);
    if (status) cudaMemcpyAsync(status, &s.counts[CNT_STATUS], sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
    return check_launch("csr_transpose");
}
