// Graph ingest on the device: canonical CSR from an edge list, and the CSC (transpose) of a CSR.
// Both are stable radix sorts plus offset look-ups, so the result depends only on the multiset of edges: rows ordered by
// (row, col), columns by (col, CSR position), parallel edges kept.
//
// The CSR is the (col, row) pairs sorted by column and then, key and value exchanged, by row: the other id travels as the
// value, so nothing is gathered between the sorts (entries equal in both ids need no order).  The transpose sorts
// (col, position) and looks up the row of every position afterwards.  B200, 10^7 interactions (2 * 10^7 entries, 500 k nodes),
// CSR and CSC together: 3.23 -> 1.52 ms.
#include <algorithm>

#include "radix.cuh"
#include "segwalk.cuh"

namespace e2egrec {
namespace {

struct IngestScratch {
    int32_t *counts;                 // int32[4]: CNT_STATUS is the status word of the run
    int32_t *a, *k0, *v0, *k1, *v1;  // arrays of m
    SortState sort[2];
    char *zero;                      // the part that has to be zero beforehand
    size_t zero_bytes, bytes;
};

IngestScratch carve_ingest(int64_t m, void *base)
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
    for (int32_t **p : {&s.a, &s.k0, &s.v0, &s.k1, &s.v1}) *p = (int32_t *)take(mm * 4);
    const int64_t tiles = ceil_div((int64_t)mm, kSortTile);
    const size_t begin = off;
    s.zero = base ? static_cast<char *>(base) + off : nullptr;
    for (SortState &ss : s.sort) {
        ss.ghist = (unsigned *)take(kSortCountWords * sizeof(unsigned));
        ss.tiles = tiles;
        ss.state = (unsigned *)take(sort_state_bytes(tiles));
    }
    s.zero_bytes = off - begin;
    s.bytes = off;
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
// 0, which the first pass of a sort makes of them.
__global__ void __launch_bounds__(256)
id_hist_kernel(const int32_t *__restrict__ ids0, const int32_t *__restrict__ ids1, int64_t m, int64_t n, int bits, int passes,
               unsigned *__restrict__ ghist0, unsigned *__restrict__ ghist1, int32_t *counts)
{
    extern __shared__ unsigned hist_sm[];                        // [arrays][passes][1 << bits]
    const int R = 1 << bits, per = passes * R;
    const int all = ids1 ? 2 * per : per;
    for (int d = threadIdx.x; d < all; d += 256) hist_sm[d] = 0;
    __syncthreads();
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < m; i += (int64_t)gridDim.x * 256) {
        uint32_t v0 = (uint32_t)ids0[i], v1 = ids1 ? (uint32_t)ids1[i] : 0u;
        if (v0 >= (uint64_t)n) { bad = true; v0 = 0; }
        if (v1 >= (uint64_t)n) { bad = true; v1 = 0; }
        for (int p = 0; p < passes; ++p) {
            atomicAdd(&hist_sm[p * R + ((v0 >> (p * bits)) & (R - 1))], 1u);
            if (ids1) atomicAdd(&hist_sm[per + p * R + ((v1 >> (p * bits)) & (R - 1))], 1u);
        }
    }
    if (bad) atomicOr((unsigned *)&counts[CNT_STATUS], E2EGREC_DEV_RANGE);
    __syncthreads();
    for (int d = threadIdx.x; d < all; d += 256) {
        if (!hist_sm[d]) continue;
        const int e = d % per;
        atomicAdd(&(d < per ? ghist0 : ghist1)[(e / R) * kMaxRadix + e % R], hist_sm[d]);
    }
}

// row_of[e] = row of CSR position e.  A warp owns 1024 consecutive positions: it finds its first row by a search over the
// offsets and then goes through them 32 rows at a time, lane i holding the end of row base + i; a position's row is the
// number of ends at or before it, found by bisection across the lanes.
__global__ void __launch_bounds__(256)
expand_rows_kernel(const int64_t *__restrict__ indptr, int64_t n_rows, int64_t m, int32_t *__restrict__ row_of)
{
    constexpr int kSpan = 1024;
    const int lane = threadIdx.x & 31;
    const int64_t k0 = (((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5) * kSpan;
    if (k0 >= m) return;
    const int len = (int)min((int64_t)kSpan, m - k0);
    int64_t base = warp_seg_containing(indptr, n_rows, k0);
    auto load_ends = [&](int64_t b) -> int { return b + lane < n_rows ? (int)min(indptr[b + lane + 1] - k0, (int64_t)kSpan) : kSpan; };
    int ends = load_ends(base);
    int quiet = 0;
    for (int e0 = 0; e0 < len;) {
        const int last = __shfl_sync(0xffffffffu, ends, 31);     // positions before it belong to this window of rows
        if (last > e0) {
            quiet = 0;
            const int e = e0 + lane;
            int r = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, ends, r + step - 1) <= e) r += step;
            if (e < last && e < len) row_of[k0 + e] = (int32_t)max(min(base + r, n_rows - 1), (int64_t)0);
            e0 = min(e0 + 32, last);
            if (e0 < last) continue;
            if (e0 >= len) break;
        } else {
            ++quiet;
        }
        base = quiet < kQuietWindows ? base + 32 : window_found(base, warp_seg_containing(indptr, n_rows, k0 + e0));
        ends = load_ends(base);
    }
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

SortPlan plan_for(int64_t key_range) { return sort_plan((int32_t)std::min<int64_t>(std::max<int64_t>(key_range, 2), 0x7fffffff)); }

void id_hist(const int32_t *ids0, const int32_t *ids1, int64_t m, int64_t n, const SortPlan &sp, IngestScratch &s, cudaStream_t st)
{
    cudaMemsetAsync(s.zero, 0, s.zero_bytes, st);
    const size_t smem = (size_t)(ids1 ? 2 : 1) * sp.passes * (1 << sp.bits) * sizeof(unsigned);
    note_launch();
    id_hist_kernel<<<(unsigned)std::min<int64_t>(ceil_div(m, 2048), 148 * 8), 256, smem, st>>>(ids0, ids1, m, n, sp.bits, sp.passes,
                                                                                             s.sort[0].ghist, s.sort[1].ghist, s.counts);
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
    IngestScratch s = carve_ingest(n_edges, ws);
    if (!ws) { *ws_bytes = s.bytes; return E2EGREC_OK; }
    if (*ws_bytes < s.bytes) { *ws_bytes = s.bytes; return E2EGREC_ERR_WORKSPACE; }
    if (reinterpret_cast<uintptr_t>(ws) % 256) return E2EGREC_ERR_ALIGN;
    if (!indptr || (n_edges > 0 && (!row || !col || !indices))) return E2EGREC_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t m = n_edges;
    note_launch();
    ingest_begin_kernel<<<1, 1, 0, st>>>(s.counts, (int32_t)m);
    if (m > 0) {
        const SortPlan sp = plan_for(n_nodes);
        const int32_t clamp = (int32_t)std::max<int64_t>(n_nodes, 1);
        id_hist(col, row, m, n_nodes, sp, s, st);
        // (col, row) by column, then (row, col) by row
        const int32_t *k = col, *v = row;
        int32_t *ka = s.k0, *va = s.v0, *kb = s.k1, *vb = s.v1;
        for (int q = 0; q < 2 * sp.passes; ++q) {
            const int sort = q / sp.passes, pass = q % sp.passes;
            if (q == sp.passes) std::swap(k, v);
            const bool last = q == 2 * sp.passes - 1;
            sort_pass<int32_t>(sp, k, v, nullptr, m, q == 0 ? clamp : 0, q == 0 ? clamp : 0, pass, s.sort[sort], false, last ? s.a : ka,
                               last ? indices : va, SortMap{}, &s.counts[CNT_STATUS], st);
            k = ka;
            v = va;
            std::swap(ka, kb);
            std::swap(va, vb);
        }                                                        // s.a = rows sorted
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
    IngestScratch s = carve_ingest(csr->n_edges, ws);
    if (!ws) { *ws_bytes = s.bytes; return E2EGREC_OK; }
    if (*ws_bytes < s.bytes) { *ws_bytes = s.bytes; return E2EGREC_ERR_WORKSPACE; }
    if (reinterpret_cast<uintptr_t>(ws) % 256) return E2EGREC_ERR_ALIGN;
    if (!csr->indptr || !csc_ptr || (csr->n_edges > 0 && (!csr->indices || !csc_row || !csc_eid))) return E2EGREC_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t m = csr->n_edges;
    const int32_t *sorted = s.k0;
    note_launch();
    ingest_begin_kernel<<<1, 1, 0, st>>>(s.counts, (int32_t)m);
    if (m > 0) {
        const SortPlan sp = plan_for(n_cols);
        id_hist(csr->indices, nullptr, m, n_cols, sp, s, st);
        note_launch();
        expand_rows_kernel<<<(unsigned)ceil_div(m, 8 * 1024), 256, 0, st>>>(csr->indptr, csr->n_nodes, m, s.a);
        const int32_t *k = csr->indices, *v = nullptr;           // value = CSR position
        int32_t *ka = s.k0, *va = s.v0, *kb = s.k1, *vb = s.v1;
        for (int q = 0; q < sp.passes; ++q) {
            const int32_t clamp = q == 0 ? (int32_t)std::max<int64_t>(n_cols, 1) : 0;
            if (q == sp.passes - 1)
                sort_pass<int64_t>(sp, k, v, nullptr, m, clamp, (int32_t)m, q, s.sort[0], false, ka, csc_eid, SortMap{},
                                   &s.counts[CNT_STATUS], st);
            else
                sort_pass<int32_t>(sp, k, v, nullptr, m, clamp, (int32_t)m, q, s.sort[0], false, ka, va, SortMap{},
                                   &s.counts[CNT_STATUS], st);
            k = ka;
            v = va;
            std::swap(ka, kb);
            std::swap(va, vb);
        }
        sorted = k;                                              // the columns in order
        note_launch();
        rows_of_kernel<<<(unsigned)std::min<int64_t>(ceil_div(m, 1024), 148 * 16), 256, 0, st>>>(csc_eid, s.a, m, csc_row);
    }
    note_launch();
    offsets_kernel<<<wide_grid(n_cols + 1), 256, 0, st>>>(sorted, m, n_cols, s.counts, csc_ptr);
    if (status) cudaMemcpyAsync(status, &s.counts[CNT_STATUS], sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
    return check_launch("csr_transpose");
}
