// Steps of the walks over segment offsets (device code; plain C++ for tests on the host).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define E2EGREC_HD __host__ __device__ __forceinline__
#else
#define E2EGREC_HD inline
#endif

namespace e2egrec {

constexpr int kQuietWindows = 4;

// A walk looks at windows of 32 segments.  After kQuietWindows windows without an entry it asks a search where the next
// entry's segment is; this is where it goes on from the window at `base` when the search says `found`.  Never the same window
// again: offsets that decrease, which no entry point accepts but none can refuse, could make a search go back, and the walk
// ends nevertheless, after one window per 32 segments at most.
template <typename T> E2EGREC_HD T window_found(T base, T found)
{
    const T next = base + 32;
    return found > next ? found : next;
}

// The expansion of offsets into one row per entry goes over spans of entries.  The row to be noted at its first entry, at
// `beg` of a span of `len` entries, or -1: it began before the span (the span's first row is known), begins behind it or has no
// entries.  Row n_rows, "beginning" at the last offset, is met where the offsets end before the entries, which no entry
// point accepts but none can refuse: those entries count as the last row's, so that no number beyond it leaves.
E2EGREC_HD int32_t row_to_note(int64_t row, int64_t n_rows, int beg, int end, int len)
{
    return beg > 0 && beg < end && beg < len ? (int32_t)(row < n_rows ? row : n_rows - 1) : -1;
}
// Whether the window of 32 rows behind the one at `base`, which begins at `after`, has a row to be noted (row n_rows included).
E2EGREC_HD bool more_rows(int64_t base, int64_t n_rows, int after, int len) { return after < len && base + 32 <= n_rows; }

}  // namespace e2egrec
