// Steps of the walks over segment offsets (device code; plain C++ for tests on the host).
#pragma once

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

}  // namespace e2egrec
