// Steps of the walks over segment offsets (device code; plain C++ for tests on the host).
#pragma once

#ifdef __CUDACC__
#define E2EGREC_HD __host__ __device__ __forceinline__
#else
#define E2EGREC_HD inline
#endif

namespace e2egrec {

constexpr int kQuietWindows = 4;

// First segment of the window of 32 that a walk looks at after the one that begins at `base`.  `quiet`: windows without an
// entry in a row; from the fourth on the walk asks find() where the next entry's segment is.  Never the same window again:
// offsets that decrease, which no entry point accepts but none can refuse, could make find() go back, and the walk ends
// nevertheless, after one window per 32 segments at most.
template <typename T, class Find> E2EGREC_HD T next_window(T base, int quiet, Find find)
{
    const T next = base + 32;
    if (quiet < kQuietWindows) return next;
    const T found = find();
    return found > next ? found : next;
}

}  // namespace e2egrec
