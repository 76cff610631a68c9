// What the tile-list kernels (bin.cu) may index and write, whatever the depth order
// holds: a wait that ran out in the order (sort.cu) leaves ids that are stale,
// repeated, another view's or no id at all.  Plain C++, so that the rules can be run
// on the host too.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define UPS_HD __host__ __device__ __forceinline__
#else
#define UPS_HD inline
#endif

namespace ups {

// Whether gv is one of view v's N Gaussian-views (v N + N <= 2^31).  An id that is not
// counts as a Gaussian without tiles: another view's would index this view's tiles by
// that view's columns and rows, and its Gaussian set past the end.
UPS_HD bool of_view(uint32_t gv, uint32_t v, uint32_t N) { return gv - v * N < N; }

// Next free position (and end) of a tile's list while a run of Gaussians is filled in; n:
// entries that the list buffer has room for.  An uncapped list has no end of its own: its
// positions come from counts that are taken again from an order that may repeat an id,
// or (for Gaussians whose rows are evaluated again) by another kernel than the one that
// sized the buffer, so every position is held against the buffer.
template <bool CAPPED> struct Slot;
template <> struct Slot<true> {
    uint32_t next, stop;  // stop <= n
    UPS_HD bool room() const { return next < stop; }
    UPS_HD bool fits(uint32_t pos, uint32_t) const { return pos < stop; }
};
template <> struct Slot<false> {
    uint32_t next;
    UPS_HD bool room() const { return true; }
    UPS_HD bool fits(uint32_t pos, uint32_t n) const { return pos < n; }
};

}  // namespace ups
