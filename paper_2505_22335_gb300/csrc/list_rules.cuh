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

}  // namespace ups
