// A ghost row's interpolation sum, shared by the solvers' ghost kernels.
#pragma once

#include <cuda_runtime.h>

#include "ibm_internal.cuh"

namespace ibm {

// One row's eight sources (-1: none) and weights, loaded in 16-byte pieces before anything depends on
// them.  The rows are independent gathers, bound by latency: sources, then their values, are two
// round trips when each set of eight is issued at once (a loop that skips absent sources takes
// them one after another: 8.5 us for the 24,000 rows of an ellipsoid at 256^3, 5.3 us here, and 4.6 and 2.2 us at 64^3).
template <typename W>
struct GhostRow {
  long long q[8];
  W w[8];
  __device__ __forceinline__ GhostRow(const long long *src, const W *wt, long long g) {
    const longlong2 *s2 = reinterpret_cast<const longlong2 *>(src + 8 * g);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const longlong2 a = s2[c];
      q[2 * c] = a.x;
      q[2 * c + 1] = a.y;
    }
    if constexpr (sizeof(W) == 4) {
      const float4 *w4 = reinterpret_cast<const float4 *>(wt + 8 * g);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const float4 a = w4[c];
        w[4 * c] = a.x; w[4 * c + 1] = a.y; w[4 * c + 2] = a.z; w[4 * c + 3] = a.w;
      }
    } else {
      const double2 *w2 = reinterpret_cast<const double2 *>(wt + 8 * g);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double2 a = w2[c];
        w[2 * c] = a.x; w[2 * c + 1] = a.y;
      }
    }
  }
  // sum of w v over the sources in order, in T; value(q) reads a source (GHOST_CORNER set when it is
  // itself a ghost)
  template <typename T, class V>
  __device__ __forceinline__ T sum(V value) const {
    T v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = q[c] >= 0 ? value(q[c]) : (T)0;
    T s = (T)0;
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (q[c] >= 0) s += (T)w[c] * v[c];
    return s;
  }
};

}  // namespace ibm
