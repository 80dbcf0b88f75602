// What the FP64 1D1V moment passes and their reverse mode share: the gather
// coefficients of the nodes and the markers of a block.
#pragma once

#include <cuda_runtime.h>

#include "pic_internal.cuh"

namespace pic {
namespace {

constexpr int kMomMaxNodes = 1792;        // tables and one tile (64 bytes a node at order 2) leave
                                          // room for two blocks on an SM up to 1760 nodes

// The end of this block's run of markers.
__device__ __forceinline__ int64_t chunk_end(const Es1dConst &c) {
  const int64_t e = (blockIdx.x + 1) * c.chunk;
  return e < c.n_total ? e : c.n_total;
}

// Coefficients of a node: order 1 {a, b}; order 2 {a, b} and c, 4 words a node.
template <int ORDER>
struct Poly {
  static constexpr int kWords = ORDER == 1 ? 2 : 4;
};

// table <- the coefficients of F (nc values in shared memory)
template <int ORDER>
__device__ __forceinline__ void build_poly(double *table, const double *F, int nc) {
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    const double fp = F[i + 1 == nc ? 0 : i + 1], f0 = F[i];
    if (ORDER == 1) {
      *(double2 *)(table + 2 * i) = make_double2(f0, fp - f0);
    } else {
      const double fm = F[i == 0 ? nc - 1 : i - 1];
      const double cc = fma(0.5, fm + fp, -f0);
      *(double2 *)(table + 4 * i) = make_double2(fma(0.25, cc, f0), 0.5 * (fp - fm));
      table[4 * i + 2] = cc;
    }
  }
}

template <int ORDER>
__device__ __forceinline__ double gather_poly(const double *table, int i, double d) {
  const double2 ab = *(const double2 *)(table + Poly<ORDER>::kWords * i);
  if (ORDER == 1) return __fma_rn(ab.y, d, ab.x);
  return __fma_rn(__fma_rn(table[4 * i + 2], d, ab.y), d, ab.x);
}

__device__ __forceinline__ void clear_doubles(double *a, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) a[i] = 0.0;
}

}  // namespace
}  // namespace pic
