// rows2d.h - sizes and indices of the 2D solver's stacked vectors: K rows of nc cells, one per
// direction pair, and in the prediction the rho row after them.  Plain C++, so that the limits
// are checked on the host without a device.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define GRTE2_HD __host__ __device__
#else
#define GRTE2_HD
#endif

namespace grte2 {

// What creation accepts: the pairs' cell and vertex indices, up to K (nx+1)(ny+1), fit 32 bits.
// (The built-in set has 20 pairs.)
GRTE2_HD constexpr bool rows_fit(int64_t pairs, int64_t nx, int64_t ny) {
  return (pairs > 20 ? pairs : 20) * (nx + 1) * (ny + 1) < (int64_t)1 << 31;
}

// First index of the rho row.  The row ends at (K+1) nc, which passes 2^31 on grids that rows_fit
// accepts (20 pairs: from 10113 x 10113 cells), so this index and the sums from it have 64 bits.
GRTE2_HD constexpr int64_t rho_row(int64_t K, int64_t nc) { return K * nc; }

}  // namespace grte2
