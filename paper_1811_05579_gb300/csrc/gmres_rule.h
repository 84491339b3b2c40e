// gmres_rule.h - how the FP64/mixed Krylov kernels of the 1D path (k_gmres) share an instance: slices,
// the shared memory of the largest slice, and the cluster size.  Plain C++, so that the rule is
// checked on the host without a device.
#pragma once
#include <algorithm>
#include <cstdint>

#ifdef __CUDACC__
#define GRTE_HD __host__ __device__
#else
#define GRTE_HD
#endif

namespace grte {

constexpr int kTriThreads = 256;   // threads per CTA of the preconditioner slices
// padded length of a shared-memory x of n values
GRTE_HD inline int64_t tri_xs_len(int64_t n) { return n + (n >> 5) + 1; }

constexpr int kCL = 8, kCLMax = 16;

// CTAs that share the N cells of one instance: a lone one up to a cell per thread, above
// that the whole cluster.  The work on a slice is a chain of short dependent steps, so a
// CTA takes hardly longer for 128 cells than for 16, and a lone slice needs no cluster
// barrier, no spikes and no interface system: all Krylov kernels of a 128-cell step took
// 190 us over 8 slices, 184 over 2 and 165 in one; at 1000 cells 132 us over 8 slices
// and 137 over 4.
constexpr int kLoneCells = kTriThreads;
GRTE_HD inline int slice_count(int64_t N, int ncl) { return N <= kLoneCells ? 1 : ncl; }

// Cells of the largest slice of a handle's instances (at most one too many).
inline int64_t largest_slice(const int64_t* nx, int n_inst, int ncl) {
  int64_t s = 0;
  for (int i = 0; i < n_inst; ++i) s = std::max<int64_t>(s, nx[i] / slice_count(nx[i], ncl) + 1);
  return s;
}
// Dynamic shared memory of the kernels for such slices: the slice's unknowns, or none where they
// pass the limit and stay in global memory.
inline int64_t gmres_dyn_bytes(int64_t slice, int64_t limit) {
  const int64_t b = (tri_xs_len(slice) * 8 + 15) / 16 * 16;
  return b <= limit ? b : 0;
}

// Cluster size of the Krylov kernels.  Sixteen CTAs halve the binary64 work per SM, which
// bounds a large FP64 instance: us per kernel with 8 / 16 CTAs, 32 angles, 55.9 / 43.9 at 8192
// cells, 40.3 / 33.4 at 4096, 29.7 / 28.8 at 2048, 28.8 / 30.6 at 1500, 26.6 / 28.7 at 1000.  But
// they fill a GPC, so seven such clusters fit at a time: 12 runs of 2048 cells take 29.4 / 30.5.
// resident(dyn): whether a cluster of sixteen with dyn bytes of dynamic shared memory per CTA,
// what the launches will ask for, can be resident; beyond the portable size that is not given.
constexpr int64_t kWideCells = 2048;
constexpr int kWideInst = 7;
template <class Resident>
int gmres_cluster(const int64_t* nx, int n_inst, bool mixed, int64_t limit, Resident resident) {
  if (mixed || n_inst > kWideInst || *std::max_element(nx, nx + n_inst) < kWideCells) return kCL;
  return resident(gmres_dyn_bytes(largest_slice(nx, n_inst, kCLMax), limit)) ? kCLMax : kCL;
}

}  // namespace grte
