// Layout changes between the host's cell-major state arrays ([row][direction], binary64) and
// the device's direction-major lines ([direction][row], binary64 or binary32), as 32 x 32
// tiles through shared memory so that both sides move full 128- or 256-byte rows.  The host
// arrays cross the bus as they are, into scratch that a step overwrites.
// Bound: the copy over the bus.  One 8192-cell, 32-angle instance (2.1 MB per array): on the
// host each array took a transposing loop over strided memory, a temporary of its size and,
// in mixed precision, a second one.  Setting six such instances from T alone: 2.76 -> 0.24 ms
// (E and O are filled on the device); a 512^2 2D state from T alone: 8 -> 1 ms.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace grte {

constexpr int kIoTile = 32, kIoRows = 8;   // blocks of 32 x 8 threads, 4 rows per thread

// dst[k*rows + i] = src[i*M + k] - ac U[i]   (U null: the value itself)
template <typename R>
__global__ void k_lines_in(const double* __restrict__ src, R* __restrict__ dst, int64_t rows, int M,
                           const double* __restrict__ U, double ac) {
  __shared__ double tile[kIoTile][kIoTile + 1];
  const int64_t i0 = (int64_t)blockIdx.x * kIoTile;
  const int k0 = blockIdx.y * kIoTile;
  for (int r = threadIdx.y; r < kIoTile; r += kIoRows) {
    const int64_t i = i0 + r;
    const int k = k0 + threadIdx.x;
    if (i < rows && k < M) tile[r][threadIdx.x] = src[i * M + k];
  }
  __syncthreads();
  const int64_t i = i0 + threadIdx.x;
  if (i >= rows) return;
  const double base = U ? ac * U[i] : 0.0;
  for (int r = threadIdx.y; r < kIoTile; r += kIoRows)
    if (k0 + r < M) dst[(int64_t)(k0 + r) * rows + i] = (R)(U ? tile[threadIdx.x][r] - base : tile[threadIdx.x][r]);
}

// dst[i*M + k] = ac U[i] + src[k*rows + i]   (U null: the value itself)
template <typename R>
__global__ void k_lines_out(const R* __restrict__ src, double* __restrict__ dst, int64_t rows, int M,
                            const double* __restrict__ U, double ac) {
  __shared__ double tile[kIoTile][kIoTile + 1];
  const int64_t i0 = (int64_t)blockIdx.x * kIoTile;
  const int k0 = blockIdx.y * kIoTile;
  {
    const int64_t i = i0 + threadIdx.x;
    const double base = U && i < rows ? ac * U[i] : 0.0;
    for (int r = threadIdx.y; r < kIoTile; r += kIoRows)
      if (i < rows && k0 + r < M) {
        const double v = (double)src[(int64_t)(k0 + r) * rows + i];
        tile[r][threadIdx.x] = U ? base + v : v;
      }
  }
  __syncthreads();
  for (int r = threadIdx.y; r < kIoTile; r += kIoRows) {
    const int64_t i = i0 + r;
    const int k = k0 + threadIdx.x;
    if (i < rows && k < M) dst[i * M + k] = tile[threadIdx.x][r];
  }
}

inline dim3 io_grid(int64_t rows, int M) {
  return dim3((unsigned)((rows + kIoTile - 1) / kIoTile), (unsigned)((M + kIoTile - 1) / kIoTile));
}
inline dim3 io_block() { return dim3(kIoTile, kIoRows); }

// U = T^4
static __global__ void k_fourth_power(const double* __restrict__ T, double* __restrict__ U, int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) U[i] = (T[i] * T[i]) * (T[i] * T[i]);
}

}  // namespace grte
