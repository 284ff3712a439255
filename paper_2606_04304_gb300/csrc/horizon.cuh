// The in-horizon pixels of an N x N image, l^2 + m^2 < 1, row by row: in every row
// they are one run of columns, so a plan needs N pairs of numbers instead of a
// test and a list entry per pixel (0.2 ms at 256^2, 60 us a drift search of eight epochs),
// and the device expands its own list.
#pragma once

#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace ovro {

struct Horizon {
  int n = 0;
  std::vector<int> start;      // [n + 1] list index of each row's first pixel
  std::vector<int> col;        // [n] its column

  Horizon() = default;
  // l = (c - N/2) cell; l^2 + m^2 in FP64 is monotone in |c - N/2|, so the last
  // column inside is found from an estimate by the test itself.
  Horizon(int size, double cell) : n(size), start(size + 1, 0), col(size, 0) {
    const int half = n / 2;
    for (int r = 0; r < n; ++r) {
      const double m = static_cast<double>(r - half) * cell;
      auto inside = [&](int k) {
        const double l = static_cast<double>(k) * cell;
        return l * l + m * m < 1.0;
      };
      const double est = std::sqrt(std::max(0.0, 1.0 - m * m)) / std::fabs(cell);
      int k = est < half ? static_cast<int>(est) : half;
      while (k < half && inside(k + 1)) ++k;
      while (k >= 0 && !inside(k)) --k;
      col[r] = half - std::min(k, half);
      start[r + 1] = start[r] + (k < 0 ? 0 : std::min(k, half) + 1 + std::min(k, n - 1 - half));
    }
  }
  int size() const { return n ? start[n] : 0; }
  // image index of the p-th pixel
  int pixel(int p) const {
    const int r = static_cast<int>(std::upper_bound(start.begin(), start.end(), p) - start.begin()) - 1;
    return r * n + col[r] + (p - start[r]);
  }
};

// One CTA per image row; rows: start [n + 1], then col [n].
static __global__ void k_horizon(const int* __restrict__ rows, int n, int* __restrict__ pix) {
  const int r = blockIdx.x, s0 = rows[r], s1 = rows[r + 1], c0 = rows[n + 1 + r];
  for (int i = threadIdx.x; i < s1 - s0; i += blockDim.x) pix[s0 + i] = r * n + c0 + i;
}

// The list on the device; d_rows: 2 n + 1 ints of scratch (a copy from pageable
// memory is staged before the call returns).
inline int upload_horizon(const Horizon& h, int* d_rows, int* d_pix, cudaStream_t st) {
  std::vector<int> rows(h.start);
  rows.insert(rows.end(), h.col.begin(), h.col.end());
  OVRO_CUDA_TRY(cudaMemcpyAsync(d_rows, rows.data(), rows.size() * sizeof(int), cudaMemcpyHostToDevice, st));
  k_horizon<<<h.n, 128, 0, st>>>(d_rows, h.n, d_pix);
  OVRO_LAUNCH_CHECK();
  return OVRO_OK;
}

}  // namespace ovro
