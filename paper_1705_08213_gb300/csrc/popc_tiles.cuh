// Tiles of the 2-way popcount kernel and their launches.  Host-callable, so
// that they can be checked without a GPU.
#pragma once

#include <math.h>
#include <stdint.h>

namespace ccc {
namespace {

// Row-major upper triangle, with its diagonal, of nB x nB tiles: row I holds
// the nB - I tiles J >= I.
struct PopcTri {
  int64_t nB;
  // Tiles before a row.
  __host__ __device__ int64_t start(int64_t row) const { return row * nB - row * (row - 1) / 2; }
  __host__ __device__ void coords(int64_t t, int64_t &I, int64_t &J) const {
    const double b = 2.0 * static_cast<double>(nB) + 1.0;
    int64_t r = static_cast<int64_t>((b - sqrt(b * b - 8.0 * static_cast<double>(t))) * 0.5);
    if (r < 0) r = 0;
    if (r >= nB) r = nB - 1;
    while (r > 0 && start(r) > t) --r;
    while (r + 1 < nB && start(r + 1) <= t) ++r;
    I = r;
    J = r + (t - start(r));
  }
  // Tiles in the row blocks that SNPs [i_begin, i_end) of n_v fall in.
  static int64_t in_rows(int64_t n_v, int64_t i_begin, int64_t i_end, int64_t side, int64_t *first) {
    const PopcTri tri{(n_v + side - 1) / side};
    const int64_t B0 = (i_begin > 0 ? i_begin : 0) / side;
    const int64_t B1 = i_end < n_v ? (i_end + side - 1) / side : tri.nB;
    *first = tri.start(B0);
    return tri.start(B1) - *first;
  }
};

// A grid holds at most 2^31 - 1 blocks: `tiles` tiles from t0 on, in as few
// launches(first tile, tiles) as that takes; stops at the first that fails.
template <class Launch>
inline int popc_launches(int64_t t0, int64_t tiles, Launch launch) {
  constexpr int64_t kMaxGrid = 0x7fffffff;
  int rc = 0;
  for (int64_t t = 0; t < tiles && rc == 0; t += kMaxGrid)
    rc = launch(t0 + t, tiles - t < kMaxGrid ? tiles - t : kMaxGrid);
  return rc;
}

// Calls that are taken: at most 2^31 - 1 tiles of 64 x 64 SNPs (4,194,240 SNPs
// for the whole triangle; minutes of work), whatever the kernel's own tile.
inline bool popc_in_range(int64_t n_v, int64_t i_begin, int64_t i_end) {
  int64_t first;
  return PopcTri::in_rows(n_v, i_begin, i_end, 64, &first) <= 0x7fffffff;
}

}  // namespace
}  // namespace ccc
