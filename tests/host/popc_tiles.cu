// Host check of the 2-way popcount kernel's tiles and launches.
//
// usage: popc_tiles SIDE n_v i_begin i_end
//   One line "first count I0 J0 I1 J1" per launch: its tiles and the tile
//   coordinates of its first and last one; then "in_range 0|1".
#include <cstdio>
#include <cstdlib>

#include "popc_tiles.cuh"

using namespace ccc;

int main(int argc, char **argv) {
  if (argc != 5) return 2;
  const long long side = std::atoll(argv[1]), n_v = std::atoll(argv[2]);
  const long long i0 = std::atoll(argv[3]), i1 = std::atoll(argv[4]);
  const PopcTri tri{(n_v + side - 1) / side};
  int64_t t0;
  const int64_t tiles = PopcTri::in_rows(n_v, i0, i1, side, &t0);
  popc_launches(t0, tiles, [&](int64_t first, int64_t count) {
    int64_t a, b, c, d;
    tri.coords(first, a, b);
    tri.coords(first + count - 1, c, d);
    std::printf("%lld %lld %lld %lld %lld %lld\n", static_cast<long long>(first),
                static_cast<long long>(count), static_cast<long long>(a), static_cast<long long>(b),
                static_cast<long long>(c), static_cast<long long>(d));
    return 0;
  });
  std::printf("in_range %d\n", popc_in_range(n_v, i0, i1) ? 1 : 0);
}
