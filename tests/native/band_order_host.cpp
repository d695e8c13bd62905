// Host form of the adjoint band's colours and list (lbm_flow_adjoint.cuh).  Test
// infrastructure.
#include <stdlib.h>

#include <vector>

#include "lbm_flow_adjoint.cuh"

template <bool SEAM>
static int check(int nx, int ny, int per_y, int percent, int seed) {
  using namespace lbm;
  const int n = nx * ny, m = band_main(nx, ny, per_y);
  srand(seed);
  auto colour = [&](int s) { return band_colour(s % nx, s / nx, s, m); };
  for (int s = 0; s < n; ++s) {
    const int x = s % nx, y = s / nx;
    if (x + 1 < nx && colour(s) == colour(s + 1)) return 1;
    const int up = y + 1 < ny ? s + nx : per_y ? x : -1;
    if (up >= 0 && colour(s) == colour(up)) return 1;
  }
  std::vector<int> nodes;
  for (int s = 0; s < n; ++s)
    if (rand() % 100 < percent) nodes.push_back(s);
  for (size_t i = nodes.size(); i > 1; --i) std::swap(nodes[i - 1], nodes[rand() % i]);
  std::vector<int> list(n, -1), pos(n, -1), seen(n, 0);
  int count[4] = {0, 0, 0, 0};
  for (int s : nodes) band_append(list.data(), count, pos.data(), n, m, s, colour(s));
  const BandOrder<SEAM> o(count, n, m);
  if (o.e4 != (int)nodes.size()) return 3;
  for (int j = 0; j < o.e4; ++j) {
    const int at = o.entry(j);
    if (at < 0 || at >= n || list[at] < 0 || pos[list[at]] != at || o.order(at) != j) return 2;
    const int c = j < o.e1 ? 0 : j < o.e2 ? 1 : j < o.e3 ? 2 : 3;
    if (colour(list[at]) != c || seen[list[at]]++) return 3;
  }
  return 0;
}

// A random band (every node with probability percent / 100) of an nx x ny lattice,
// listed in random order.  Returns 0, or what failed: 1 neighbours of one colour, 2
// the list's places and the band's order not inverse, 3 a node missing or out of
// its colour's range.
extern "C" int band_order_check(int nx, int ny, int per_y, int percent, int seed) {
  return lbm::band_main(nx, ny, per_y) < nx * ny ? check<true>(nx, ny, per_y, percent, seed)
                                                 : check<false>(nx, ny, per_y, percent, seed);
}
