// Host form of the split step's tile arithmetic (lbm_tiles.cuh): near tiles cover
// whatever the enthalpy kernels touch, and the near pass's units cover the near
// tiles once.  Test infrastructure.
#include <stdlib.h>

#include <set>
#include <vector>

#include "lbm_tiles.cuh"

namespace {
struct Grid {
  int nx, ny, per_x, per_y, etx, ety, ntiles, seam, egrid;
  int *flags, *nearmap, *list;
};
int ffs0(unsigned v) { return v ? __builtin_ctz(v) : -1; }
int wrap(int v, int n, int per) {
  if (v >= 0 && v < n) return v;
  return per ? ((v % n) + n) % n : -1;
}
}  // namespace

// Lists `count` tiles (of the given seed; the whole row and column through one of
// them too when `cross` is set) of an nx x ny lattice.  Returns 0 or what failed:
// 1 a node of a listed tile's region in a tile not near, 2 near_listed
// differs, 3 a part of a near tile not taken once, or one of a far tile taken, by
// the near pass from the list (lattices without a seam).
extern "C" int near_tiles_check(int nx, int ny, int per_x, int per_y, int count, int cross,
                                int seed) {
  using namespace lbm;
  Grid g{nx, ny, per_x, per_y, (nx + TE - 1) / TE, (ny + TE - 1) / TE};
  g.ntiles = g.etx * g.ety;
  g.seam = seam_axes(nx, ny, per_x, per_y);
  g.egrid = 1;
  std::vector<int> flags(2 * g.ntiles, 0), map(2 * g.ntiles, 0), list(2 * g.ntiles, 0);
  g.flags = flags.data();
  g.nearmap = map.data();
  g.list = list.data();
  const int par = seed & 1, stamp = 7;
  srand(seed);
  std::set<int> listed;
  for (int i = 0; i < count; ++i) listed.insert((int)(rand() % g.ntiles));
  if (cross) {
    const int t = *listed.begin();
    for (int x = 0; x < g.etx; ++x) listed.insert(t / g.etx * g.etx + x);
    for (int y = 0; y < g.ety; ++y) listed.insert(y * g.etx + t % g.etx);
  }
  std::vector<int> order(listed.begin(), listed.end());
  for (size_t i = order.size(); i > 1; --i) std::swap(order[i - 1], order[rand() % i]);
  for (int t : order) {
    flags[par * g.ntiles + t] = stamp;
    for (int k = 0; k < 9; ++k)   // as mark_tile leaves it
      if (near_place(g, t, k) >= 0) map[par * g.ntiles + near_place(g, t, k)] = stamp;
  }
  for (size_t i = 0; i < order.size(); ++i) list[par * g.ntiles + i] = order[i];

  // near by asking the flags (near_listed takes the map above COUNT_TILES)
  const int places = g.seam ? 16 : 9;
  std::vector<char> nr(g.ntiles, 0);
  for (int t = 0; t < g.ntiles; ++t)
    for (int k = 0; k < places; ++k) {
      nr[t] |= listed_at(g, t, k, par, stamp);
      if (k < 9 && listed_at(g, t, k, par, stamp) != listed_beside(g, t, k, par, stamp)) return 2;
    }
  for (int t = 0; t < g.ntiles; ++t)
    if (nr[t] != near_listed(g, t, par, stamp) ||
        (!g.seam && nr[t] != near_beside(g, t, par, stamp)))
      return 2;

  for (int t : order) {
    const int X0 = t % g.etx * TE, Y0 = t / g.etx * TE;
    for (int ly = 0; ly < RE; ++ly)
      for (int lx = 0; lx < RE; ++lx) {
        const int x = wrap(X0 - RH + lx, nx, per_x), y = wrap(Y0 - RH + ly, ny, per_y);
        if (x >= 0 && y >= 0 && !nr[y / TE * g.etx + x / TE]) return 1;
      }
  }

  if (near_from_list_step(g) && g.seam) return 3;
  if (g.seam) return 0;
  std::vector<int> taken(4 * g.ntiles, 0);
  const int cnt = (int)order.size();
  for (int u = 0; u < 36 * cnt + 5; ++u) {
    int t, k, px, py;
    if (!near_tile(g, u, cnt, par, t, k, px, py)) continue;
    unsigned at = 0u;
    for (int j = 0; j < 9; ++j) at |= listed_beside(g, t, j, par, stamp) ? 1u << j : 0u;
    if (ffs0(at) != 8 - k) continue;
    if (px != t % g.etx * TE || py / TE != t / g.etx || py >= ny || py % TY) return 3;
    ++taken[4 * t + py % TE / TY];
  }
  for (int t = 0; t < g.ntiles; ++t)
    for (int r = 0; r < 4; ++r)
      if (taken[4 * t + r] != (nr[t] && t / g.etx * TE + TY * r < ny ? 1 : 0)) return 3;
  return 0;
}
