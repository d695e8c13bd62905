// Enthalpy tiles around one another: which tiles a step's enthalpy kernels may
// touch, and how the near-tile pass finds its work.
//
// The next step's stream-collide pass takes the tiles away from the listed ones
// beside the solve and the commit, so that a "near" tile is one that holds a
// node of a listed tile's region (the tile and RH nodes around it).  Those are
// the tile and its eight neighbours, with one exception: on a periodic axis whose
// last tile is narrower than RH, a region reaches through that tile into the one
// beyond it (and the narrow tile's own region, TE + 2 RH nodes wide like every
// other, wraps through tile 0 into tile 1).
//
// Templated on the lattice's description (Dev, or a host struct with the same
// members): nx, ny, etx, ety, per_x, per_y, seam, ntiles, egrid, flags, nearmap,
// list.  LBM_HD marks the functions for the host (the CPU tests) and the device.
#pragma once

#ifndef LBM_HD
#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif
#endif

namespace lbm {

constexpr int TX = 32;       // fused kernel tile (threads x)
constexpr int TY = 8;        // fused kernel tile (threads y)
constexpr int TE = 32;       // enthalpy tile edge
constexpr int RH = 8;        // enthalpy halo width
constexpr int RE = TE + 2 * RH;
constexpr int COUNT_TILES = 1152;   // up to this many tiles the solve counts the listed ones itself

// bit 0 / 1: the x / y axis is periodic and its last tile is narrower than RH
// (with up to three tiles an axis, all are neighbours already)
LBM_HD int seam_axes(int nx, int ny, int per_x, int per_y) {
  const bool sx = per_x && nx > 3 * TE && nx % TE != 0 && nx % TE < RH;
  const bool sy = per_y && ny > 3 * TE && ny % TE != 0 && ny % TE < RH;
  return (sx ? 1 : 0) | (sy ? 2 : 0);
}

// Places around a tile: 0..8 the 3 x 3 tiles row by row (4 the tile itself), and
// with a seam 9..15 those across it: (across x, rows -1 0 1), (columns -1 0 1,
// across y), (across both).
// tile a's counterpart across the narrow last one of `tiles` on an axis, or -1
LBM_HD int tile_across(int a, int tiles) {
  return a == 0 ? tiles - 2 : a == tiles - 2 ? 0 : a == 1 ? tiles - 1 : a == tiles - 1 ? 1 : -1;
}
LBM_HD int tile_beside(int a, int o, int tiles, int per) {
  a += o;
  if (per) a = a < 0 ? tiles - 1 : a >= tiles ? 0 : a;
  return a >= 0 && a < tiles ? a : -1;
}
// the tile at place k of tile t, or -1
template <typename D>
LBM_HD int near_place(const D& d, int t, int k) {
  const int ty = t / d.etx, tx = t - ty * d.etx;
  const bool ax = k >= 9 && (k < 12 || k == 15), ay = k >= 12;
  const int ox = k < 9 ? k % 3 - 1 : k - 13, oy = k < 9 ? k / 3 - 1 : k - 10;
  const int xx = !ax ? tile_beside(tx, ox, d.etx, d.per_x)
                     : d.seam & 1 ? tile_across(tx, d.etx) : -1;
  const int yy = !ay ? tile_beside(ty, oy, d.ety, d.per_y)
                     : d.seam & 2 ? tile_across(ty, d.ety) : -1;
  return xx < 0 || yy < 0 ? -1 : yy * d.etx + xx;
}

// Was the tile at place k of tile t listed in the step of parity par with this
// stamp?  (places 0..8; all)
template <typename D>
LBM_HD bool listed_beside(const D& d, int t, int k, int par, int stamp) {
  const int ty = t / d.etx, tx = t - ty * d.etx;
  int xx = tx + k % 3 - 1, yy = ty + k / 3 - 1;
  if (d.per_x) xx = xx < 0 ? d.etx - 1 : xx >= d.etx ? 0 : xx;
  if (d.per_y) yy = yy < 0 ? d.ety - 1 : yy >= d.ety ? 0 : yy;
  if (xx < 0 || xx >= d.etx || yy < 0 || yy >= d.ety) return false;
  return d.flags[par * d.ntiles + yy * d.etx + xx] == stamp;
}
template <typename D>
LBM_HD bool listed_at(const D& d, int t, int k, int par, int stamp) {
  const int o = near_place(d, t, k);
  return o >= 0 && d.flags[par * d.ntiles + o] == stamp;
}
// Is tile t near, i.e. was a tile around it listed?  Places 0..8 are nine
// independent loads on a small lattice, where they wait once, and one on a large
// one, whose CTAs are many (2048^2: nine took 3% of the step) and whose marks keep a
// map of it.  (A lattice with tensor maps is walled: no seam.)
template <typename D>
LBM_HD bool near_beside(const D& d, int t, int par, int stamp) {
  if (d.ntiles > COUNT_TILES) return d.nearmap[par * d.ntiles + t] == stamp;
  bool hit = false;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int k = 0; k < 9; ++k) hit |= listed_beside(d, t, k, par, stamp);
  return hit;
}
template <typename D>
LBM_HD bool near_listed(const D& d, int t, int par, int stamp) {
  bool hit = near_beside(d, t, par, stamp);
  if (d.seam)
    for (int k = 9; k < 16; ++k) hit |= listed_at(d, t, k, par, stamp);
  return hit;
}

// Near-tile pass of a lattice whose step keeps a list (more tiles than CTAs in
// the solve): its work is found from the list, not by asking every tile.  Unit u
// of 36 a listed tile: one of the nine tiles around it and four 32x8 parts of
// that, taken by the first listed tile (row by row) among the nine around it.
// cnt: listed tiles of the step of parity par with this stamp.  (px, py): the
// part's first node; k: the place it was reached by (taken if 8 - k is the first
// place of t that is listed).  Lattices without a seam only.
template <typename D>
LBM_HD bool near_from_list(const D& d) {
  return d.ntiles > d.egrid;
}
// The ordinary-load pass, one 32x8 tile per CTA, asks every tile as long as there
// are few: at 768 x 640 (1920 of them) it ends 3 us sooner so.  With a seam, too.
template <typename D>
LBM_HD bool near_from_list_step(const D& d) {
  return near_from_list(d) && !d.seam &&
         (long long)((d.nx + TX - 1) / TX) * ((d.ny + TY - 1) / TY) > 8 * d.egrid;
}
template <typename D>
LBM_HD bool near_tile(const D& d, int u, int cnt, int par, int& t, int& k, int& px, int& py) {
  if (u >= 36 * cnt) return false;
  const int li = u / 36, r = u - 36 * li;
  k = r >> 2;
  const int l = d.list[par * d.ntiles + li];
  const int ly = l / d.etx, lx = l - ly * d.etx;
  int xx = lx + k % 3 - 1, yy = ly + k / 3 - 1;
  if (d.per_x) xx = xx < 0 ? d.etx - 1 : xx >= d.etx ? 0 : xx;
  if (d.per_y) yy = yy < 0 ? d.ety - 1 : yy >= d.ety ? 0 : yy;
  if (xx < 0 || xx >= d.etx || yy < 0 || yy >= d.ety) return false;
  t = yy * d.etx + xx;
  px = xx * TE;
  py = yy * TE + 8 * (r & 3);
  return py < d.ny;
}

}  // namespace lbm
