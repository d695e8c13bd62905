// Utility kernels: initial equilibria, macroscopic outputs, FP64 reductions,
// checkpoint gather/scatter and input validation.
#include "lbm_adjoint.cuh"

namespace lbm {

// ---- population gathers for any node, any layout --------------------------

__device__ __forceinline__ bool flow_active(const Dev& d, int x, int y) {
  if (is_wall(d, x, y)) {
    if (!d.flow_walls) return false;
    int ix, iy;   // an extrapolated wall node carries flow with its inward node
    inward_of(d, x, y, ix, iy);
    return d.fl[(long long)iy * d.nx + ix] >= d.f_act;
  }
  return d.fl[(long long)y * d.nx + x] >= d.f_act;
}

// g_i of non-wall node (x, y) in the given layout
__device__ __forceinline__ void gather_g(const Dev& d, int x, int y, int layout, float g[5]) {
  const long long n = d.n, s = (long long)y * d.nx + x;
  (void)n;
  g[0] = ld_g(d, 0, s);
  for (int i = 1; i < 5; ++i) {
    if (layout == 0) {
      g[i] = ld_g(d, i, s);
    } else {
      const int sx = wrapx(d, x - ex9(i)), sy = wrapy(d, y - ey9(i));
      g[i] = ld_g(d, opp5(i), (long long)sy * d.nx + sx);
    }
  }
}

// f_i of node (x, y): nodes without flow hold theirs in their own slots
__device__ __forceinline__ void gather_f(const Dev& d, int x, int y, int layout, float f[9]) {
  const long long n = d.n, s = (long long)y * d.nx + x;
  const bool self = flow_active(d, x, y);
  (void)n;
  f[0] = ld_f(d, 0, s);
  for (int i = 1; i < 9; ++i) {
    if (layout == 0 || !self) {
      f[i] = ld_f(d, i, s);
    } else {
      const int sx = wrapx(d, x - ex9(i)), sy = wrapy(d, y - ey9(i));
      if (flow_active(d, sx, sy)) f[i] = ld_f(d, opp9(i), (long long)sy * d.nx + sx);
      else f[i] = ld_f(d, i, s);
    }
  }
}

__device__ float node_T(const Dev& d, int x, int y, int layout);

// temperature of a non-wall node
__device__ __forceinline__ float interior_T(const Dev& d, int x, int y, int layout) {
  float g[5];
  gather_g(d, x, y, layout, g);
  return g[0] + g[1] + g[2] + g[3] + g[4];
}

// temperature of any node; wall nodes report the temperature their wall
// imposes (Dirichlet value, or the inward neighbour's for an adiabatic wall;
// a corner follows its vertical wall, then its horizontal wall's Dirichlet
// value, then its diagonal neighbour)
__device__ float node_T(const Dev& d, int x, int y, int layout) {
  if (!is_wall(d, x, y)) return interior_T(d, x, y, layout);
  int side;
  if (d.wall_l && x == 0) side = 0;
  else if (d.wall_r && x == d.nx - 1) side = 1;
  else if (d.wall_b && y == 0) side = 2;
  else side = 3;
  if (d.bc[side] == 1) return side == 0 ? d.wallTl[y] : d.Tbc[side];
  const bool vx = (d.wall_l || d.wall_r) && (x == 0 || x == d.nx - 1);
  const bool vy = (d.wall_b || d.wall_t) && (y == 0 || y == d.ny - 1);
  if (vx && vy) {
    const int hs = (y == 0) ? 2 : 3;
    if (d.bc[hs] == 1) return d.Tbc[hs];
    return interior_T(d, x == 0 ? 1 : d.nx - 2, y == 0 ? 1 : d.ny - 2, layout);
  }
  switch (side) {
    case 0: return interior_T(d, 1, y, layout);
    case 1: return interior_T(d, d.nx - 2, y, layout);
    case 2: return interior_T(d, x, 1, layout);
    default: return interior_T(d, x, d.ny - 2, layout);
  }
}

// ---- kernels ----------------------------------------------------------------

// Loading fields, one CTA per enthalpy tile: the material fields and f_l copied,
// the populations at their rest equilibria, the left wall's profile from the
// side's value when wallTl (the profile, if it is to be set) is not null, the
// tile's activity, and no stamps, lists or sentinel left.  One pass in place of
// three copies, three clears and two kernels (48^2: lbm_set_fields 75 -> 58 us).
template <typename S>
__global__ void __launch_bounds__(256) load_fields_kernel(Dev d, const float* phi, const float* K,
                                                          const float* T0, const float* fl0,
                                                          float* wallTl) {
  const int tile = blockIdx.x, tid = threadIdx.x, n = (int)d.n;
  const int X0 = (tile % d.etx) * TE, Y0 = (tile / d.etx) * TE;
  S* F = static_cast<S*>(d.f);
  int any = 0;
#pragma unroll
  for (int j = 0; j < TE * TE / 256; ++j) {
    const int x = X0 + tid % TE, y = Y0 + tid / TE + j * (256 / TE);
    if (x >= d.nx || y >= d.ny) continue;
    const int s = y * d.nx + x;
    const float T = T0[s], fl = fl0[s];
    const_cast<float*>(d.phi)[s] = phi[s];
    const_cast<float*>(d.K)[s] = K[s];
    d.fl[s] = fl;
    // f^eq(rho0, u = 0) = w_i rho0, Eq. (29); stored as the deviation f - w_i rho0 = 0
#pragma unroll
    for (int i = 0; i < 9; ++i) Pop<S>::st(F + i * n + s, 0.f);
    // g^eq(T0, u = 0), Eq. (39): w~_i T0
#pragma unroll
    for (int i = 0; i < 5; ++i) st_g(d, i, s, (i == 0 ? d.wt0 : d.wt1) * T);
    any |= !is_wall(d, x, y) && fl >= d.f_act;
  }
  any = __syncthreads_or(any);
  if (tid == 0) d.tact[tile] = (unsigned char)(any ? 1 : 0);
  if (tid < 5) d.flags[tid * d.ntiles + tile] = 0;   // flags, near map and status words
  if (tile == 0 && tid < 4) d.lcount[tid] = 0;
  if (tile == 0 && tid == 4) d.stats[5] = 0;
  if (wallTl && X0 == 0 && tid < TE && Y0 + tid < d.ny) wallTl[Y0 + tid] = d.Tbc[0];
}

// Macroscopic fields.  Bound by its loads and stores (f, g, f_l, phi, K in,
// five fields out: 88 bytes a node); every load of a lattice node is issued
// before any value is chosen, the populations of both candidate slots of each
// link included (they lie in lines the neighbours read anyway), so that a node
// waits for memory once instead of once per link (2048^2: 107 -> 72 us).
template <typename S>
__global__ void __launch_bounds__(256) macros_kernel(Dev d, int layout, float* ux, float* uy,
                                                     float* rho, float* T, float* fl) {
  const int n = (int)d.n, nx = d.nx;
  const int s = blockIdx.x * 256 + threadIdx.x;
  if (s >= n) return;
  const int y = s / nx, x = s - y * nx;
  const S* F = static_cast<const S*>(d.f);
  const S* G = static_cast<const S*>(d.g);
  const bool wall = is_wall(d, x, y);
  const float fls = d.fl[s];
  float f[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = Pop<S>::ld(F + i * n + s);
  float Tn, vx = 0.f, vy = 0.f;
  if (wall) {
    Tn = node_T(d, x, y, layout);
  } else {
    const float r0 = std::is_same<S, float>::value ? 0.f : d.wt0 * d.g_ref;
    const float r1 = std::is_same<S, float>::value ? 0.f : d.wt1 * d.g_ref;
    const float phi = d.phi[s], K = d.K[s];
    float g[5];
    g[0] = Pop<S>::ld(G + s) + r0;
    if (layout == 0) {
#pragma unroll
      for (int i = 1; i < 5; ++i) g[i] = Pop<S>::ld(G + i * n + s) + r1;
    } else {
      const int cx[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
      const int cy[3] = {y == 0 ? d.ny - 1 : y - 1, y, y == d.ny - 1 ? 0 : y + 1};
      float str[9], fln[9];
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        const int t = cy[1 - ey9(i)] * nx + cx[1 - ex9(i)];   // x - e_i
        fln[i] = d.fl[t];
        str[i] = Pop<S>::ld(F + opp9(i) * n + t);
        if (i < 5) g[i] = Pop<S>::ld(G + opp5(i) * n + t) + r1;
      }
      if (fls >= d.f_act) {
#pragma unroll
        for (int i = 1; i < 9; ++i) {
          const int sx = cx[1 - ex9(i)], sy = cy[1 - ey9(i)];
          const bool act = is_wall(d, sx, sy) ? d.flow_walls && flow_active(d, sx, sy)
                                              : fln[i] >= d.f_act;
          if (act) f[i] = str[i];
        }
      }
    }
    Tn = g[0] + g[1] + g[2] + g[3] + g[4];
    if (d.flow && fls >= d.f_act) {   // a wall's velocity is the wall's, 0
      const float jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8];
      const float jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8];
      float Fx, Fy;
      velocity(jx, jy, Tn, fls, phi, K, d, vx, vy, Fx, Fy);
    }
  }
  float dr = 0.f;
#pragma unroll
  for (int i = 0; i < 9; ++i) dr += f[i];
  if (ux) ux[s] = vx;
  if (uy) uy[s] = vy;
  if (rho) rho[s] = d.rho0 + dr;   // stored populations are f_i - w_i rho0
  if (T) T[s] = Tn;
  if (fl) fl[s] = fls;
}

// lo += what hi + v loses in FP32 (Knuth's two-sum), hi = hi + v: hi + lo stays
// the exact sum to about 2^-48 of it
__device__ __forceinline__ void two_sum(float& hi, float& lo, float v) {
  const float s = hi + v, t = s - hi;
  lo += (hi - (s - t)) + (v - t);
  hi = s;
}

// per-block FP64 partial sums in a fixed order:
// [0] mass, [1] enthalpy, [2] sum f_l, [3] non-wall count, [4] Nusselt sum, [5] Nusselt rows
//
// Bound by the FP64 pipe (two lanes a clock on an SM), conversions from FP32
// included, not by the 68 bytes it reads per node: so each node makes eight
// FP64 operations where a plain FP64 sum of everything makes about 35.  The
// nine deviations add up in FP32 pairs (two_sum), rho0 is counted and
// multiplied once, f_l = 0 and 1 are counted, phi f_l is an exact FP32 pair and
// dT / (sigma St) multiplies the sum.  (2048^2, FP32: 336 -> 121 us.)
//
// The mass needs no gather: in the AA layout every slot of a lattice node is
// read by exactly one lattice node (its own, or the neighbour the population
// streams to), so the nodes' own slots hold the sum in both layouts.  Only flow
// walls, whose nodes hold and read populations of lattice nodes, need it.
template <typename S>
__global__ void __launch_bounds__(RB) reduce_kernel(Dev d, int layout, double* partials) {
  __shared__ double sh[6][RB];
  const int tid = threadIdx.x;
  const int n = (int)d.n, nx = d.nx;
  const S* F = static_cast<const S*>(d.f);
  const S* G = static_cast<const S*>(d.g);
  const float r0 = std::is_same<S, float>::value ? 0.f : d.wt0 * d.g_ref;
  const float r1 = std::is_same<S, float>::value ? 0.f : d.wt1 * d.g_ref;
  const bool gather = layout == 1 && d.flow && d.flow_walls;
  double mass = 0, heat = 0, latent = 0, liquid = 0;
  int count = 0, ones = 0;   // non-wall nodes, those with f_l = 1
  for (int s = blockIdx.x * RB + tid; s < n; s += gridDim.x * RB) {
    const int y = s / nx, x = s - y * nx;
    if (is_wall(d, x, y)) continue;
    float f[9], g[5];
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = Pop<S>::ld(F + i * n + s);
    g[0] = Pop<S>::ld(G + s) + r0;
    if (layout == 0) {
#pragma unroll
      for (int i = 1; i < 5; ++i) g[i] = Pop<S>::ld(G + i * n + s) + r1;
    } else {
      const int xm = x == 0 ? s + nx - 1 : s - 1, xp = x == nx - 1 ? s - x : s + 1;
      const int ym = y == 0 ? n - nx + x : s - nx, yp = y == d.ny - 1 ? x : s + nx;
      g[1] = Pop<S>::ld(G + 3 * n + xm) + r1;
      g[2] = Pop<S>::ld(G + 4 * n + ym) + r1;
      g[3] = Pop<S>::ld(G + n + xp) + r1;
      g[4] = Pop<S>::ld(G + 2 * n + yp) + r1;
    }
    const float fl = d.fl[s], phi = d.phi[s];
    if (gather) gather_f(d, x, y, layout, f);
    float hi = f[0], lo = 0.f;
#pragma unroll
    for (int i = 1; i < 9; ++i) two_sum(hi, lo, f[i]);
    if (fabsf(hi) <= 1e37f) {
      mass += (double)hi;
      mass += (double)lo;
    } else {   // NaN, Inf, or out of FP32's range on the way
      for (int i = 0; i < 9; ++i) mass += (double)f[i];
    }
    heat += (double)(g[0] + g[1] + g[2] + g[3] + g[4]);
    ++count;
    // a = phi dT / (sigma(f_l) St), Eq. (38) with Eq. (7)
    if (d.sigma_var) {
      const double fd = (double)fl;
      latent += (double)phi * fd * (double)d.sigma /
                ((double)d.sigma_s + fd * ((double)d.sigma - d.sigma_s));
      liquid += fd;
    } else if (fl == 1.f) {
      latent += (double)phi;
      ++ones;
    } else if (fl != 0.f) {
      const float p = phi * fl;
      latent += (double)p;
      latent += (double)fmaf(phi, fl, -p);
      liquid += (double)fl;
    }
  }
  // the left wall's rows, spread over the grid
  double nu = 0, rows = 0;
  if (d.wall_l && nx >= 3)
    for (int y = blockIdx.x * RB + tid; y < d.ny; y += gridDim.x * RB) {
      if (d.wall_b && (y == 0 || y == d.ny - 1)) continue;
      const double T0 = node_T(d, 0, y, layout), T1 = node_T(d, 1, y, layout),
                   T2 = node_T(d, 2, y, layout);
      nu += -(-3.0 * T0 + 4.0 * T1 - T2) * 0.5 * (double)d.H_over_dT;
      rows += 1.0;
    }
  const double acc[6] = {(double)d.rho0 * count + mass, heat + (double)d.lat * latent,
                         liquid + (double)ones, (double)count, nu, rows};
  for (int k = 0; k < 6; ++k) sh[k][tid] = acc[k];
  __syncthreads();
  for (int w = RB / 2; w > 0; w >>= 1) {
    if (tid < w)
      for (int k = 0; k < 6; ++k) sh[k][tid] += sh[k][tid + w];
    __syncthreads();
  }
  if (tid < 6) partials[blockIdx.x * 6 + tid] = sh[tid][0];
}

// Does this part of a split read-out (mode 0 all, 1 tiles away from the front,
// 2 tiles near it, by the step of parity par just taken) take tile t?  (SEAM: on a
// lattice with one)
template <bool SEAM>
__device__ __forceinline__ bool takes_part(const Dev& d, int mode, int par, int t) {
  return mode == 0 || (mode == 2) == (SEAM ? near_listed(d, t, par, d.ctr[par])
                                           : near_beside(d, t, par, d.ctr[par]));
}

// The left-wall Nusselt number of the current state (the rows and the
// formula of reduce_kernel), added to acc[0]; one block, fixed summation order.
// Mode 1 leaves its rows' terms in rows[], where mode 2 finds them.
template <bool SEAM>
__global__ void __launch_bounds__(RB) wall_nusselt_kernel(Dev d, int layout, int mode, int par,
                                                          double* rows, double* acc) {
  __shared__ double sh[RB];
  const int tid = threadIdx.x;
  const int y0 = d.wall_b ? 1 : 0, y1 = d.wall_t ? d.ny - 1 : d.ny;
  double v = 0.0;
  if (d.wall_l && d.nx >= 3)
    for (int y = y0 + tid; y < y1; y += RB) {
      double r;
      if (takes_part<SEAM>(d, mode, par, (y / TE) * d.etx)) {
        const double T0 = node_T(d, 0, y, layout), T1 = node_T(d, 1, y, layout),
                     T2 = node_T(d, 2, y, layout);
        r = -(-3.0 * T0 + 4.0 * T1 - T2) * 0.5 * (double)d.H_over_dT;
        if (mode == 1) rows[y] = r;
      } else {
        r = mode == 2 ? rows[y] : 0.0;
      }
      v += r;
    }
  if (mode == 1) return;
  sh[tid] = v;
  __syncthreads();
  for (int w = RB / 2; w > 0; w >>= 1) {
    if (tid < w) sh[tid] += sh[tid + w];
    __syncthreads();
  }
  if (tid == 0 && d.wall_l && d.nx >= 3 && y1 > y0) acc[0] += sh[0] / (double)(y1 - y0);
}

// The partial sums of all blocks, in a fixed order: each thread its share of
// the blocks, then a tree (one thread over 1024 blocks, a serial chain of
// loads and FP64 adds, took 366 us; this 8 us).
__global__ void __launch_bounds__(RB) reduce_final_kernel(const double* partials, int nblocks,
                                                          double* out) {
  __shared__ double sh[6][RB];
  const int tid = threadIdx.x;
  double t[6] = {0, 0, 0, 0, 0, 0};
  for (int b = tid; b < nblocks; b += RB)
    for (int k = 0; k < 6; ++k) t[k] += partials[b * 6 + k];
  for (int k = 0; k < 6; ++k) sh[k][tid] = t[k];
  __syncthreads();
  for (int w = RB / 2; w > 0; w >>= 1) {
    if (tid < w)
      for (int k = 0; k < 6; ++k) sh[k][tid] += sh[k][tid + w];
    __syncthreads();
  }
  if (tid != 0) return;
  out[0] = sh[0][0];
  out[1] = sh[1][0];
  out[2] = sh[3][0] > 0 ? sh[2][0] / sh[3][0] : 0.0;
  out[3] = sh[5][0] > 0 ? sh[4][0] / sh[5][0] : 0.0;
}

// f (9 planes) and g (5 planes) in the natural layout; each output is optional
__global__ void get_state_kernel(Dev d, int layout, float* f, float* g) {
  const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= d.n) return;
  const int y = (int)(s / d.nx), x = (int)(s - (long long)y * d.nx);
  const long long n = d.n;
  const bool wall = is_wall(d, x, y);
  if (f) {
    float fv[9];
    if (wall)
      for (int i = 0; i < 9; ++i) fv[i] = ld_f(d, i, s);
    else
      gather_f(d, x, y, layout, fv);
    for (int i = 0; i < 9; ++i) f[i * n + s] = fv[i];
  }
  if (g) {
    float gv[5];
    if (wall)
      for (int i = 0; i < 5; ++i) gv[i] = ld_g(d, i, s);
    else
      gather_g(d, x, y, layout, gv);
    for (int i = 0; i < 5; ++i) g[i * n + s] = gv[i];
  }
}

__global__ void set_state_kernel(Dev d, const float* f, const float* g) {
  const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= d.n) return;
  const long long n = d.n;
  if (f)
    for (int i = 0; i < 9; ++i) st_f(d, i, s, f[i * n + s]);
  if (g)
    for (int i = 0; i < 5; ++i) st_g(d, i, s, g[i * n + s]);
}

__global__ void validate_kernel(Dev d, const float* phi, const float* K, const float* T0,
                                const float* fl0, int* bad) {
  const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= d.n) return;
  const float p = phi[s], k = K[s], t = T0[s], l = fl0[s];
  bool ok = (p > 0.f && p <= 1.f) && (!d.flow || p < 1.f) && (k > 0.f) && isfinite(t) &&
            (l >= 0.f && l <= 1.f);
  if (!ok) atomicExch(bad, 1);
}

// The whole state of an FP32 lattice in natural layout (f as deviations, 9
// planes; g, 5 planes; f_l) into dst, 15 n floats; with ctr non-null into base +
// ctr[0] 15 n, after which (not in mode 1) ctr[0] advances (ctr[1]: 0, scratch),
// so one captured launch serves every replay of a graph.  mode and par as in
// takes_part: the next step's stream-collide pass over the far tiles may start
// once mode 1 is done with them.
template <bool SEAM>
__global__ void __launch_bounds__(256) keep_state_kernel(Dev d, int layout, int mode, int par,
                                                         float* base, unsigned* ctr) {
  const int n = (int)d.n, nx = d.nx;
  const float* F = static_cast<const float*>(d.f);
  const float* G = static_cast<const float*>(d.g);
  float* dst = base + (ctr ? (long long)ctr[0] * 15 * n : 0LL);
  const int x = blockIdx.x * 32 + threadIdx.x;
  for (int yb = blockIdx.y * 8; yb < d.ny; yb += gridDim.y * 8) {
    if (mode != 0 && !takes_part<SEAM>(d, mode, par, (yb / TE) * d.etx + (int)blockIdx.x)) continue;
    const int y = yb + threadIdx.y;
    if (x >= nx || y >= d.ny) continue;
    const int s = y * nx + x;
    const bool wall = is_wall(d, x, y);
    const float fls = d.fl[s];
    // every load is issued before any value is chosen (gather_f / gather_g
    // with the candidates of both layouts loaded up front)
    float own[9], str[9], gown[5], gstr[5];
    bool act[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) own[i] = F[i * n + s];
#pragma unroll
    for (int i = 0; i < 5; ++i) gown[i] = G[i * n + s];
    const bool swapped = layout == 1 && !wall;
    if (swapped) {
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        const int sx = wrapx(d, x - ex9(i)), sy = wrapy(d, y - ey9(i));
        const int t = sy * nx + sx;
        act[i] = flow_active(d, sx, sy);
        str[i] = F[opp9(i) * n + t];
        if (i < 5) gstr[i] = G[opp5(i) * n + t];
      }
    }
    const bool self = !wall && fls >= d.f_act;
    const long long nn = n;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const float v = (swapped && self && i > 0 && act[i]) ? str[i] : own[i];
      dst[i * nn + s] = v;
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) dst[(9 + i) * nn + s] = (swapped && i > 0) ? gstr[i] : gown[i];
    dst[14 * nn + s] = fls;
  }
  if (ctr && mode != 1) {
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      __threadfence();
      if (atomicAdd(ctr + 1, 1u) == gridDim.x * gridDim.y - 1) {
        ctr[1] = 0;
        ctr[0] = ctr[0] + 1;
      }
    }
  }
}

// Sentinel: every population and f_l of every node, flag stats[5] on the first
// value that is not finite (NaN or Inf).
__global__ void nonfinite_kernel(Dev d) {
  bool bad = false;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < d.n;
       s += (long long)gridDim.x * blockDim.x) {
    bool ok = isfinite(d.fl[s]);
    for (int i = 0; i < 9; ++i) ok = ok && isfinite(ld_pop(d, d.f, i * d.n + s));
    for (int i = 0; i < 5; ++i) ok = ok && isfinite(ld_pop(d, d.g, i * d.n + s));
    bad = bad || !ok;
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicExch(&d.stats[5], 1);
}

static unsigned grid1(long long n, int b) { return (unsigned)((n + b - 1) / b); }

void launch_load_fields(const Dev& d, const float* phi, const float* K, const float* T0,
                        const float* fl0, float* wallTl, cudaStream_t s) {
  if (d.storage == 1)
    load_fields_kernel<__half><<<d.ntiles, 256, 0, s>>>(d, phi, K, T0, fl0, wallTl);
  else if (d.storage == 2)
    load_fields_kernel<__nv_bfloat16><<<d.ntiles, 256, 0, s>>>(d, phi, K, T0, fl0, wallTl);
  else load_fields_kernel<float><<<d.ntiles, 256, 0, s>>>(d, phi, K, T0, fl0, wallTl);
}
// one CTA per enthalpy tile: does a non-wall node of it carry flow?
__global__ void __launch_bounds__(256) tile_activity_kernel(Dev d) {
  const int tile = blockIdx.x;
  const int X0 = (tile % d.etx) * TE, Y0 = (tile / d.etx) * TE;
  int any = 0;
  for (int k = threadIdx.x; k < TE * TE; k += blockDim.x) {
    const int x = X0 + k % TE, y = Y0 + k / TE;
    if (x < d.nx && y < d.ny && !is_wall(d, x, y) && d.fl[(long long)y * d.nx + x] >= d.f_act)
      any = 1;
  }
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) d.tact[tile] = (unsigned char)(any ? 1 : 0);
}

void launch_tile_activity(const Dev& d, cudaStream_t s) {
  if (d.ntiles > 0) tile_activity_kernel<<<d.ntiles, 256, 0, s>>>(d);
}

void launch_macros(const Dev& d, int layout, float* ux, float* uy, float* rho, float* T,
                   float* fl, cudaStream_t s) {
  const unsigned g = grid1(d.n, 256);
  if (d.storage == 1) macros_kernel<__half><<<g, 256, 0, s>>>(d, layout, ux, uy, rho, T, fl);
  else if (d.storage == 2)
    macros_kernel<__nv_bfloat16><<<g, 256, 0, s>>>(d, layout, ux, uy, rho, T, fl);
  else macros_kernel<float><<<g, 256, 0, s>>>(d, layout, ux, uy, rho, T, fl);
}
int reduce_blocks(const Dev& d) {
  long long b = (d.n + RB - 1) / RB;
  return (int)(b < 1024 ? b : 1024);
}
void launch_reduce(const Dev& d, int layout, double* partials, double* out, int nblocks,
                   cudaStream_t s) {
  if (d.storage == 1) reduce_kernel<__half><<<nblocks, RB, 0, s>>>(d, layout, partials);
  else if (d.storage == 2)
    reduce_kernel<__nv_bfloat16><<<nblocks, RB, 0, s>>>(d, layout, partials);
  else reduce_kernel<float><<<nblocks, RB, 0, s>>>(d, layout, partials);
  reduce_final_kernel<<<1, RB, 0, s>>>(partials, nblocks, out);
}
void launch_wall_nusselt(const Dev& d, int layout, int mode, int par, double* rows, double* acc,
                         cudaStream_t s) {
  const auto kernel = d.seam ? wall_nusselt_kernel<true> : wall_nusselt_kernel<false>;
  kernel<<<1, RB, 0, s>>>(d, layout, mode, par, rows, acc);
}
void launch_get_state(const Dev& d, int layout, float* f, float* g, cudaStream_t s) {
  get_state_kernel<<<grid1(d.n, 256), 256, 0, s>>>(d, layout, f, g);
}
void launch_set_state(const Dev& d, const float* f, const float* g, cudaStream_t s) {
  set_state_kernel<<<grid1(d.n, 256), 256, 0, s>>>(d, f, g);
}
void launch_keep_state(const Dev& d, int layout, float* base, unsigned* ctr, cudaStream_t s,
                       int mode, int par) {
  const int nby = (d.ny + 7) / 8, most = 2432 / d.etx;   // about two waves of blocks
  const dim3 grid(d.etx, nby < most ? nby : most > 1 ? most : 1);
  const auto kernel = d.seam ? keep_state_kernel<true> : keep_state_kernel<false>;
  kernel<<<grid, dim3(32, 8), 0, s>>>(d, layout, mode, par, base, ctr);
}
void launch_nonfinite(const Dev& d, int nblocks, cudaStream_t s) {
  nonfinite_kernel<<<nblocks, 256, 0, s>>>(d);
}
void launch_validate(const Dev& d, const float* phi, const float* K, const float* T0,
                     const float* fl0, int* bad, cudaStream_t s) {
  validate_kernel<<<grid1(d.n, 256), 256, 0, s>>>(d, phi, K, T0, fl0, bad);
}

}  // namespace lbm
