// Iterative enthalpy method for f_l(n+1) and the latent-heat source, Eq. (38),
// (40)-(42) and the inner iteration of Sec. 3.2.
//
// The fused kernel streamed the source-free thermal populations, so a node y
// sees T*(y) = sum_i g_i(y).  The latent source S~ = (S0, 0, 0, varpi S0, 0)
// of node x, S0 = -a(x) (f_l(n+1) - f_l(n)), a = phi dT / (sigma St), adds
// N^-1 S~ = S0 w~ to the post-collision populations of x, which stream to the
// neighbours: T(y) = T*(y) + sum_i w~_i S0(y - e_i).  With h = T + a f_l, the
// enthalpy relation f_l = clamp((h - T_s)/(T_l - T_s + a), 0, 1) is solved for
// f_l(n+1) as a fixed point.
//
// Work list.  The fused kernel stamps every 32x32 tile that may hold a phase
// change this step with the step's number (a counter it advances); tiles
// numerous enough to make walking the stamps slow are also put on a list.  Both
// kernels below run a fixed grid of CTAs that take the listed tiles in turn, so
// steps with no front cost almost nothing.  Stamps and the per-tile status
// words need no clearing between steps.
//
// enthalpy_solve: per listed tile, load T*, f_l(n) and a on the tile plus an
// 8-node halo, list the nodes that are not clamped whatever happens around
// them, and run red-black Gauss-Seidel sweeps over those; each
// node update solves its own term exactly,
//   f(x) = clamp((T*(x) + w~_0 a f_l(n) - T_s - w~_1 sum_{i>0} q(x - e_i)) / (T_l - T_s + w~_0 a), 0, 1),
//   q = a (f - f_l(n)),
// which has the same fixed point as the plain iteration (the map is monotone
// with slope < 1).  Sweeps stop when no node moves by more than about four
// float32 ulps of its value and of the terms it is computed from: Gauss-Seidel
// from f_l(n) approaches the fixed point from one side, so a looser stop would
// bias every step the same way, and a tighter one can chase a rounding cycle
// forever (at the melting threshold v is a small difference of two larger
// terms).  Two more sweeps follow the stop, which shrink what is left of the
// one-sided error down to rounding noise.  Nodes outside
// the halo keep f = f_l(n).  The tile's own results go to scratch as
// (f_l(n), f_l(n+1)).
//
// enthalpy_commit: per listed tile, store f_l(n+1), add the streamed source of
// every changed node to the five populations it reaches, and, before an odd
// step, swap the two slots of every flow link whose "both ends carry flow"
// state changed, so the AA layout matches the new flow mask.
#include <type_traits>

#include "lbm_internal.cuh"

namespace lbm {

// Over-relaxation factor of the projected SOR sweeps.  The Jacobi map of the
// self-solved update has spectral radius at most 4 w~_1 a / (T_l - T_s + w~_0 a),
// which is 2/3 with the paper's varpi = -2; red-black SOR on this diagonally
// dominant system converges for 0 < omega < 2, fastest near 2 / (1 + sqrt(1 - rho^2))
// (about 1.15 - 1.3).  The fixed point does not depend on omega.
constexpr float SOR_OMEGA = 1.15f;
constexpr int SOR_SWEEPS = 8;   // over-relaxed sweeps before plain Gauss-Seidel

__device__ __forceinline__ bool solved(const Dev& d, int tile, int stamp) {
  return (d.proc[tile] >> 3) == stamp;
}

// T* at node (x, y) from the populations after the step, stored as S:
// natural layout (layout 0) or swapped (layout 1, population i of x sits in
// x - e_i).  Neighbours one step away (xm, xp, ym, yp) wrap once at most.
template <typename S>
__device__ __forceinline__ float tstar_t(const Dev& d, int s, int xm, int xp, int ym, int yp,
                                         int x, int y, int layout) {
  const int n = (int)d.n;
  const S* G = static_cast<const S*>(d.g);
  // the stored g deviations add up to T* - T_m (the weights sum to 1)
  const float ref = std::is_same<S, float>::value ? 0.f : d.g_ref;
  if (layout == 0)
    return Pop<S>::ld(G + s) + Pop<S>::ld(G + n + s) + Pop<S>::ld(G + 2 * n + s) +
           Pop<S>::ld(G + 3 * n + s) + Pop<S>::ld(G + 4 * n + s) + ref;
  return Pop<S>::ld(G + s) + Pop<S>::ld(G + 3 * n + y * d.nx + xm) +
         Pop<S>::ld(G + 4 * n + ym * d.nx + x) + Pop<S>::ld(G + n + y * d.nx + xp) +
         Pop<S>::ld(G + 2 * n + yp * d.nx + x) + ref;
}

// bar.sync / bar.red.or on named barrier 1 over the first `threads` threads
__device__ __forceinline__ void sub_sync(int threads) {
  asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}
__device__ __forceinline__ bool sub_sync_or(int threads, bool v) {
  unsigned r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n"
      " selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r)
      : "r"((unsigned)v), "r"(threads)
      : "memory");
  return r != 0;
}

// ---- the solve's shared-memory layout ----------------------------------------
// A region (tile and halo) of RE x RE nodes inside a ring of one, split by
// colour: node (lx, ly) of colour c = (lx + ly) & 1 sits at
// c CN + (ly + 1) CW + (lx + 1) / 2.  A warp's nodes of one colour, and each of
// their four neighbours (all of the other colour), are then consecutive words
// (no bank conflicts), and the ring (a = q = 0) needs no boundary tests.
constexpr int CW = (RE + 2) / 2;        // 25 words a row of one colour
constexpr int CN = CW * (RE + 2);       // nodes of one colour, ring included
constexpr int CHALF = RE * RE / 2;      // nodes of one colour in the region
struct SolveSmem {
  float2 bi[2 * CN];             // T* + w~0 a f_l(n) - T_s, and 1 / (T_l - T_s + w~0 a)
  float2 af[2 * CN];             // a and f_l(n); a = 0 on walls, outside and on the ring
  float q[2 * CN];               // a (f - f_l(n))
  float f[2 * CN];               // current iterate
  unsigned short nodes[2][CHALF];   // the nodes the sweeps update, by colour: place | lx odd << 15
  int cnt[2];                    // how many
  int bits;                      // what changed in the tile
  int mine;                      // listed tiles of this CTA
  unsigned short tile[COUNT_TILES];
  int wsum[32];
};

// The tiles the step listed, counted from their stamps by every CTA for itself
// (at most COUNT_TILES of them): CTA bid takes those of rank bid, bid + nblk,
// ...  Returns their number; the CTA's own are in sm.tile[0 .. sm.mine).  They
// are also put on the step's list, for the commit kernel.
template <int PAR>
__device__ __forceinline__ int count_tiles(const Dev& d, SolveSmem& sm, int stamp, int bid,
                                           int nblk) {
  constexpr int J = (COUNT_TILES + EB - 1) / EB;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int* fl = d.flags + PAR * d.ntiles;
  int got[J];
#pragma unroll
  for (int j = 0; j < J; ++j) got[j] = j * EB + tid < d.ntiles ? fl[j * EB + tid] : 0;
  unsigned vote[J];
  int total = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    vote[j] = __ballot_sync(0xffffffffu, j * EB + tid < d.ntiles && got[j] == stamp);
    total += __popc(vote[j]);
  }
  if (lane == 0) sm.wsum[warp] = total;
  if (tid == 0) sm.mine = 0;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < EB / 32; ++w) {
    const int v = sm.wsum[w];
    before += w < warp ? v : 0;
    all += v;
  }
#pragma unroll
  for (int j = 0; j < J; ++j) {
    if ((vote[j] >> lane) & 1u) {
      const int rank = before + __popc(vote[j] & ((1u << lane) - 1u));
      if (rank % nblk == bid) {
        sm.tile[atomicAdd(&sm.mine, 1)] = (unsigned short)(j * EB + tid);
        d.list[PAR * d.ntiles + rank] = j * EB + tid;
      }
    }
    before += __popc(vote[j]);
  }
  __syncthreads();
  return all;
}

// The sweeps over the listed nodes (c0 and c1 of the two colours), on the first
// sw threads of the CTA (whole warps), M nodes of a colour a thread (M sw holds
// them all).  A thread keeps its nodes' coefficients and current values in
// registers, so that a sweep only exchanges q through shared memory; a thread
// without a node works on a corner of the ring, which no node reads, so that
// nothing branches (half a sweep 0.19 -> 0.13 us).  One node a thread and more
// warps beat two, three or four nodes a thread and fewer (256 x 4 slab: 14.9
// against 15.1 us a step with two, 17.5 and 18.1 with branches and three, four).
template <int M>
__device__ __forceinline__ void sweep_nodes(const Dev& d, SolveSmem& sm, int c0, int c1, int sw,
                                            int& sweeps, bool& unfinished) {
  const int tid = threadIdx.x;
  const float w1 = d.wt1;
  int pp[2][M], oo[2][M], ww[2][M];   // the node's place, its place in the other colour, its west
  float cb[2][M], cinv[2][M], ca[2][M], cfn[2][M], cf[2][M];
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const int j = tid + m * sw;
      const bool on = j < (c ? c1 : c0);
      const int v = on ? sm.nodes[c][j] : CW;   // (CW: row 1 of the ring's west side)
      const int r = v & 0x7fff;
      const int p = c * CN + r;
      const float2 bi = sm.bi[p], af = sm.af[p];
      pp[c][m] = on ? p : 0;                    // 0: a corner of the ring
      oo[c][m] = (1 - c) * CN + r;
      ww[c][m] = oo[c][m] - (v >> 15);
      cb[c][m] = on ? bi.x : 0.f;
      cinv[c][m] = on ? bi.y : 0.f;
      ca[c][m] = on ? af.x : 0.f;
      cfn[c][m] = on ? af.y : 0.f;
      cf[c][m] = on ? sm.f[p] : 0.f;
    }
  int it = 0, polish = 2;   // extra sweeps after the stop test passes
  bool more = true;
  for (; it < d.max_inner && (more || polish > 0); ++it) {
    if (!more) --polish;
    // over-relaxed for the first sweeps, then plain Gauss-Seidel: at the last
    // few ulps over-relaxation can cycle instead of meeting the stop test
    const float om = (more && it < SOR_SWEEPS) ? SOR_OMEGA : 1.f;
    bool changed = false;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float nb[M];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const float* q = sm.q + ww[c][m];
        const float* o = sm.q + oo[c][m];
        nb[m] = ((q[0] + q[1]) + o[-CW]) + o[CW];
      }
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const float fo = cf[c][m];
        const float raw = (cb[c][m] - w1 * nb[m]) * cinv[c][m];
        float v = (om == 1.f) ? raw : fo + om * (raw - fo);
        v = fminf(fmaxf(v, 0.f), 1.f);
        // converged at about four ulps of v and of the terms that make it
        const float tol =
            4.8e-7f * (v + (fabsf(cb[c][m]) + w1 * fabsf(nb[m])) * cinv[c][m]);
        changed |= fabsf(v - fo) > tol;
        cf[c][m] = v;
        // (a (v - f_l(n)) is exactly 0 on a node that does not move: a
        // spurious source there would cost a rounding of its neighbours'
        // 16-bit populations in the commit)
        sm.q[pp[c][m]] = ca[c][m] * (v - cfn[c][m]);
      }
      if (c == 0) {
        if (sw == 32) __syncwarp();
        else sub_sync(sw);
      }
    }
    // the second colour's barrier also collects the convergence vote
    bool any;
    if (sw == 32) {
      any = __any_sync(0xffffffffu, changed);
      __syncwarp();
    } else {
      any = sub_sync_or(sw, changed);
    }
    if (more) more = any;
  }
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int m = 0; m < M; ++m)
      if (pp[c][m] != 0) sm.f[pp[c][m]] = cf[c][m];
  sweeps = it;
  unfinished = more;
}

// One listed tile.  EB threads in rows of RE: a thread's nodes lie one above
// the other, an even number of rows apart, so they share a column and a colour
// and every index follows from the first by a constant.
//
// listed: null for a tile known to be listed; else where its stamp is, read
// beside the tile's nodes (which a tile not listed then reads for nothing).
template <int PAR, typename S>
__device__ __forceinline__ void solve_tile(const Dev& d, SolveSmem& sm, int tile, int ctr,
                                           const int* listed) {
  constexpr int LAYOUT = 1 - PAR;
  constexpr int RT = EB / RE;                      // rows the CTA covers at once
  constexpr int NK = RE / RT;                      // nodes of a thread
  static_assert(2 * EB >= CHALF, "room for every node");
  static_assert(EB % RE == 0 && RE % RT == 0 && RT % 2 == 0 && EB % 32 == 0, "block size");
  constexpr unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31;
  const float w0 = d.wt0, w1 = d.wt1, Ts = d.T_s, dTt = d.dTt;
  const int X0 = (tile % d.etx) * TE, Y0 = (tile / d.etx) * TE;
  const int ly0 = tid / RE, lx = tid - ly0 * RE;
  const bool odd = (lx + ly0) & 1;                 // colour of the thread's nodes
  const int r0 = (ly0 + 1) * CW + ((lx + 1) >> 1);   // place in the colour; + RT CW a node
  const int p0 = (odd ? CN : 0) + r0;
  if (tid < 2) sm.cnt[tid] = 0;
  if (tid == 2) sm.bits = 0;
  float fnv[NK], av[NK], Tv[NK];
  unsigned off = 0u;   // bit j: this thread's node j is a wall node or outside
  // a region inside the wall ring needs no wrapping and holds no wall node: its
  // loads go straight to their addresses, all of a thread's in flight together
  if (X0 - RH >= 1 && X0 + TE + RH <= d.nx - 1 && Y0 - RH >= 1 && Y0 + TE + RH <= d.ny - 1) {
    const int gx = X0 - RH + lx;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
      const int gy = Y0 - RH + ly0 + j * RT, s = gy * d.nx + gx;
      fnv[j] = d.fl[s];
      av[j] = d.phi[s];
      Tv[j] = tstar_t<S>(d, s, gx - 1, gx + 1, gy - 1, gy + 1, gx, gy, LAYOUT);
    }
  } else {
    const int gx = wrapx(d, X0 - RH + lx);
    const int xm = (gx == 0) ? d.nx - 1 : gx - 1, xp = (gx == d.nx - 1) ? 0 : gx + 1;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
      fnv[j] = av[j] = Tv[j] = 0.f;
      const int gy = wrapy(d, Y0 - RH + ly0 + j * RT);
      bool out = true;
      if (gx >= 0 && gy >= 0) {
        const int s = gy * d.nx + gx;
        fnv[j] = d.fl[s];
        out = is_wall(d, gx, gy);
        if (!out) {
          const int ym = (gy == 0) ? d.ny - 1 : gy - 1, yp = (gy == d.ny - 1) ? 0 : gy + 1;
          av[j] = d.phi[s];
          Tv[j] = tstar_t<S>(d, s, xm, xp, ym, yp, gx, gy, LAYOUT);
        }
      }
      if (out) off |= 1u << j;
    }
  }
  if (listed) {
    const int at = *listed;
    // (the values are wanted here: the loads stay above the branch)
#pragma unroll
    for (int j = 0; j < NK; ++j) asm volatile("" ::"f"(fnv[j]), "f"(av[j]), "f"(Tv[j]));
    if (at != ctr) return;
  }
  float bv[NK], iv[NK];
#pragma unroll
  for (int j = 0; j < NK; ++j) {
    const bool out = (off >> j) & 1u;
    const float fn = fnv[j];
    const float a = out ? 0.f : av[j] * d.lat * sigma_ratio(d, fn);   // phi dT / (sigma(f_l(n)) St)
    // (explicit roundings: every instance of the kernel computes the same bits)
    const float wa = __fmul_rn(w0, a);
    av[j] = a;
    bv[j] = out ? 0.f : __fmaf_rn(wa, fn, Tv[j]) - Ts;
    iv[j] = out ? 0.f : 1.f / __fadd_rn(dTt, wa);
    const int p = p0 + j * RT * CW;
    sm.af[p] = make_float2(a, fn);
    sm.bi[p] = make_float2(bv[j], iv[j]);
    sm.q[p] = 0.f;
    sm.f[p] = fn;
  }
  __syncthreads();
  // Nodes whose update is clamped whatever their neighbours do are fixed now
  // and left out of the sweeps: with q_j in [-a_j f_l(n)_j, a_j (1 - f_l(n)_j)],
  // the unclamped value (b - w~_1 sum_j q_j) inv stays <= 0 (or >= 1) when it
  // does so at the extreme sum (by a margin that covers rounding; none is
  // needed where f_l(n) = 0 at the node and around it and b <= 0, the untouched
  // solid at T_s: no q there is negative).  The nodes left, a band along the
  // front, are listed by colour; the fixed point is unchanged.
  unsigned keep = 0u;
  const int o0 = (odd ? 0 : CN) + r0, wst = o0 - (lx & 1);   // other colour; west neighbour
#pragma unroll
  for (int j = 0; j < NK; ++j) {
    const int r = j * RT * CW;
    const float2 nb[4] = {sm.af[wst + r], sm.af[wst + r + 1], sm.af[o0 + r - CW],
                          sm.af[o0 + r + CW]};
    float nlo = 0.f, nhi = 0.f;   // extreme neighbour sums of q
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      nlo -= nb[i].x * nb[i].y;
      nhi += nb[i].x * (1.f - nb[i].y);
    }
    const float fn = fnv[j];
    const float hi_raw = (bv[j] - w1 * nlo) * iv[j], lo_raw = (bv[j] - w1 * nhi) * iv[j];
    float v = -1.f;
    if (hi_raw < -1e-6f || (bv[j] <= 0.f && fn == 0.f && nlo == 0.f)) v = 0.f;
    else if (lo_raw > 1.f + 1e-6f) v = 1.f;
    if ((off >> j) & 1u) continue;
    if (v >= 0.f) {
      sm.f[p0 + r] = v;
      sm.q[p0 + r] = av[j] * (v - fn);
    } else {
      keep |= 1u << j;
    }
  }
  // list them: one place per warp and colour, then each lane's nodes in turn
  {
    const unsigned of_odd = __ballot_sync(FULL, odd);
    const unsigned own = odd ? of_odd : ~of_odd;
    unsigned vote[NK];
    int n0 = 0, n1 = 0;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
      vote[j] = __ballot_sync(FULL, (keep >> j) & 1u);
      n0 += __popc(vote[j] & ~of_odd);
      n1 += __popc(vote[j] & of_odd);
    }
    int at0 = 0, at1 = 0;
    if (lane == 0) {
      if (n0) at0 = atomicAdd(&sm.cnt[0], n0);
      if (n1) at1 = atomicAdd(&sm.cnt[1], n1);
    }
    at0 = __shfl_sync(FULL, at0, 0);
    at1 = __shfl_sync(FULL, at1, 0);
    int at = odd ? at1 : at0;
    const unsigned below = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
      const unsigned u = vote[j] & own;
      if ((keep >> j) & 1u)
        sm.nodes[odd][at + __popc(u & below)] =
            (unsigned short)((r0 + j * RT * CW) | ((lx & 1) << 15));
      at += __popc(u);
    }
  }
  __syncthreads();
  const int c0 = sm.cnt[0], c1 = sm.cnt[1], most = max(c0, c1);
  int it = 0;
  bool more = most > 0;   // (nothing left to sweep: solved by the fixing pass)
  if (most <= EB) {
    const int sw = min(EB, (most + 31) & ~31);
    if (tid < sw) sweep_nodes<1>(d, sm, c0, c1, sw, it, more);
  } else {
    const int sw = min(EB, 32 * ((most + 63) / 64));
    if (tid < sw) sweep_nodes<2>(d, sm, c0, c1, sw, it, more);
  }
  __syncthreads();
  unsigned ch = 0u;
  for (int k = tid; k < TE * TE; k += EB) {
    const int ly = k / TE, lt = k - ly * TE;
    const int gx = X0 + lt, gy = Y0 + ly;
    if (gx >= d.nx || gy >= d.ny) continue;
    const int r = ((lt + ly) & 1) * CN + (ly + RH + 1) * CW + ((lt + RH + 1) >> 1);
    const float fo = sm.af[r].y, fnw = sm.f[r];
    d.scr[gy * d.nx + gx] = make_float2(fo, fnw);
    if (fnw != fo) ch |= (fo >= d.f_act) != (fnw >= d.f_act) ? 6u : 2u;
  }
  ch = __reduce_or_sync(FULL, ch);
  if (lane == 0 && ch) atomicOr(&sm.bits, (int)ch);
  __syncthreads();
  if (tid == 0) {
    if (more) {
      atomicExch(&d.stats[0], 1);
      d.stats[3] = tile;
    }
    atomicAdd(&d.stats[1], 1);
    atomicMax(&d.stats[2], it);
    d.proc[tile] = ((ctr & 0x0FFFFFFF) << 3) | 1 | sm.bits;
  }
  __syncthreads();
}

// CTA bid of nblk (the whole grid of a single lattice's launch, a range of a
// batched one) takes listed tiles bid, bid + nblk, ...
//
// Bound by latency: one tile's chain of the stamps, the loads, the fixing pass
// and some thirteen sweeps, on one SM (8 us of the 17.5 us step at 256^2).  It
// took 23 us there (40 us beside the far tiles at 2048^2) when the sweeps ran
// over the bounding box of the nodes left: solid at exactly T_s is not clamped
// by the margin test, so the box was half the region, three nodes a thread, and
// each sweep worked out every node's place again.
template <int PAR, typename S>
__device__ __forceinline__ void enthalpy_solve_body(const Dev& d, int bid, int nblk) {
  const long long tr0 = trace_start(d);
  extern __shared__ __align__(16) unsigned char solve_smem[];
  SolveSmem& sm = *reinterpret_cast<SolveSmem*>(solve_smem);
  const int tid = threadIdx.x;
  if (d.ntiles <= nblk) allow_dependents();
  const int ctr = d.ctr[PAR];
  // the ring: no node there, a = q = 0
  for (int k = tid; k < 4 * (RE + 2); k += EB) {
    const int e = k / (RE + 2), i = k - e * (RE + 2);
    const int px = e == 0 ? 0 : e == 1 ? RE + 1 : i, py = e == 2 ? 0 : e == 3 ? RE + 1 : i;
    const int p = ((px + py) & 1) * CN + py * CW + (px >> 1);
    sm.af[p] = make_float2(0.f, 0.f);
    sm.q[p] = 0.f;
  }
  if (d.ntiles <= nblk) {   // a CTA for every tile: whose it is needs no count
    if (bid < d.ntiles) solve_tile<PAR, S>(d, sm, bid, ctr, d.flags + PAR * d.ntiles + bid);
  } else if (d.ntiles > COUNT_TILES) {   // the stream-collide pass kept a list
    int tile = bid < d.ntiles ? d.list[PAR * d.ntiles + bid] : 0;
    const int cnt = d.lcount[PAR];
    for (int li = bid; li < cnt; li += nblk) {
      if (li != bid) tile = d.list[PAR * d.ntiles + li];
      solve_tile<PAR, S>(d, sm, tile, ctr, nullptr);
    }
    if (tid == 0 && bid == 0) d.lcount[2 + PAR] = cnt;
  } else {
    const int rank = count_tiles<PAR>(d, sm, ctr, bid, nblk);
    for (int i = 0; i < sm.mine; ++i) solve_tile<PAR, S>(d, sm, sm.tile[i], ctr, nullptr);
    if (tid == 0 && bid == 0) d.lcount[PAR] = d.lcount[2 + PAR] = rank;
  }
  if (tid == 0 && d.trace) trace_end(d, 100 * PAR + 20, ctr, tr0);
}

template <int PAR, typename S>
__global__ void __launch_bounds__(EB, 1) enthalpy_solve_kernel(Dev d) {
  enthalpy_solve_body<PAR, S>(d, (int)blockIdx.x, (int)gridDim.x);
}

// (two CTAs an SM, where a batch lists many small tiles at once: 24 lattices, 64 steps
// 6.34 ms; one CTA's worth of registers 6.66, three CTAs on 32 registers, with spills,
// 6.59)
template <int PAR, typename S>
__global__ void __launch_bounds__(EB, 2) enthalpy_solve_batch_kernel(const __grid_constant__ BatchPlan P) {
  const int c = plan_lattice(P, (int)blockIdx.x);
  enthalpy_solve_body<PAR, S>(P.d[c], (int)blockIdx.x - P.start[c], P.start[c + 1] - P.start[c]);
}

// x changed flow activity and is the inward node of a flow wall w next to it:
// w's links to its other lattice neighbours x' change state with x.  Those x'
// that kept their activity leave the link to x (a changed x' takes it itself).
template <int PAR>
__device__ __noinline__ void wall_links(const Dev& d, int x, int y, bool ao, bool an,
                                        int stamp) {
  const int n = (int)d.n;
  for (int j = 1; j < 9; ++j) {
    const int wx = wrapx(d, x + ex9(j)), wy = wrapy(d, y + ey9(j));
    if (wx < 0 || wy < 0 || !is_wall(d, wx, wy)) continue;
    int ix, iy;
    inward_of(d, wx, wy, ix, iy);
    if (ix != x || iy != y) continue;
    for (int k = 1; k < 9; ++k) {
      const int px = wrapx(d, wx + ex9(k)), py = wrapy(d, wy + ey9(k));
      if (px < 0 || py < 0 || is_wall(d, px, py) || (px == x && py == y)) continue;
      const int ps = py * d.nx + px;
      const bool vs = solved(d, (py / TE) * d.etx + (px / TE), stamp);
      const float fo = vs ? d.scr[ps].x : d.fl[ps], fnw = vs ? d.scr[ps].y : fo;
      const bool xo = fo >= d.f_act, xn = fnw >= d.f_act;
      if (xo != xn || (xo && ao) == (xn && an)) continue;
      // the pair (x', w): population opp(k) at w, population k at x'
      const long long A = (long long)opp9(k) * n + (wy * d.nx + wx);
      const long long B = (long long)k * n + ps;
      const float t = ld_pop(d, d.f, A);
      st_pop(d, d.f, A, ld_pop(d, d.f, B));
      st_pop(d, d.f, B, t);
    }
  }
}

template <int PAR, bool WALLS>
__device__ __forceinline__ void enthalpy_commit_body(const Dev& d, int bid, int nblk) {
  const long long tr0 = trace_start(d);
  constexpr int LAYOUT = 1 - PAR;
  constexpr int RW = TE + 2;              // tile plus a one-node ring
  __shared__ float2 sp[RW * RW];          // (f_l(n), f_l(n+1)); (-1,-1) on walls / outside
  __shared__ unsigned char ssolved[RW * RW];
  static_assert(CB == TE * TE, "one thread per node of a tile");
  const int tid = threadIdx.x;
  // as in the solve: a CTA for every tile (tile bid, if it is listed), or the
  // step's list, whose first entry is read beside the count (a CTA without a
  // tile reads a place of the list that is not in use)
  const bool direct = d.ntiles <= nblk;
  const int ctr = d.ctr[PAR], stamp = ctr & 0x0FFFFFFF;
  int at = 0, cnt = d.ntiles;
  if (direct) {
    allow_dependents();
    // the pass before the solve stamped the tiles: a CTA without one is done
    if (bid < d.ntiles) at = d.flags[PAR * d.ntiles + bid];
    if (bid != 0 && at != ctr) cnt = 0;
    else wait_for_previous();
    if (at != ctr) cnt = 0;
  } else {
    if (bid < d.ntiles) at = d.list[PAR * d.ntiles + bid];
    cnt = d.lcount[PAR];
  }
  const int n = (int)d.n;
  int tile = direct ? bid : at;
  for (int li = bid; li < cnt; li += nblk) {
    if (li != bid) tile = d.list[PAR * d.ntiles + li];
    const int tx0 = tile % d.etx, ty0 = tile / d.etx;
    const int X0 = tx0 * TE, Y0 = ty0 * TE;
    // this thread's node, read beside the tile's status word
    const int x = X0 + tid % TE, y = Y0 + tid / TE, s = y * d.nx + x;
    const bool node = x < d.nx && y < d.ny && !is_wall(d, x, y);
    float2 p = make_float2(0.f, 0.f);
    float ph = 0.f;
    if (node) {
      p = d.scr[s];
      ph = d.phi[s];
    }
    const int pb = d.proc[tile] & 7;
    // flow links need attention only around tiles where a node's activity
    // changed (nine threads look at the tile and those around it)
    int around = 0;
    if (LAYOUT == 1 && d.flow && tid < 9) {
      int tx = tx0 + tid % 3 - 1, ty = ty0 + tid / 3 - 1;
      if (d.per_x) tx = tx < 0 ? d.etx - 1 : tx >= d.etx ? 0 : tx;
      if (d.per_y) ty = ty < 0 ? d.ety - 1 : ty >= d.ety ? 0 : ty;
      if (tx >= 0 && tx < d.etx && ty >= 0 && ty < d.ety) around = d.proc[ty * d.etx + tx];
    }
    bool lk = false;
    if (LAYOUT == 1 && d.flow) lk = __syncthreads_or((around >> 3) == stamp && (around & 4));
    if ((pb & 2) || lk) {
      if (lk) {
        // old/new liquid fraction of the tile and its ring: scratch in tiles
        // solved this step, the (unchanged) stored value elsewhere
#pragma unroll 2
        for (int k = tid; k < RW * RW; k += CB) {
          const int ly = k / RW, lx = k - ly * RW;
          const int gx = wrapx(d, X0 - 1 + lx), gy = wrapy(d, Y0 - 1 + ly);
          float2 v = make_float2(-1.f, -1.f);
          unsigned char sol = 0;
          if (gx >= 0 && gy >= 0) {
            const bool wall = is_wall(d, gx, gy);
            // a flow wall node carries flow with its inward node (marked 2)
            int vx = gx, vy = gy;
            if (WALLS && wall) inward_of(d, gx, gy, vx, vy);
            if (!wall || WALLS) {
              const int gs = vy * d.nx + vx;
              const bool vs = solved(d, (vy / TE) * d.etx + (vx / TE), stamp);
              sol = wall ? 2 : vs ? 1 : 0;
              if (vs) {
                v = d.scr[gs];
              } else {
                const float f = d.fl[gs];
                v = make_float2(f, f);
              }
            }
          }
          sp[k] = v;
          ssolved[k] = sol;
        }
        __syncthreads();
      }
      int flows = 0;   // a node of the tile carries flow after the step
      if (node) {
        const int ly = tid / TE, lx = tid % TE;
        const float fn = p.x, fnew = p.y;
        flows = fnew >= d.f_act;
        if (fnew != fn) {
          d.fl[s] = fnew;
          const float S0 = -ph * d.lat * sigma_ratio(d, fn) * (fnew - fn);
          // N^-1 S~ = S0 w~, streamed: population i of node x + e_i gains w~_i S0
          int slot[5];
          float old[5];
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            const int rx = wrapx(d, x + ex9(i)), ry = wrapy(d, y + ey9(i));
            const bool to = rx >= 0 && ry >= 0 && !is_wall(d, rx, ry);
            slot[i] = !to ? -1 : (LAYOUT == 1) ? opp5(i) * n + s : i * n + ry * d.nx + rx;
            old[i] = to ? ld_pop(d, d.g, slot[i]) : 0.f;
          }
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            if (slot[i] < 0) continue;
            const float w = (i == 0) ? d.wt0 : d.wt1;
            // (16-bit storage: rounded stochastically, or every small source
            // would be lost to rounding in the same direction)
            st_pop_round(d, d.g, slot[i], old[i] + w * S0,
                         mix32((unsigned)slot[i] ^ mix32((unsigned)stamp)));
          }
        }
        if (lk) {
          const bool ao = fn >= d.f_act, an = fnew >= d.f_act;
          const int c = (ly + 1) * RW + (lx + 1);
#pragma unroll
          for (int i = 1; i < 9; ++i) {
            const int q = c + ey9(i) * RW + ex9(i);
            const float2 pp = sp[q];
            const bool po = pp.x >= d.f_act, pn = pp.y >= d.f_act;
            if ((ao && po) == (an && pn)) continue;
            // link (x, x + e_i) belongs to x for E, N, NE, NW, otherwise to the
            // partner; a partner in a tile not solved this step cannot handle it.
            // A link to a flow wall belongs to x when x changed, else to the
            // wall's inward node (below).
            const bool own = (i == 1 || i == 2 || i == 5 || i == 6);
            if (ssolved[q] == 2 ? ao == an : (!own && ssolved[q])) continue;
            const int px = wrapx(d, x + ex9(i)), py = wrapy(d, y + ey9(i));
            const long long A = (long long)i * n + (py * d.nx + px);
            const long long B = (long long)opp9(i) * n + s;
            const float t = ld_pop(d, d.f, A);   // exact for every storage type
            st_pop(d, d.f, A, ld_pop(d, d.f, B));
            st_pop(d, d.f, B, t);
          }
        }
      }
      // links of flow walls whose inward node changed (tiles along the walls)
      if (WALLS && lk &&
          (X0 == 0 || Y0 == 0 || X0 + TE >= d.nx - 1 || Y0 + TE >= d.ny - 1)) {
        for (int k = tid; k < TE * TE; k += CB) {
          const int ly = k / TE, lx = k - ly * TE;
          const int x = X0 + lx, y = Y0 + ly;
          if (x >= d.nx || y >= d.ny || is_wall(d, x, y)) continue;
          int ix, iy;
          bool inw = false;
          for (int j = 1; j < 9 && !inw; ++j) {
            const int wx = wrapx(d, x + ex9(j)), wy = wrapy(d, y + ey9(j));
            if (wx < 0 || wy < 0 || !is_wall(d, wx, wy)) continue;
            inward_of(d, wx, wy, ix, iy);
            inw = ix == x && iy == y;
          }
          if (!inw) continue;
          const float2 p = d.scr[y * d.nx + x];
          const bool ao = p.x >= d.f_act, an = p.y >= d.f_act;
          if (ao != an) wall_links<PAR>(d, x, y, ao, an, stamp);
        }
      }
      // (the stream-collide pass copies a tile's flow populations only when
      // this is set; no fused pass reads it while the commit runs on its tile)
      if (pb & 2) {
        flows = __syncthreads_or(flows);
        if (tid == 0) d.tact[tile] = (unsigned char)(flows ? 1 : 0);
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && d.trace) trace_end(d, 100 * PAR + 30, d.ctr[PAR], tr0);
}

template <int PAR, bool WALLS>
__global__ void __launch_bounds__(CB, 2) enthalpy_commit_kernel(Dev d) {
  enthalpy_commit_body<PAR, WALLS>(d, (int)blockIdx.x, (int)gridDim.x);
}

template <int PAR>
__global__ void __launch_bounds__(CB, 2) enthalpy_commit_batch_kernel(const __grid_constant__ BatchPlan P) {
  const int c = plan_lattice(P, (int)blockIdx.x);
  enthalpy_commit_body<PAR, false>(P.d[c], (int)blockIdx.x - P.start[c], P.start[c + 1] - P.start[c]);
}

size_t enthalpy_solve_smem() { return sizeof(SolveSmem); }

template <typename S>
static void solve_setup_t(int bytes) {
  cudaFuncSetAttribute(enthalpy_solve_kernel<0, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       bytes);
  cudaFuncSetAttribute(enthalpy_solve_kernel<1, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       bytes);
}

void enthalpy_setup() {
  const int bytes = (int)enthalpy_solve_smem();
  solve_setup_t<float>(bytes);
  solve_setup_t<__half>(bytes);
  solve_setup_t<__nv_bfloat16>(bytes);
}

template <typename S>
static void launch_solve_t(const Dev& d, int parity, cudaStream_t s) {
  const size_t sm = enthalpy_solve_smem();
  if (parity == 0) enthalpy_solve_kernel<0, S><<<d.egrid, EB, sm, s>>>(d);
  else enthalpy_solve_kernel<1, S><<<d.egrid, EB, sm, s>>>(d);
}

void launch_enthalpy_solve(const Dev& d, int parity, cudaStream_t s) {
  if (d.storage == 1) launch_solve_t<__half>(d, parity, s);
  else if (d.storage == 2) launch_solve_t<__nv_bfloat16>(d, parity, s);
  else launch_solve_t<float>(d, parity, s);
}

void fused_batch_setup();   // lbm_fused_f32.cu

void batch_setup() {
  fused_batch_setup();
  const int bytes = (int)enthalpy_solve_smem();
  cudaFuncSetAttribute(enthalpy_solve_batch_kernel<0, float>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(enthalpy_solve_batch_kernel<1, float>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

void launch_enthalpy_solve_batch(const BatchPlan& P, int parity, cudaStream_t s) {
  const size_t sm = enthalpy_solve_smem();
  const int grid = P.start[P.count];
  if (grid <= 0) return;
  if (parity == 0) enthalpy_solve_batch_kernel<0, float><<<grid, EB, sm, s>>>(P);
  else enthalpy_solve_batch_kernel<1, float><<<grid, EB, sm, s>>>(P);
}

void launch_enthalpy_commit_batch(const BatchPlan& P, int parity, cudaStream_t s) {
  const int grid = P.start[P.count];
  if (grid <= 0) return;
  if (parity == 0) enthalpy_commit_batch_kernel<0><<<grid, CB, 0, s>>>(P);
  else enthalpy_commit_batch_kernel<1><<<grid, CB, 0, s>>>(P);
}

template <int PAR, bool WALLS>
static void launch_commit_one(const Dev& d, cudaStream_t s) {
  if (early_launches(d))
    launch_early(enthalpy_commit_kernel<PAR, WALLS>, dim3(d.cgrid), dim3(CB), 0, s, d);
  else enthalpy_commit_kernel<PAR, WALLS><<<d.cgrid, CB, 0, s>>>(d);
}

void launch_enthalpy_commit(const Dev& d, int parity, cudaStream_t s) {
  // flow walls add their links to the re-pairing (a variant of its own, which
  // leaves the common one's registers alone)
  if (d.flow && d.flow_walls) {
    if (parity == 0) launch_commit_one<0, true>(d, s);
    else launch_commit_one<1, true>(d, s);
  } else {
    if (parity == 0) launch_commit_one<0, false>(d, s);
    else launch_commit_one<1, false>(d, s);
  }
}

}  // namespace lbm
