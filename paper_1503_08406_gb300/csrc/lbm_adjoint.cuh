// Host entry points of the adjoint of the conduction step (lbm_adjoint.cu).
#pragma once
#include "lbm_flow_adjoint.cuh"
#include "lbm_internal.cuh"

namespace lbm {

// all buffers n floats unless noted
struct AdjBuffers {
  float* a;          // a = phi dT / (sigma St)
  float* lamg;       // 5 n: adjoint of the populations after the step being reversed
  float* lamf;       // adjoint of f_l after the step (in), before it (out)
  // band nodes, by place in the band's order (BandOrder):
  float4* bc;        // c of the four neighbours, 0 off the band
  int4* bi;          // their places
  float4* bk;        // right-hand side, a w~_1 (both divided by the self term), T_l - T_s + a
  float* mu;         // mu (bands too wide for shared memory)
  float* nu;         // nu = c mu of the step being reversed by node, 0 off the band
  unsigned* done;    // CTAs of the band kernel that are done (0 between launches)
  float* lamgpre;    // 5 n: adjoint of the populations before the step
  float* lama;       // accumulated adjoint of a
  float* lamtw;      // ny: accumulated adjoint of the left wall profile
  int* pos;          // n: a band node's place in the band list (band_append)
  int band_m;        // band_main of the lattice
  float At[25];      // transposed collision matrix (u = 0), passed to kernels by value
};
struct Mat5 {
  float m[25];
};
// Objective terms the reverse sweep adds per state: the adjoint of the
// populations at x = 1 and x = 2 (all five planes) and of the left wall
// profile (the time-averaged left-wall Nusselt number: -2, 1/2 and 3/2 times
// H / (dT rows N)); zero for the melted fraction.
struct NuSrc {
  float g1, g2, tw;
};
// the left-wall Nusselt number of the current state (lbm_reduce's out[3]),
// added to acc[0] (lbm_aux.cu); mode and par as for launch_keep_state: mode 1
// leaves the terms of its rows in rows[ny], where mode 2 finds them
void launch_wall_nusselt(const Dev& d, int layout, int mode, int par, double* rows, double* acc,
                         cudaStream_t s);
// a = phi dT / (sigma St); lam_g = the Nusselt terms of the last state (rows that
// are no horizontal wall); lam_f = melt on non-wall nodes (1 / their number for
// the melted fraction, else 0)
void adj_seed(const Dev& d, float* lamf, float* lamg, float* a, float melt, NuSrc nu,
              cudaStream_t s);
// v[0..n) *= k
void adj_scale(long long n, float* v, float k, cudaStream_t s);
// v[0..n) *= w[0..n)
void adj_mul(long long n, float* v, const float* w, cudaStream_t s);
// J into out[0]; out holds 129 doubles (the rest: partial sums)
void adj_objective(const Dev& d, const float* fl, double* out, cudaStream_t s);
// the band (non-wall nodes with 0 < f < 1) on a list of n entries, four counts
// (band_append)
void adj_list(const Dev& d, const AdjBuffers& b, const float* f, int* list, int* count,
              cudaStream_t s);
// d.fl to base + k n, k = ctr[0], which then advances (ctr[1]: scratch, 0)
void adj_save(const Dev& d, float* base, unsigned* ctr, cudaStream_t s);
// One step of the reverse sweep, given f_l before (f0) and after (f1) it and
// the band after it (list, count): from b.lamg / b.lamf (after the step) to
// b.lamgpre / b.lamf (before it), the Nusselt terms (nu) of the state before
// it included.  old_list / old_count hold the band the previous call solved on
// (b.nu is still set there); they are emptied and refilled with the band before
// this step, for the next call.  The caller swaps b.lamg and b.lamgpre and the
// two lists.
void adj_step(const Dev& d, const AdjBuffers& b, const float* f0, const float* f1, int* list,
              int* count, int* old_list, int* old_count, int mu_sweeps, NuSrc nu,
              cudaStream_t s);
// One reversed step of the coupled adjoint (flow on): the band kernel on
// b.lamg / b.lamf (A.lg1 is b.lamg, A.lfl is b.lamf, A.fl1 the band's f_l),
// then lbm::coupled_reverse_node over every node; the band before the step is
// listed at A.next_list (its counts at A.next_count), which hold the previous
// call's band until then.
void adj_coupled_step(const Dev& d, const AdjBuffers& b, const CoupledStep<float>& A, int* list,
                      int* count, int mu_sweeps, cudaStream_t s);
// once per process before adj_step: the band kernel's shared-memory opt-in
bool adj_init();

}  // namespace lbm
