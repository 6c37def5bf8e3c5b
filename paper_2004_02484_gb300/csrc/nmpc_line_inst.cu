// Whole solves of 1D instances, one launch per solve: every instance is solved
// to the end by its own CTA (or cluster of CTAs), with its iterates resident
// in shared memory.  The line path's other form (nmpc_line.cuh) launches one
// kernel per iteration over every stage of every instance; there a stage's
// five float64 fields come from L2 and go back every iteration, a launch
// waits for the slowest stage of the whole batch, and a batch's last
// instances (or a single one) pay a launch of 4 to 9 us per iteration.
#include "nmpc_core.cuh"
#include "nmpc_line_inst.h"

#include <algorithm>
#include <cmath>
#include <map>
#include <tuple>

namespace nmpc_dev {

constexpr int LI_MAX_WARPS = 64;  // of one instance, over its cluster

// Warps a CTA may have, by cells per lane: the registers of a lane's cells
// (64, 96 or 128 a thread).
__host__ __device__ constexpr int li_max_warps(int cpl) { return cpl <= 2 ? 32 : (cpl <= 4 ? 20 : 16); }

// Shared memory of one CTA (byte offsets): rows of 32 cpl cells (cell l cpl + t
// of a stage at t 32 + l: a warp's accesses hit distinct banks), stages
// row0 .. row0 + rows - 1 of x and lambda, per warp a copy of the stage after
// its own, x0, the controls; the residual history; every warp's norms.
struct LiLayout {
  size_t x, lam, nxt, x0, u, hist_r, hist_e, red_r, red_e, red_q, ref, v3, act, bytes;
};
__host__ __device__ inline LiLayout li_layout(int cpl, int rows, int warps, int nu) {
  const size_t row = (size_t)32 * cpl * 8;
  LiLayout L;
  size_t o = 0;
  L.x = o; o += rows * row;
  L.lam = o; o += rows * row;
  L.nxt = o; o += warps * row;
  L.x0 = o; o += row;
  L.u = o; o += (size_t)rows * nu * 8;
  L.hist_r = o; o += RES_SLOTS * 8;
  L.hist_e = o; o += RES_SLOTS * 8;
  L.red_r = o; o += LI_MAX_WARPS * 8;
  L.red_e = o; o += LI_MAX_WARPS * 8;
  L.red_q = o; o += LI_MAX_WARPS * 8;
  L.ref = o; o += row / 2;
  L.v3 = o; o += (size_t)warps * nu * 4;
  L.act = o; o += (size_t)nu * 4;
  L.bytes = (o + 15) & ~size_t(15);
  return L;
}
// First stage of warp gw of wt.
__host__ __device__ inline int li_stage(int gw, int wt, int N) { return gw * N / wt; }

// Maximum over the warp of non-negative floats (their bits order as integers;
// a NaN is above infinity).
__device__ __forceinline__ float warp_max_nn(float v) {
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// a b - c d, the first product unrounded
__device__ __forceinline__ float diff_products(float a, float b, float c, float d) {
  return __fmaf_rn(a, b, -__fmul_rn(c, d));
}

template <int CPL, typename V>
__device__ __forceinline__ void li_nsum(const V (&v)[CPL], V (&out)[CPL], int lane) {
  V lft = __shfl_up_sync(0xffffffffu, v[CPL - 1], 1);
  V rgt = __shfl_down_sync(0xffffffffu, v[0], 1);
  lft = (lane == 0) ? V(0) : lft;
  rgt = (lane == 31) ? V(0) : rgt;
#pragma unroll
  for (int t = 0; t < CPL; ++t) out[t] = (t > 0 ? v[t - 1] : lft) + (t < CPL - 1 ? v[t + 1] : rgt);
}

// One instance.  Warp gw of the instance's wt warps owns the stages
// li_stage(gw) .. li_stage(gw + 1) - 1 and walks them upwards in every
// iteration, updating x_i, lambda_i in place: x_{i-1} of iterate k stays in
// registers from the stage before (the stage below a warp's first one is
// read before anything of the iteration is written), lambda_{i+1} is not
// overwritten yet (the stage above a warp's last one is copied before).  A
// lane holds CPL consecutive cells; the arithmetic of a stage is k_line's, with
// the multiply-adds written out as k_line's were contracted by the compiler that
// this was measured with (the neighbour sums too: hence the same cells per
// lane).  Single instances then walk the same iterates; in a batch a few differ in
// the last bits (1024 ragged instances: solutions equal to 4e-14 relative); the
// tests ask for 1e-9.
// An iteration whose residual is float64 evaluates the norms of all stages
// first and updates only if the solve goes on, since the returned iterate is
// the one whose residual passed.  A split residual that diverges is known only
// after the update, so that instance asks for a solve by iterations (*retry),
// which returns the iterate before it; it stores nothing, so S^0 and its control
// words are there for that (the other instances of the launch are done).
// What bounds it: the float64 pipe (56% busy on 304 instances of 256 cells:
// two differences and two updates a cell) and latency (0.45 instructions a
// cycle a scheduler, 16 warps a SM at 128 registers).  1024 ragged instances
// (M 32..256, N 10..60): 54.6 -> 41.2 ms a solve, 38.0 with the sweeps a
// constant; one instance of M = 32, N = 20 on 8 CTAs: 1007 -> 561 us, 0.50 to
// 0.53 ms with the constant (828 us on one CTA, whose warps share one float64
// pipe).  Eight cells a lane spill 324 bytes at 128 registers.
// NLO: the sweeps per solve as a constant (2, the default), or 0 to read them.
template <int CPL, int NLO>
__global__ void __launch_bounds__(32 * li_max_warps(CPL), 1)
    k_line_inst(IterArgs A, const int* list, int csize, int rows_max, int nu_max, int* retry) {
  extern __shared__ __align__(16) unsigned char smem[];
  asm volatile("griddepcontrol.launch_dependents;");
  const int rank = blockIdx.x % csize;  // rank in the cluster (clusters are consecutive blocks)
  const int b = list[blockIdx.x / csize];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
  const int wt = W * csize, gw = rank * W + warp;
  const InstDev I = A.inst[b];
  const int M = I.mx, N = I.N, nu = I.nu;
  const int a0 = li_stage(gw, wt, N), a1 = li_stage(gw + 1, wt, N);
  const int row0 = li_stage(rank * W, wt, N), row1 = li_stage(rank * W + W, wt, N);
  constexpr int ROW = 32 * CPL;
  const LiLayout Lo = li_layout(CPL, rows_max, W, nu_max);
  double* X = reinterpret_cast<double*>(smem + Lo.x);
  double* Lm = reinterpret_cast<double*>(smem + Lo.lam);
  double* NX = reinterpret_cast<double*>(smem + Lo.nxt) + warp * ROW;
  double* X0 = reinterpret_cast<double*>(smem + Lo.x0);
  double* U = reinterpret_cast<double*>(smem + Lo.u);
  unsigned long long* hist_r = reinterpret_cast<unsigned long long*>(smem + Lo.hist_r);
  unsigned long long* hist_e = reinterpret_cast<unsigned long long*>(smem + Lo.hist_e);
  unsigned long long* red_r = reinterpret_cast<unsigned long long*>(smem + Lo.red_r);
  unsigned long long* red_e = reinterpret_cast<unsigned long long*>(smem + Lo.red_e);
  double* red_q = reinterpret_cast<double*>(smem + Lo.red_q);
  float* RF = reinterpret_cast<float*>(smem + Lo.ref);
  float* v3s = reinterpret_cast<float*>(smem + Lo.v3) + warp * nu_max;
  int* act = reinterpret_cast<int*>(smem + Lo.act);
  // the instance's barrier
  auto sync_all = [&]() {
    if (csize > 1) cg::this_cluster().sync();
    else __syncthreads();
  };

  // ---- S^0, the reference (float32) and x0 into shared memory ----
  const double* Xg = A.xin[0] + I.s_off;
  const double* Lg = A.lin[0] + I.s_off;
  const double* Ug = A.uin[0] + I.u_off;
  for (int s = a0; s < a1; ++s)
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
      const int q = i * 32 + lane, p = (q % CPL) * 32 + q / CPL;
      X[(s - row0) * ROW + p] = q < M ? __ldcg(Xg + (long long)s * M + q) : 0.0;
      Lm[(s - row0) * ROW + p] = q < M ? __ldcg(Lg + (long long)s * M + q) : 0.0;
    }
  for (int q = threadIdx.x; q < ROW; q += blockDim.x) {
    const int p = (q % CPL) * 32 + q / CPL;
    X0[p] = q < M ? A.x0[I.g_off + q] : 0.0;
    RF[p] = q < M ? d2f(A.ref[I.g_off + q]) : 0.0f;
  }
  for (int e = threadIdx.x; e < (row1 - row0) * nu; e += blockDim.x)
    U[e] = __ldcg(Ug + (long long)row0 * nu + e);
  for (int a = threadIdx.x; a < nu; a += blockDim.x) act[a] = A.act[I.act_off + a];
  const int q0 = lane * CPL;
  sync_all();
  unsigned long long mine = 0ull;  // the actuators on this lane's cells
  for (int a = 0; a < nu; ++a)
    if (act[a] >= q0 && act[a] < q0 + CPL) mine |= 1ull << a;

  const float th = I.fh, tdc = I.fdc, tcx = I.fcx, tb0 = I.fb0;
  const double alpha = A.alpha;
  const int n_lo = NLO > 0 ? NLO : A.n_lo, n_u_it = A.n_u_it;
  double xp[CPL];  // x_{i-1} of iterate k, the lane's cells

  // x below the warp's first stage into xp; lambda above its last one into NX
  auto below = [&]() {
    const double* src = X0;
    if (a0 < a1 && a0 > 0) {
      if (a0 > row0) {
        src = X + (a0 - 1 - row0) * ROW;
      } else {  // the CTA before holds it
        const int r0 = li_stage((rank - 1) * W, wt, N);
        src = cg::this_cluster().map_shared_rank(X, rank - 1) + (a0 - 1 - r0) * ROW;
      }
    }
#pragma unroll
    for (int t = 0; t < CPL; ++t) xp[t] = src[t * 32 + lane];
  };
  auto above = [&]() {
    if (a0 >= a1 || a1 >= N) return;
    const double* src = a1 < row1 ? Lm + (a1 - row0) * ROW
                                  : cg::this_cluster().map_shared_rank(Lm, rank + 1);
#pragma unroll
    for (int t = 0; t < CPL; ++t) NX[t * 32 + lane] = src[t * 32 + lane];
  };
  // the warp's norms to every CTA of the cluster
  auto publish = [&](unsigned long long r, unsigned long long e, double q) {
    if (lane < csize) {
      unsigned long long *rr = red_r, *re = red_e;
      double* rq = red_q;
      if (lane != rank) {
        rr = cg::this_cluster().map_shared_rank(rr, lane);
        re = cg::this_cluster().map_shared_rank(re, lane);
        rq = cg::this_cluster().map_shared_rank(rq, lane);
      }
      rr[gw] = r;
      re[gw] = e;
      rq[gw] = q;
    }
  };

  // one pass over the warp's stages: norms and (update) the iteration
  auto stages = [&](auto FULL_, bool update, bool publ) {
    constexpr bool FULL = decltype(FULL_)::value;
    double vmax = 0.0, vsq = 0.0, e_max = 0.0;
    float fmx = 0.0f, fs = 0.0f;
    for (int s = a0; s < a1; ++s) {
      const bool last = (s == N - 1);
      double* Xr = X + (s - row0) * ROW + lane;
      double* Lr = Lm + (s - row0) * ROW + lane;
      const double* Ln = (s + 1 < a1) ? Lr + ROW : NX + lane;
      double* Us = U + (s - row0) * nu;
      float K1[CPL], K3[CPL], dp[CPL], ax[CPL], rg[CPL];
      // stage-gradient rows of the lane's controls: norms, K2 (b3)
      float b3 = 0.0f;  // of the lane's only control; several are formed again below
      float k2m = 0.0f;
      for (unsigned long long m = mine; m; m &= m - 1) {
        const int a = __ffsll((long long)m) - 1;
        const double K2 = I.h * (I.r * Us[a] + I.b0 * Lr[(act[a] - q0) * 32]);
        if constexpr (FULL) {
          vmax = fmax(vmax, abs_or_inf(K2));
          vsq += K2 * K2;
        } else {
          const float K2f = d2f(K2);
          fmx = fmax_nan(fmx, fabsf(K2f));
          fs += K2f * K2f;
          k2m = fmaxf(k2m, fabsf(K2f));
        }
        b3 = (float)K2;
        v3s[a] = 0.0f;
      }
      if constexpr (FULL) {
        double xd[CPL], ld[CPL], ph[CPL], ns[CPL], lphi[CPL];
#pragma unroll
        for (int t = 0; t < CPL; ++t) {
          xd[t] = Xr[t * 32];
          ld[t] = Lr[t * 32];
          ph[t] = I.k0 * (xd[t] + 0.5 * I.k1 * xd[t] * xd[t]);
        }
        li_nsum<CPL, double>(ph, ns, lane);
#pragma unroll
        for (int t = 0; t < CPL; ++t) lphi[t] = I.cx * ns[t] - I.dcoef * ph[t];
        li_nsum<CPL, double>(ld, ns, lane);
#pragma unroll
        for (int t = 0; t < CPL; ++t) {
          const bool valid = q0 + t < M;
          const double x = xd[t], lam = ld[t];
          const double rc = valid ? A.ref[I.g_off + q0 + t] : 0.0;
          const double ln = last ? I.hqf * (x - rc) : Ln[t * 32];
          const double mu = I.cx * ns[t] - I.dcoef * lam;
          const double dphi = I.k0 * (1.0 + I.k1 * x);
          double srcd = 0.0;  // controls on this cell
          for (unsigned long long m = mine; m; m &= m - 1) {
            const int a = __ffsll((long long)m) - 1;
            if (act[a] == q0 + t) srcd += Us[a];
          }
          const double t1 = I.h * (lphi[t] + srcd * I.b0);
          const double t3 = I.h * (I.q * (x - rc) + dphi * mu);
          const double K1d = xp[t] - x + t1;
          const double K3d = ln - lam + t3;
          if (valid) {
            vmax = fmax(vmax, fmax(abs_or_inf(K1d), abs_or_inf(K3d)));
            vsq += K1d * K1d + K3d * K3d;
          }
          K1[t] = d2f(K1d);
          K3[t] = d2f(K3d);
          dp[t] = d2f(dphi);
          ax[t] = d2f(I.h * (I.q + I.k0 * I.k1 * mu) + (last ? I.hqf : 0.0));
          rg[t] = valid ? rcp_T(-1.0f - th * tdc * dp[t]) : 0.0f;
        }
      } else {
        // controls' sources on the lane's cells
        float srcf[CPL];
#pragma unroll
        for (int t = 0; t < CPL; ++t) srcf[t] = 0.0f;
        for (unsigned long long m = mine; m; m &= m - 1) {
          const int a = __ffsll((long long)m) - 1, tc = act[a] - q0;
          const float ua = d2f(Us[a]);
#pragma unroll
          for (int t = 0; t < CPL; ++t)
            if (t == tc) srcf[t] += ua;
        }
        float xv[CPL], lv[CPL], ph[CPL], ns[CPL], lphi[CPL];
        float4 mg = make_float4(0.f, 0.f, k2m, 0.f);
#pragma unroll
        for (int t = 0; t < CPL; ++t) {
          xv[t] = d2f(Xr[t * 32]);
          lv[t] = d2f(Lr[t * 32]);
          ph[t] = __fmul_rn(I.fk0, __fmaf_rn(__fmul_rn(I.fk1h, xv[t]), xv[t], xv[t]));
          mg.x = fmaxf(mg.x, fabsf(xv[t]));
          mg.y = fmaxf(mg.y, fabsf(lv[t]));
        }
        li_nsum<CPL, float>(ph, ns, lane);
#pragma unroll
        for (int t = 0; t < CPL; ++t) lphi[t] = diff_products(I.fcx, ns[t], I.fdc, ph[t]);
        li_nsum<CPL, float>(lv, ns, lane);
        const float hqff = last ? I.fhqf : 0.0f;
#pragma unroll
        for (int t = 0; t < CPL; ++t) {
          const bool valid = q0 + t < M;
          const double x = Xr[t * 32], lam = Lr[t * 32];
          const float rv = RF[t * 32 + lane];
          const float mu = diff_products(I.fcx, ns[t], I.fdc, lv[t]);
          const float dphi = __fmul_rn(I.fk0, __fmaf_rn(I.fk1, xv[t], 1.0f));
          const float t1 = __fmaf_rn(I.fb0, srcf[t], lphi[t]);
          const float t3 = __fmaf_rn(dphi, mu, __fmul_rn(I.fq, __fsub_rn(xv[t], rv)));
          // the O(1) differences in float64 (see k_line)
          const double d3 = last ? -lam : Ln[t * 32] - lam;
          const float dx = d2f(xp[t] - x), dl = d2f(d3);
          const float K1f = __fmaf_rn(I.fh, t1, dx);
          const float K3h = __fmaf_rn(I.fh, t3, dl);
          const float K3f = __fadd_rn(K3h, __fmul_rn(hqff, __fsub_rn(xv[t], rv)));
          const float K1v = valid ? K1f : 0.0f, K3v = valid ? K3f : 0.0f;
          mg.z = fmaxf(mg.z, valid ? fmaxf(fabsf(dx), fabsf(dl)) : 0.0f);
          mg.w = fmaxf(mg.w, valid ? fabsf(rv) : 0.0f);
          fmx = fmax_nan(fmx, fmax_nan(fabsf(K1v), fabsf(K3v)));
          fs += K1v * K1v + K3v * K3v;
          K1[t] = K1f;
          K3[t] = K3f;
          dp[t] = dphi;
          ax[t] = __fmaf_rn(I.fh, __fmaf_rn(I.fk01, mu, I.fq), hqff);
          rg[t] = valid ? rcp_T(__fmaf_rn(-__fmul_rn(th, tdc), dp[t], -1.0f)) : 0.0f;
        }
        const float mags[4] = {warp_max_nn(mg.x), warp_max_nn(mg.y), warp_max_nn(mg.z),
                               warp_max_nn(mg.w)};
        float usum = 0.0f;
        for (int a = 0; a < nu; ++a) usum += fabsf(d2f(Us[a]));
        const double e = split_bound(I, last, mags, usum);
        e_max = fmax(e_max, e);
      }
      if (!update) {
#pragma unroll
        for (int t = 0; t < CPL; ++t) xp[t] = Xr[t * 32];
        continue;
      }

      // ---- lower layer: n_u_it + 1 applications of P^{-1} ----
      const float auu = I.fauu;
      const bool one = (mine & (mine - 1)) == 0ull;
      float v1[CPL], y5[CPL], y4[CPL], w1[CPL], ns[CPL];
#pragma unroll
      for (int t = 0; t < CPL; ++t) v1[t] = -K1[t] * rg[t];  // first F_x sweep (v3 = 0)
      for (int it = 0; it <= n_u_it; ++it) {
        if (it > 0) {
          // F_u v3 - K1 changes only on the control cells: refresh v1 there
          // (the first control on a cell carries the cell's total v3)
          for (unsigned long long m = mine; m; m &= m - 1) {
            const int a = __ffsll((long long)m) - 1, tc = act[a] - q0;
            float inj = 0.0f;
            bool first = true;
            for (unsigned long long m2 = mine; m2; m2 &= m2 - 1) {
              const int a2 = __ffsll((long long)m2) - 1;
              if (act[a2] != act[a]) continue;
              first = first && a2 >= a;
              inj += v3s[a2];
            }
            if (!first) continue;
#pragma unroll
            for (int t = 0; t < CPL; ++t)
              if (t == tc) v1[t] = __fmul_rn(CPL == 1 ? __fmaf_rn(__fmul_rn(th, tb0), inj, -K1[t]) : __fsub_rn(__fmul_rn(__fmul_rn(th, tb0), inj), K1[t]), rg[t]);
          }
        }
        // F_x v5 = F_u v3 - K1: sweep m + 1 = v1 - D^{-1} h (offdiag) (Phi' sweep m)
#pragma unroll
        for (int t = 0; t < CPL; ++t) y5[t] = v1[t];
        for (int sw = 1; sw < n_lo; ++sw) {
          // the neighbours' Phi' sweep, a product inside the lane rounded with
          // the sum where k_line's were
          float pw[CPL];
#pragma unroll
          for (int t = 0; t < CPL; ++t) pw[t] = __fmul_rn(dp[t], y5[t]);
          float lft = __shfl_up_sync(0xffffffffu, pw[CPL - 1], 1);
          float rgt = __shfl_down_sync(0xffffffffu, pw[0], 1);
          lft = (lane == 0) ? 0.0f : lft;
          rgt = (lane == 31) ? 0.0f : rgt;
#pragma unroll
          for (int t = 0; t < CPL; ++t) {
            const int tl = t > 0 ? t - 1 : 0, tr = t < CPL - 1 ? t + 1 : 0;
            const float l = t > 0 ? pw[tl] : lft, r = t < CPL - 1 ? pw[tr] : rgt;
            // (not the lane's first and last, which its neighbours read too)
            const bool fl = t - 1 >= 1 && t - 1 <= CPL - 2, fr = t + 1 <= CPL - 2;
            if (fl) ns[t] = __fmaf_rn(dp[tl], y5[tl], r);
            else if (fr) ns[t] = __fmaf_rn(dp[tr], y5[tr], l);
            else ns[t] = __fadd_rn(l, r);
          }
#pragma unroll
          for (int t = 0; t < CPL; ++t) y5[t] = __fmaf_rn(-rg[t], __fmul_rn(th, __fmul_rn(tcx, ns[t])), v1[t]);
        }
        // F_x^T v4 = -K3 - A_xx v5
#pragma unroll
        for (int t = 0; t < CPL; ++t) {
          w1[t] = __fmul_rn(__fmaf_rn(-ax[t], y5[t], -K3[t]), rg[t]);
          y4[t] = w1[t];
        }
        for (int sw = 1; sw < n_lo; ++sw) {
          li_nsum<CPL, float>(y4, ns, lane);
#pragma unroll
          for (int t = 0; t < CPL; ++t) y4[t] = __fmaf_rn(-rg[t], __fmul_rn(__fmul_rn(th, dp[t]), __fmul_rn(tcx, ns[t])), w1[t]);
        }
        if (it < n_u_it) {
          // A_uu v3 = K2 + F_u^T y_lambda (A_ux = 0)
          for (unsigned long long m = mine; m; m &= m - 1) {
            const int a = __ffsll((long long)m) - 1, tc = act[a] - q0;
            float y = y4[0];
#pragma unroll
            for (int t = 1; t < CPL; ++t) y = (t == tc) ? y4[t] : y;
            float k2 = b3;
            if (!one) k2 = (float)(I.h * (I.r * Us[a] + I.b0 * Lr[tc * 32]));
            v3s[a] = __fdiv_rn(__fmaf_rn(__fmul_rn(th, tb0), y, k2), auu);
          }
        }
      }
      // every lane has read the stage's controls (usum) before their owners
      // overwrite them
      __syncwarp();
      // ---- S_i <- S_i - alpha Delta s_i (float64) ----
#pragma unroll
      for (int t = 0; t < CPL; ++t) {
        const double x = Xr[t * 32];
        xp[t] = x;
        if (q0 + t < M) {
          Xr[t * 32] = fma(alpha, f2d(y5[t]), x);
          Lr[t * 32] = fma(alpha, f2d(y4[t]), Lr[t * 32]);
        }
      }
      for (unsigned long long m = mine; m; m &= m - 1) {
        const int a = __ffsll((long long)m) - 1;
        Us[a] -= alpha * (double)v3s[a];
      }
    }
    if (!publ) return;
    if constexpr (FULL) {
      for (int o = 16; o > 0; o >>= 1) {
        vmax = dmax_nan(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        vsq += __shfl_xor_sync(0xffffffffu, vsq, o);
      }
      publish((unsigned long long)__double_as_longlong(vmax), RES_FULL_MARK, vsq);
    } else {
      for (int o = 16; o > 0; o >>= 1) fs += __shfl_xor_sync(0xffffffffu, fs, o);
      // (as the bits of the floats that the norm and the bound are)
      publish(__float_as_uint(warp_max_nn(fmx)), __float_as_uint((float)e_max), f2d(fs));
    }
  };
  // the instance's norms: every warp reduces what all of them published (a
  // split pass's are floats widened: their maxima in two warp reductions)
  auto collect = [&](unsigned long long& r, unsigned long long& e, bool full) {
    r = e = 0ull;
    if (!full) {
      unsigned rf = 0u, ef = 0u;
      for (int w = lane; w < wt; w += 32) {
        rf = max(rf, (unsigned)red_r[w]);
        ef = max(ef, (unsigned)red_e[w]);
      }
      rf = __reduce_max_sync(0xffffffffu, rf);
      ef = __reduce_max_sync(0xffffffffu, ef);
      r = (unsigned long long)__double_as_longlong(f2d(__uint_as_float(rf)));
      e = (unsigned long long)__double_as_longlong(f2d(__uint_as_float(ef)));
      return;
    }
    for (int w = lane; w < wt; w += 32) {
      r = max(r, red_r[w]);
      e = max(e, red_e[w]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      r = max(r, __shfl_xor_sync(0xffffffffu, r, o));
      e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    }
  };

  int st = ST_RUNNING, k = 0, f64 = 0;
  double r0 = 0.0, r = 0.0;
  bool prev_full = false, again = false;
  const bool f0 = A.full0[b] != 0;
  for (;; ++k) {
    bool full = (k == A.max_iter) || (k == 0 && f0);
    if (k > 0) {
      unsigned long long rb, eb;
      collect(rb, eb, prev_full);
      r = __longlong_as_double((long long)rb);
      if (k == 1) r0 = r;
      if (threadIdx.x == 0) {  // read by later iterations' decisions
        hist_r[(k - 1) % RES_SLOTS] = rb;
        hist_e[(k - 1) % RES_SLOTS] = eb;
      }
      if (!prev_full && (!(r <= 1.79e308) || r > A.div_limit * fmax(r0, 1e-300))) {
        again = true;  // S^{k-1} is gone
        break;
      }
      full = full || switch_to_full(A, k, r, prev_full, eb,
                                    [&](int kk, double& r2, unsigned long long& e2) {
                                      r2 = __longlong_as_double((long long)hist_r[kk % RES_SLOTS]);
                                      e2 = hist_e[kk % RES_SLOTS];
                                    });
    }
    below();
    above();
    sync_all();
    if (full) {
      ++f64;
      stages(std::true_type{}, false, true);
      sync_all();
      unsigned long long rb, eb;
      collect(rb, eb, true);
      r = __longlong_as_double((long long)rb);
      if (k == 0) r0 = r;
      if (k == A.max_iter)
        st = (r <= A.tol) ? ST_CONVERGED : ((r <= 1.79e308) ? ST_MAX_ITER : ST_DIVERGED);
      else if (!(r <= 1.79e308) || r > A.div_limit * fmax(r0, 1e-300))
        st = ST_DIVERGED;
      else if (r <= A.tol)
        st = ST_CONVERGED;
      if (st != ST_RUNNING) break;
      below();
      sync_all();
      stages(std::true_type{}, true, false);
    } else {
      stages(std::false_type{}, true, true);
    }
    prev_full = full;
    sync_all();
  }
  if (again) {
    if (threadIdx.x == 0) atomicExch(retry, 1);
  } else {
    // S^k and its norms (the books of the solve)
    double* Xo = A.xout[0] + I.s_off;
    double* Lout = A.lout[0] + I.s_off;
    double* Uo = A.uout[0] + I.u_off;
    for (int s = a0; s < a1; ++s)
#pragma unroll
      for (int i = 0; i < CPL; ++i) {
        const int q = i * 32 + lane, p = (q % CPL) * 32 + q / CPL;
        if (q < M) {
          Xo[(long long)s * M + q] = X[(s - row0) * ROW + p];
          Lout[(long long)s * M + q] = Lm[(s - row0) * ROW + p];
        }
      }
    for (int s = a0; s < a1; ++s)
      for (int a = lane; a < nu; a += 32) Uo[(long long)s * nu + a] = U[(s - row0) * nu + a];
    if (rank == 0 && threadIdx.x == 0) {
      double q = 0.0;
      for (int w = 0; w < wt; ++w) q += red_q[w];
      A.status[b] = st;
      A.iters[b] = k;
      A.final_buf[b] = 0;
      A.fin_inf[b] = r;
      A.fin_2[b] = sqrt(q);
      A.f64_count[b] = f64;
      atomicSub(A.n_active, 1);
    }
  }
  // no CTA leaves while another may read its shared memory; the launch ends
  // after the launch before it (they overlap)
  sync_all();
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace nmpc_dev

namespace {

using nmpc_dev::InstDev;
using nmpc_dev::IterArgs;
using Kernel = void (*)(IterArgs, const int*, int, int, int, int*);

template <int NLO>
Kernel kernel_with(int cpl) {
  switch (cpl) {
    case 1: return nmpc_dev::k_line_inst<1, NLO>;
    case 2: return nmpc_dev::k_line_inst<2, NLO>;
    case 4: return nmpc_dev::k_line_inst<4, NLO>;
    default: return nmpc_dev::k_line_inst<8, NLO>;
  }
}
Kernel kernel_of(int cpl, int n_lo) { return n_lo == 2 ? kernel_with<2>(cpl) : kernel_with<0>(cpl); }

// Cells per lane, as on the line path: the smallest of 1, 2, 4, 8 that covers
// mx (at most 256) cells.
int li_cells_per_lane(int mx) { return mx <= 32 ? 1 : (mx <= 64 ? 2 : (mx <= 128 ? 4 : 8)); }

int rows_of(int N, int csize, int warps) {
  int rows = 0;
  for (int r = 0; r < csize; ++r)
    rows = std::max(rows, nmpc_dev::li_stage(r * warps + warps, csize * warps, N) -
                              nmpc_dev::li_stage(r * warps, csize * warps, N));
  return rows;
}

}  // namespace

std::vector<LineInstLaunch> line_inst_plan(const std::vector<InstDev>& inst,
                                           const std::vector<int>& which, int num_sms,
                                           int max_smem, std::vector<int>* list) {
  std::vector<LineInstLaunch> plan;
  list->clear();
  // few instances (their CTAs have a SM each): as many warps as stages, for
  // the shortest iteration; a batch: CTAs of which two or more share a SM, so
  // that one computes while the other waits at its barrier
  const int n = (int)which.size();
  // CTAs an instance may take for speed (256 cells, N = 60, us an iteration:
  // 20 instances on clusters of four 12.7, of two 21.6; 64 cells, N = 20, 76
  // instances 5.9 against 10.6 in the batch form).  Clusters of four fill 144
  // of 152 SMs; a 37th would wait for a place (24.7).
  int spread = 1;
  while (spread < 8 && n * spread * 2 <= num_sms - (spread > 1 ? num_sms / 19 : 0)) spread *= 2;
  auto most_warps = [](bool few, int cpl) {
    return few ? nmpc_dev::li_max_warps(cpl) : std::min(8, nmpc_dev::li_max_warps(cpl) / 2);
  };
  auto ctas_of = [&](bool few, int cpl, const InstDev& I) {  // 0: does not fit
    const size_t room = few ? (size_t)max_smem : std::min<size_t>(max_smem, 110 * 1024);
    for (int c = 1; c <= 8; c *= 2) {
      const int w = std::min(most_warps(few, cpl), (I.N + c - 1) / c);
      if (c * w > nmpc_dev::LI_MAX_WARPS) return 0;
      // few: at most four stages a SM, whose warps share its float64 pipe
      if (few && c < spread && c * 4 < I.N) continue;
      if (nmpc_dev::li_layout(cpl, rows_of(I.N, c, w), w, I.nu).bytes <= room) return c;
    }
    return 0;
  };
  // (cells per lane, CTAs, few) -> instances
  std::map<std::tuple<int, int, bool>, std::vector<int>> classes;
  for (int b : which) {
    const InstDev& I = inst[b];
    const int cpl = li_cells_per_lane(I.mx);
    int c = ctas_of(true, cpl, I);
    // (eight cells a lane and more stages than warps: 38 .. 72 instances of 256
    // cells, N = 60, 21.7 us, in the batch form 19.5 .. 20.3; with fewer cells a
    // lane more warps fit: 128 cells 15.0 against 17.7)
    const bool few = c > 0 && n * c <= num_sms &&
                     !(cpl == 8 && c > 1 && I.N > c * most_warps(true, cpl));
    if (!few) c = ctas_of(false, cpl, I);
    if (!c) return {};
    classes[{cpl, c, few}].push_back(b);
  }
  // Batch-form CTAs against one launch per iteration (us an iteration): a warp
  // here takes t_stage for each of its stages, k_line t_wave for 16 stages a SM.
  // The slowest instance's float64 iterations, which walk the stages twice, come
  // on top (a third with eight cells a lane and clusters, measured).  Few long
  // instances leave SMs without a CTA and their warps with many stages: N = 66, one
  // instance of 64 cells 28.9 against 10.1, N = 160, twelve of 32 cells 47 against
  // 10.9, N = 65, 40 of 256 cells 34 against 29; or the last wave of CTAs is nearly
  // empty: 76 of 256 cells, N = 66, 46.6 against 43 (72: 26.7 against 34).
  static const double t_stage[9] = {0, 2.3, 3.1, 0, 4.3, 0, 0, 0, 8.0};
  static const double t_wave[9] = {0, 8.5, 10, 0, 12, 0, 0, 0, 15.5};
  bool batch = false;
  double longest = 0, work = 0, stages = 0, by_launches = 0;
  for (auto it = classes.rbegin(); it != classes.rend(); ++it) {
    const int cpl = std::get<0>(it->first), c = std::get<1>(it->first);
    std::vector<int>& v = it->second;
    std::stable_sort(v.begin(), v.end(), [&](int a, int b) { return inst[a].N > inst[b].N; });
    LineInstLaunch L{cpl, c, 0, (int)list->size(), (int)v.size(), 0, 0, 0};
    L.warps = std::min(most_warps(std::get<2>(it->first), cpl), (inst[v[0]].N + c - 1) / c);
    int rows = 0, nu = 0;
    for (int b : v) {
      rows = std::max(rows, rows_of(inst[b].N, c, L.warps));
      nu = std::max(nu, inst[b].nu);
      list->push_back(b);
    }
    L.rows = rows;
    L.nu = nu;
    L.smem = nmpc_dev::li_layout(cpl, rows, L.warps, nu).bytes;
    if (L.smem > (size_t)max_smem) return {};
    plan.push_back(L);
    const bool few = std::get<2>(it->first);
    batch = batch || !few;
    const int sms = num_sms - (c > 2 ? num_sms / 19 : 0);
    const double t = (rows + L.warps - 1) / L.warps * t_stage[cpl];
    double waves = (double)L.n * c / (few ? sms : 2 * sms);
    // (CTAs of one length: 1.06, 1.4, 2.1 and 4.2 waves of them take 1.7, 1.8, 2.7
    // and 4.7 times one; a slow instance prolongs a second wave that has begun)
    if (classes.size() == 1) waves = waves > 1.0 ? waves + 0.55 : 1.0;
    longest = std::max(longest, t * (cpl == 8 && c > 1 ? 1.35 : 1.1));
    work += waves * t * (classes.size() == 1 && waves > 1.0 && waves < 2.0 ? 1.25 : 1.05);
    for (int b : v) {
      stages += inst[b].N;
      by_launches += inst[b].N * t_wave[cpl];
    }
  }
  if (batch) {
    by_launches *= std::ceil(stages / (16.0 * num_sms)) / stages;
    if (std::max(longest, work) > by_launches) {
      list->clear();
      return {};
    }
  }
  return plan;
}

// Every kernel may use all of a CTA's shared memory (the attribute is the
// function's, whichever handle launches it).
cudaError_t line_inst_configure(int max_smem) {
  for (int cpl = 1; cpl <= 8; cpl *= 2) {
    for (int n_lo = 1; n_lo <= 2; ++n_lo) {
      const cudaError_t e = cudaFuncSetAttribute(
          kernel_of(cpl, n_lo), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

cudaError_t line_inst_solve(const std::vector<LineInstLaunch>& plan, const IterArgs& A,
                            const int* list_d, int* retry, cudaStream_t st) {
  for (size_t i = 0; i < plan.size(); ++i) {
    const LineInstLaunch& L = plan[i];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(L.n * L.csize));
    cfg.blockDim = dim3((unsigned)(32 * L.warps));
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int na = 0;
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = (unsigned)L.csize;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
    if (i > 0) {  // its CTAs start as those of the launch before have all started
      attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[na].val.programmaticStreamSerializationAllowed = 1;
      ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel_of(L.cpl, A.n_lo), A, list_d + L.first, L.csize,
                                             L.rows, L.nu, retry);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
