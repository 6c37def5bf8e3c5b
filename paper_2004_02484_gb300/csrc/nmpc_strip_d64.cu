// Kernels of the strip path for batches of stages that would also fit a
// cluster: the two-column strips with the cluster path's split residual (D64)
// and the actuator patches that go with them (a translation unit of its own:
// they compile beside the other kernels).
#include "nmpc_core.cuh"
#include "nmpc_strip_d64.h"

namespace nmpc_dev {
#include "nmpc_patch.cuh"

// v3 of two actuators per warp, one per half: the u fixed-point iteration of
// Sec. 5.2 (eqs. 22-24) in the full-field form's own order, on the cells
// within 2 (n_lo - 1) grid steps of the actuator (13 for n_lo = 2), lane q of
// a half holding cell q.  No other actuator's cell is among them (the host
// checks), so v3 comes out as the cluster path's, operation by operation.
// k_patch computes a square of 49 cells, four of five of which its single
// result does not depend on, and a second right-hand side.
// Cell q of the diamond: itself, its four neighbours, the eight at two steps.
__constant__ signed char diamond_x[13] = {0, -1, 1, 0, 0, -2, 2, 0, 0, -1, 1, -1, 1};
__constant__ signed char diamond_y[13] = {0, 0, 0, -1, 1, 0, 0, -2, 2, -1, -1, 1, 1};
// the cells of the left, right, upper and lower neighbours of cells 0 .. 4
__constant__ signed char diamond_n[5][4] = {
    {1, 2, 3, 4}, {5, 0, 9, 11}, {0, 6, 10, 12}, {9, 10, 7, 0}, {11, 12, 0, 8}};

template <int n_lo>
__global__ void __launch_bounds__(128) k_patch_d64(IterArgs A, int MODE, int j) {
  const int lane = threadIdx.x & 31, q = lane & 15, base = lane & 16;
  pdl_trigger();
  const int k = (MODE == MODE_SOLVE) ? *(volatile int*)A.iter_k + launch_iter(A, j) : 0;
  const int half = launch_half(A, j);
  const int rd = (MODE == MODE_SOLVE) ? (k & 1) : 0;
  pdl_wait();
  if (MODE == MODE_SOLVE && A.n_tail > 0 && blockIdx.x == 0 && threadIdx.x == 0)
    *A.strip_run = *(volatile int*)A.n_active;
  const int first = (A.rb && half) ? A.n_patches_even : 0;
  const int end = A.rb ? (half ? A.n_patches : A.n_patches_even) : A.n_patches;
  const int item = first + (blockIdx.x * 128 + (int)threadIdx.x) / 16;
  const bool on = item < end;
  if (!__any_sync(0xffffffffu, on)) return;
  const int4 it = A.patches[on ? item : end - 1];
  const int b = it.x, s = it.y, a = it.z;
  bool run = on, full = false;
  if (MODE == MODE_SOLVE) {
    const Decision d = decide(A, b, k);
    run = run && !d.skip && k != A.max_iter;  // a residual-only iteration needs no v3
    full = d.full != 0;
  } else {
    full = A.full_all != 0;
  }
  if (!__any_sync(0xffffffffu, run)) return;
  const InstDev& I = A.inst[b];
  const int mx = I.mx, my = I.my;
  const bool last = (s == I.N - 1);
  const int ca = A.act[I.act_off + a], ay = ca / mx, ax = ca - ay * mx;
  const int qc = q < 13 ? q : 0;
  const int gx = ax + diamond_x[qc], gy = ay + diamond_y[qc];
  const bool in = gx >= 0 && gx < mx && gy >= 0 && gy < my;
  const long long so = I.s_off + (long long)s * I.ng;
  const double* Xg = A.xin[rd] + so;
  const double* Lg = A.lin[rd] + so;
  // red-black half 1: x_{i-1}, lambda_{i+1} as updated by half 0
  const bool rbn = A.rb && half == 1;
  const double* XPg = (s == 0) ? A.x0 + I.g_off : (rbn ? A.xout[rd ^ 1] : A.xin[rd]) + so - I.ng;
  const double* LNg = (rbn ? A.lout[rd ^ 1] : A.lin[rd]) + so + I.ng;
  const int c = in ? gy * mx + gx : 0;
  // a field at the cell and its four neighbours (zero outside the grid)
  struct Star {
    double m, l, r, u, d;
  };
  auto star = [&](const double* f) {
    Star v;
    v.m = in ? f[c] : 0.0;
    v.l = in && gx > 0 ? f[c - 1] : 0.0;
    v.r = in && gx < mx - 1 ? f[c + 1] : 0.0;
    v.u = in && gy > 0 ? f[c - mx] : 0.0;
    v.d = in && gy < my - 1 ? f[c + mx] : 0.0;
    return v;
  };
  const Star x = star(Xg), lm = star(Lg);
  const double xp = in ? XPg[c] : 0.0, ln = in && !last ? LNg[c] : 0.0;
  const double rc = in ? A.ref[I.g_off + c] : 0.0;
  const double ua = A.uin[rd][I.u_off + (long long)s * I.nu + a];
  const bool centre = q == 0;
  float K1, K3, dp, axx;
  if (full) {
    const double k0 = I.k0, k1 = I.k1, h = I.h;
    auto phi = [&](double w) { return k0 * (w + 0.5 * k1 * w * w); };
    const double lphi = I.cx * (phi(x.l) + phi(x.r)) + I.cy * (phi(x.u) + phi(x.d)) - I.dcoef * phi(x.m);
    const double mu = I.cx * (lm.l + lm.r) + I.cy * (lm.u + lm.d) - I.dcoef * lm.m;
    const double dphi = k0 * (1.0 + k1 * x.m);
    const double s1 = lphi + (centre ? I.b0 * ua : 0.0);
    const double s3 = I.q * (x.m - rc) + dphi * mu;
    const double lnx = last ? I.hqf * (x.m - rc) : ln;
    K1 = d2f(__fma_rn(h, s1, xp - x.m));
    K3 = d2f(__fma_rn(h, s3, lnx - lm.m));
    dp = d2f(dphi);
    axx = d2f(h * (I.q + k0 * k1 * mu) + (last ? I.hqf : 0.0));
  } else {
    const float fk0 = I.fk0, fk1h = I.fk1h, fcx = I.fcx, fcy = I.fcy, fdc = I.fdc;
    auto phi = [&](double w) {
      const float v = d2f(w);
      return __fmul_rn(fk0, __fmaf_rn(__fmul_rn(fk1h, v), v, v));
    };
    auto lap = [&](float m, float l, float r, float u, float d) {
      return __fmaf_rn(-fdc, m,
                       __fmaf_rn(fcx, __fadd_rn(l, r), __fmul_rn(fcy, __fadd_rn(u, d))));
    };
    const float xv = d2f(x.m), rv = d2f(rc);
    const float lphi = lap(phi(x.m), phi(x.l), phi(x.r), phi(x.u), phi(x.d));
    const float mu = lap(d2f(lm.m), d2f(lm.l), d2f(lm.r), d2f(lm.u), d2f(lm.d));
    dp = __fmul_rn(fk0, __fmaf_rn(I.fk1, xv, 1.0f));
    const float s1 = __fmaf_rn(I.fb0, centre ? d2f(ua) : 0.0f, lphi);
    const float dr = __fsub_rn(xv, rv);
    const float s3 = __fmaf_rn(dp, mu, __fmul_rn(I.fq, dr));
    const float hqff = last ? I.fhqf : 0.0f;
    K1 = __fmaf_rn(I.fh, s1, d2f(xp - x.m));
    K3 = __fmaf_rn(I.fh, s3, d2f(ln - lm.m));
    if (last) K3 = __fadd_rn(K3, __fmul_rn(hqff, dr));
    axx = __fmaf_rn(I.fh, __fmaf_rn(I.fk01, mu, I.fq), hqff);
  }
  const float th = I.fh, tb0 = I.fb0, tcx = I.fcx, tcy = I.fcy, auu = I.fauu;
  auto sub_prod = [](float v, float r, float off) { return __fmaf_rn(-r, off, v); };
  const float rg = in && q < 13 ? __frcp_rn(sub_prod(-1.0f, __fmul_rn(th, I.fdc), dp)) : 0.0f;
  const float b3 = (float)(I.h * (I.r * ua + I.b0 * lm.m));
  auto nsum = [&](float v) {  // over the neighbours, at the cells 0 .. 4
    const int qq = q < 5 ? q : 0;
    const float l = __shfl_sync(0xffffffffu, v, base + diamond_n[qq][0]);
    const float r = __shfl_sync(0xffffffffu, v, base + diamond_n[qq][1]);
    const float u = __shfl_sync(0xffffffffu, v, base + diamond_n[qq][2]);
    const float d = __shfl_sync(0xffffffffu, v, base + diamond_n[qq][3]);
    return __fmaf_rn(tcx, __fadd_rn(l, r), __fmul_rn(tcy, __fadd_rn(u, d)));
  };
  float v1 = __fmul_rn(-K1, rg), v3 = 0.0f;
  for (int n = 0; n < A.n_u_it; ++n) {
    if (n > 0 && centre)
      v1 = __fmul_rn(__fmaf_rn(__fmul_rn(th, tb0), v3, -K1), rg);
    float v5 = v1;
    if constexpr (n_lo > 1) v5 = sub_prod(v1, rg, __fmul_rn(th, nsum(__fmul_rn(dp, v1))));
    const float w1 = __fmul_rn(sub_prod(-K3, axx, v5), rg);
    float v4 = w1;
    if constexpr (n_lo > 1) v4 = sub_prod(w1, rg, __fmul_rn(__fmul_rn(th, dp), nsum(w1)));
    v3 = __fdiv_rn(__fmaf_rn(__fmul_rn(th, tb0), v4, b3), auu);
  }
  if (centre && run) A.v3g[I.u_off + (long long)s * I.nu + a] = (double)v3;
}
}  // namespace nmpc_dev

using nmpc_dev::k_strip2;

StripKernel strip_d64_kernel(int n_lo, bool rbn, bool full_width) {
  if (n_lo <= 1) {
    if (full_width) return rbn ? k_strip2<1, true, true, true> : k_strip2<1, false, true, true>;
    return rbn ? k_strip2<1, true, true, false> : k_strip2<1, false, true, false>;
  }
  if (full_width) return rbn ? k_strip2<2, true, true, true> : k_strip2<2, false, true, true>;
  return rbn ? k_strip2<2, true, true, false> : k_strip2<2, false, true, false>;
}

StripKernel patch_d64_kernel(int n_lo) {
  return n_lo <= 1 ? nmpc_dev::k_patch_d64<1> : nmpc_dev::k_patch_d64<2>;
}
