// Second-order-in-time solver (include/nmpc_wave.h): the double-layer method
// on a w_tt + b w_t = c Lap w - kappa w^3 + point forces (Sec. 2, eq. 1 with
// a != 0), state x = (W, V = dW/dt) (eq. 5).
//
// One launch of k_wave_dir is one iteration (two with the red-black upper
// layer: half 0 the even stages, half 1 the odd ones with the even
// neighbours' new x_{i-1}, lambda_{i+1} in the right-hand side, eq. 18's
// form).  A group of threads per (instance, stage), one or two points a
// thread: K_i (eq. 9) and its norms, the stage's coefficients, and the lower
// layer (eqs. 21-24 with the u-iteration of Sec. 5.2) whose F_x and F_x^T
// solves eliminate v6 (eq. 25): E v7 = b7 + h grad_W g b6 and E^T v9 = b9 +
// h b8 by n_lo pointwise Jacobi sweeps, v6 = h v7 - b6, v8 = h grad_W g^T v9
// - b8; then S^{k+1} = S^k - Delta S (no bounds: the full step).
// grad_W g = (c L - 3 kappa diag(W^2)) / a and grad_V g = -(b / a) I, so E
// has the stencil of L scaled by h^2 c / a off the diagonal.
#include <new>

#include "../../include/nmpc_wave.h"
#include "stage_driver.cuh"

namespace wave_dev {

using stage_drv::Ctl;
using stage_drv::Iter;
using stage_drv::Layout;
constexpr int THREADS = 256;
constexpr int MAX_NU = 64;
constexpr int NG_PER_THREAD = (NMPC_WAVE_MAX_POINTS + THREADS - 1) / THREADS;  // the plant's points

struct WInst {
  int dim, m, ng, nu, N, neu;
  long long w_off;  // w_ref
  long long a_off;  // u_ref, actuator table
  long long t_off;  // per-point tables
  double h, a, b, c, kappa, gain, q, qv, r, qf, gamma;
  double lw;        // the Laplacian's neighbour weight 1 / spacing^2
  // derived (the float64 pipe is the scarce one): 1 / a; c lw / a; kappa / a;
  // b / a; gain / a; h^2 c lw / a; E's diagonal at W = 0 and its 3 h^2;
  // h gain / a; h r + gamma and 1 / that
  double ia, cl, kia, bia, gia, se, ed0, hh3, fu, auu, rauu;
  float fauu, frauu;  // the last two in float32 (a conversion runs on the float64 pipe)
};

// The derived fields.
inline void derive(WInst& I) {
  const double d2 = 2.0 * I.dim;
  I.ia = 1.0 / I.a;
  I.cl = I.c * I.ia * I.lw;
  I.kia = I.kappa * I.ia;
  I.bia = I.b * I.ia;
  I.gia = I.gain * I.ia;
  I.se = I.h * I.h * I.cl;
  I.ed0 = -(1.0 + I.h * I.bia) - d2 * I.se;
  I.hh3 = 3.0 * I.h * I.h;
  I.fu = I.h * I.gia;
  I.auu = I.h * I.r + I.gamma;
  I.rauu = 1.0 / I.auu;
  I.fauu = (float)I.auu;
  I.frauu = 1.0f / I.fauu;
}

struct WArgs {
  const WInst* inst;
  const int* act_of;  // [sum ng]: actuator index at the point, or -(grid steps to the nearest one)
  const double* x0;
  const double* wref;
  const double* uref;
  int n_lo, n_u_it, rb, half;
};

// Shared memory of one stage: W and the (scaled) lambda_V in float64, two
// exchange fields of the lower layer's type; each with a zero at index ng.
template <typename T>
__host__ __device__ constexpr size_t stage_bytes(int ng) {
  return (((size_t)(ng + 1) * (2 * sizeof(double) + 2 * sizeof(T))) + 15) & ~size_t(15);
}

// What bounds it: the float64 pipe (2 lanes a clock a SM; the residual, the
// coefficients and, in NMPC_FP64, the lower layer run there), so the layout
// saves float64 instructions first.  A thread keeps its points' rows and
// coefficients in registers and exchanges only the field that a stencil reads
// (one barrier each, two alternating buffers); neighbours are found from the
// grid (4 additions and one multiply-add a stencil, where a table of five
// weights cost five multiply-adds and ten loads); the diagonal's reciprocal is
// taken once a point (a division each sweep before); h grad_W g b6 is common
// to every u-iteration, v8 is needed by the last one only; the maximum norm
// is taken on integers.  With n_lo = 2 the u-iterations after the first
// recompute only the points that a control can reach (2 grid steps for v9):
// all others keep the bits that they would get again.  256 membranes of
// 32x32, N = 10, float64: 81.0 -> 25.9 ms a solve (float64 pipe 85% busy; two
// points a thread in 64 registers, 512 threads and two CTAs a SM, with 344 bytes
// of spills); 256 strings of 64 points, N = 20, mixed, red-black: 21.2 -> 4.6 ms
// (one point a thread, no spills, four stages a CTA, 76%).
// The lower layer runs in T: float64, or float32 in mixed precision (the
// residual, the coefficients and the update stay float64, so the fixed point
// is the float64 root).
template <typename T, int PPT, bool NEU, bool D2>
__global__ void __launch_bounds__(PPT == 1 ? 256 : 512, PPT == 1 ? 3 : 2)
    k_wave_dir(WArgs A, Ctl C, Iter S, stage_drv::Range R) {
  extern __shared__ __align__(16) double smem[];
  __shared__ stage_drv::WarpNorms red[16];
  __shared__ T sK2[8 * MAX_NU], sV3[8 * MAX_NU];  // per control, by its point's thread only
  stage_drv::pdl_trigger();
  const int g = threadIdx.x / R.tps, t = threadIdx.x - g * R.tps;
  const int item = blockIdx.x * R.spc + g;
  stage_drv::pdl_wait();
  if (item >= R.n) return;
  const int2 it = C.work[R.first + item];
  const int b = it.x, s = it.y;
  bool norms_only;
  if (!stage_drv::begin_stage(C, b, s, t, norms_only)) return;
  const WInst& I = A.inst[b];
  const Layout& Ly = C.lay[b];
  const int ng = I.ng, nu = I.nu, nx = 2 * ng;
  const bool last = (s == I.N - 1);
  // this launch's stage size sets the fields' distance (ng_max would do too)
  double* fA = smem + (size_t)g * (stage_bytes<T>(R.ng_max) / sizeof(double));
  double* fB = fA + (ng + 1);
  T* fC = reinterpret_cast<T*>(fB + (ng + 1));
  T* fD = fC + (ng + 1);
  const int* act_of = A.act_of + I.t_off;
  const long long so = Ly.s_off + (long long)s * nx;
  const long long uo = Ly.u_off + (long long)s * nu;
  const double h = I.h;
  constexpr double d2 = D2 ? 4.0 : 2.0;  // the Laplacian's centre: -2 dim lw
  const bool gs = A.rb && A.half == 1;

  stage_drv::Nbr<NEU, D2> nb[PPT];
  int ap[PPT];
  bool on[PPT];
  if (t == 0) {
    fA[ng] = fB[ng] = 0.0;
    fC[ng] = fD[ng] = T(0);
  }
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    const int p = t + j * R.tps;
    on[j] = p < ng;
    nb[j].set(p, I.m, ng);
    ap[j] = on[j] ? act_of[p] : -0x7fffffff;
    if (on[j]) {
      fA[p] = __ldcg(S.xin + so + p);
      fB[p] = nb[j].scale(__ldcg(S.lin + so + ng + p));
    }
  }
  stage_drv::group_sync(g, R.tps);

  // K_i (eq. 9), coefficients, norms
  unsigned long long mx = 0ull;
  double sq = 0.0;
  T k1w[PPT], r7[PPT], k3w[PPT], k3v[PPT], rED[PPT], axw[PPT], kw3[PPT];
  const double cl = I.cl, bia = I.bia, hqf = last ? h * I.qf : 0.0;
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    const int p = t + j * R.tps;
    k1w[j] = r7[j] = k3w[j] = k3v[j] = rED[j] = axw[j] = kw3[j] = T(0);
    if (!on[j]) continue;
    const double w = fA[p], lv = nb[j].unscale(fB[p]);
    const double v = __ldcg(S.xin + so + ng + p), lw = __ldcg(S.lin + so + p);
    const double wr = A.wref[I.w_off + p];
    const double* prev = (s == 0) ? A.x0 + Ly.g_off + p : S.xin + so - nx + p;
    const double wp = __ldcg(prev), vp = __ldcg(prev + ng);
    const double dw = w - wr;
    const double lwn = last ? hqf * dw : __ldcg(S.lin + so + nx + p);
    const double lvn = last ? 0.0 : __ldcg(S.lin + so + nx + ng + p);
    const double lap = nb[j].sum(fA) - d2 * w;             // (L W)(p) / lw
    const double lapt = nb[j].unscale(nb[j].sum(fB)) - d2 * lv;  // (L^T lambda_V)(p) / lw
    const double kw = I.kia * w, kww = kw * w;
    double gg = cl * lap - bia * v - kww * w;
    double u = 0.0;
    if (ap[j] >= 0) {
      u = __ldcg(S.uin + uo + ap[j]);
      gg += I.gia * u;
    }
    const double K1W = wp - w + h * v;
    const double K1V = vp - v + h * gg;
    const double kww3 = 3.0 * kww;
    const double K3W = lwn - lw + h * (I.q * dw + (cl * lapt - kww3 * lv));
    const double K3V = lvn - lv + h * (I.qv * v + lw - bia * lv);
    mx = max(mx, max(max(stage_drv::abs_bits(K1W), stage_drv::abs_bits(K1V)),
                     max(stage_drv::abs_bits(K3W), stage_drv::abs_bits(K3V))));
    sq += K1W * K1W + K1V * K1V + K3W * K3W + K3V * K3V;
    if (ap[j] >= 0) {
      const double K2 = h * (I.r * (u - A.uref[I.a_off + ap[j]]) + I.gia * lv);
      mx = max(mx, stage_drv::abs_bits(K2));
      sq += K2 * K2;
      sK2[g * MAX_NU + ap[j]] = (T)K2;
      sV3[g * MAX_NU + ap[j]] = T(0);
    }
    // red-black half 1: the right-hand side takes the even neighbours' new
    // x_{i-1}, lambda_{i+1} (half 0 has written them to the other buffer);
    // the norms above stay those of K(S^k)
    double c1w = K1W, c1v = K1V, c3w = K3W, c3v = K3V;
    if (gs) {
      if (s > 0) {
        c1w += __ldcg(S.xout + so - nx + p) - wp;
        c1v += __ldcg(S.xout + so - nx + ng + p) - vp;
      }
      if (!last) {
        c3w += __ldcg(S.lout + so + nx + p) - lwn;
        c3v += __ldcg(S.lout + so + nx + ng + p) - lvn;
      }
    }
    k1w[j] = (T)c1w;
    r7[j] = (T)c1v;
    k3w[j] = (T)c3w;
    k3v[j] = (T)c3v;
    kw3[j] = (T)kww3;
    // E's diagonal: h grad_V g - 1 + h^2 grad_W g at (p, p)
    rED[j] = stage_drv::rcp((T)(I.ed0 - I.hh3 * kww));
    axw[j] = (T)(h * (I.q - 6.0 * kw * lv) + hqf);
    fD[p] = k1w[j];
  }
  stage_drv::warp_norms(mx, sq, red);
  stage_drv::group_sync(g, R.tps);
  if (t == 0) stage_drv::publish_norms(C, b, red, R.tps);
  if (norms_only) return;

  // u fixed-point iteration (Sec. 5.2) on the direction y = P^{-1}(K_1 - F_u
  // v3, K_3): v3 = (K_2 - F_u^T y_lambda) / A_uu from v3 = 0, then the last y.
  // F_u = [0; h B / a]; A_uu = h r + gamma.
  const T hT = (T)h, clT = (T)cl, sT = (T)I.se, d2T = (T)d2, axv = (T)(h * I.qv);
  const T fu = (T)I.fu;
  const T auu = sizeof(T) == 4 ? I.fauu : I.auu, rauu = sizeof(T) == 4 ? I.frauu : I.rauu;
#pragma unroll
  for (int j = 0; j < PPT; ++j)  // K1V + h grad_W g K1W
    r7[j] += hT * (clT * (nb[j].sum(fD) - d2T * k1w[j]) - kw3[j] * k1w[j]);
  T v7[PPT], t9[PPT], v9[PPT];
#pragma unroll
  for (int j = 0; j < PPT; ++j) v7[j] = t9[j] = v9[j] = T(0);
  const int n_lo = A.n_lo;
  T *ex = fC, *ex2 = fD;  // the next exchange's field, the other one
  for (int itu = 0; itu <= A.n_u_it; ++itu) {
    // the points that this u-iteration can change: all of them at first; with
    // n_lo = 2 the two fields hold the same sweeps every time (C the first
    // of E, D the first of E^T), so later ones store and recompute the points
    // at most 0, 1, 2 grid steps from an actuator
    const int near0 = (itu == 0 || n_lo != 2) ? 0x7fffffff : 0;
    const int near1 = near0 ? near0 : 1, near2 = near0 ? near0 : 2;
    T rhs[PPT], c[PPT];
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      rhs[j] = ap[j] >= 0 ? r7[j] - fu * sV3[g * MAX_NU + ap[j]] : r7[j];
      c[j] = rhs[j] * rED[j];
    }
    for (int sw = 1; sw < n_lo; ++sw) {  // E v7 = r7 - F_u v3
#pragma unroll
      for (int j = 0; j < PPT; ++j)
        if (on[j] && -ap[j] <= near0) ex[t + j * R.tps] = c[j];
      stage_drv::group_sync(g, R.tps);
#pragma unroll
      for (int j = 0; j < PPT; ++j)
        if (-ap[j] <= near1) c[j] = (rhs[j] - sT * nb[j].sum(ex)) * rED[j];
      T* x = ex;
      ex = ex2;
      ex2 = x;
    }
#pragma unroll
    for (int j = 0; j < PPT; ++j)
      if (-ap[j] <= near1) {
        v7[j] = c[j];
        const T v6 = hT * c[j] - k1w[j];
        t9[j] = (k3v[j] - axv * c[j]) + hT * (k3w[j] - axw[j] * v6);
        c[j] = t9[j] * rED[j];
      }
    for (int sw = 1; sw < n_lo; ++sw) {  // E^T v9 = b9 + h b8
#pragma unroll
      for (int j = 0; j < PPT; ++j)
        if (on[j] && -ap[j] <= near1) ex[t + j * R.tps] = nb[j].scale(c[j]);
      stage_drv::group_sync(g, R.tps);
#pragma unroll
      for (int j = 0; j < PPT; ++j)
        if (-ap[j] <= near2) c[j] = (t9[j] - sT * nb[j].unscale(nb[j].sum(ex))) * rED[j];
      T* x = ex;
      ex = ex2;
      ex2 = x;
    }
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      if (-ap[j] <= near2) v9[j] = c[j];
      // (the controls that are stored: a corrected quotient; with the product
      // alone their rms error of an iteration was 1.1 to 1.25 times that of
      // divisions.  The diagonal's keeps the product, whose errors are those of a
      // division.)
      if (itu < A.n_u_it && ap[j] >= 0) {
        const T b = sK2[g * MAX_NU + ap[j]] - fu * v9[j];
        sV3[g * MAX_NU + ap[j]] = itu == A.n_u_it - 1 ? stage_drv::quot(b, auu, rauu) : b * rauu;
      }
    }
  }
  // v8 = h grad_W g^T v9 - b8, and S^{k+1} = S^k - (v5, v3, v4)
#pragma unroll
  for (int j = 0; j < PPT; ++j)
    if (on[j]) ex[t + j * R.tps] = nb[j].scale(v9[j]);
  stage_drv::group_sync(g, R.tps);
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    const int p = t + j * R.tps;
    if (!on[j]) continue;
    const T gwt = clT * (nb[j].unscale(nb[j].sum(ex)) - d2T * v9[j]) - kw3[j] * v9[j];
    const T v6 = hT * v7[j] - k1w[j];
    const T v8 = hT * gwt - (k3w[j] - axw[j] * v6);
    S.xout[so + p] = fA[p] - (double)v6;
    S.xout[so + ng + p] = __ldcg(S.xin + so + ng + p) - (double)v7[j];
    S.lout[so + p] = __ldcg(S.lin + so + p) - (double)v8;
    S.lout[so + ng + p] = nb[j].unscale(fB[p]) - (double)v9[j];
    if (ap[j] >= 0)
      S.uout[uo + ap[j]] = __ldcg(S.uin + uo + ap[j]) - (double)sV3[g * MAX_NU + ap[j]];
  }
}

// (L v)(p) over a stage's grid, one axis after the other.
__device__ __forceinline__ double lap_at(const WInst& I, const double* v, int p) {
  double acc = -2.0 * I.dim * v[p];
  for (int axis = 0; axis < I.dim; ++axis) {
    const int st = axis ? I.m : 1, i = axis ? p / I.m : p % I.m;
    const bool lo = i > 0, hi = i < I.m - 1;
    if (I.neu) {  // the mirrored point
      acc += v[lo ? p - st : p + st] + v[hi ? p + st : p - st];
    } else {
      acc += (lo ? v[p - st] : 0.0) + (hi ? v[p + st] : 0.0);
    }
  }
  return I.lw * acc;
}

// The plant (Sec. 5.3): the true system x = (W, V) (device [sum 2 n_g], in
// place) advances by n_sub symplectic Euler steps of tau = dt / n_sub (dt < 0:
// each instance's own stage length h) with the inputs at the first-stage
// values u1 of the current state: V <- V + tau g(W, V, u1), then W <- W + tau
// V.  One CTA per instance; W, V and the forces in shared memory.
__global__ void __launch_bounds__(THREADS) k_wave_plant(WArgs A, const Layout* lay, double* x,
                                                        const double* uc, double dt, int n_sub) {
  const int b = blockIdx.x;
  const WInst I = A.inst[b];
  const Layout Ly = lay[b];
  const int ng = I.ng;
  extern __shared__ double smem[];
  double* W = smem;
  double* V = W + ng;
  double* F = V + ng;
  const int* act_of = A.act_of + I.t_off;
  for (int p = threadIdx.x; p < ng; p += THREADS) {
    W[p] = x[Ly.g_off + p];
    V[p] = x[Ly.g_off + ng + p];
    const int ap = act_of[p];
    F[p] = ap >= 0 ? I.gain * uc[Ly.u_off + ap] : 0.0;
  }
  __syncthreads();
  const double tau = (dt < 0.0 ? I.h : dt) / n_sub, ia = 1.0 / I.a;
  for (int k = 0; k < n_sub; ++k) {
    double vn[NG_PER_THREAD];
    int cnt = 0;
    for (int p = threadIdx.x; p < ng; p += THREADS, ++cnt) {
      const double w = W[p];
      const double g = (I.c * lap_at(I, W, p) - I.b * V[p] - I.kappa * w * w * w + F[p]) * ia;
      vn[cnt] = V[p] + tau * g;
    }
    __syncthreads();
    cnt = 0;
    for (int p = threadIdx.x; p < ng; p += THREADS, ++cnt) {
      V[p] = vn[cnt];
      W[p] += tau * vn[cnt];
    }
    __syncthreads();
  }
  for (int p = threadIdx.x; p < ng; p += THREADS) {
    x[Ly.g_off + p] = W[p];
    x[Ly.g_off + ng + p] = V[p];
  }
}

}  // namespace wave_dev

using wave_dev::WArgs;
using wave_dev::WInst;

struct nmpc_wave {
  nmpc_wave_opts opts{};
  std::vector<WInst> inst_h;
  stage_drv::Driver drv;
  long long n_a = 0, n_w = 0;  // sum n_u, sum n_g
  int ng_max = 0;
  WInst* inst_d = nullptr;
  int* act_of = nullptr;
  double *wref = nullptr, *uref = nullptr;
};

namespace {

void free_wave(nmpc_wave* h) {
  stage_drv::driver_free(h->drv);
  void* ptrs[] = {h->inst_d, h->act_of, h->wref, h->uref};
  for (void* p : ptrs)
    if (p) cudaFree(p);
}

int validate(const nmpc_wave_desc& d) {
  if ((d.dim != 1 && d.dim != 2) || d.horizon < 1 || d.n_u < 1 || !d.act_cell) return NMPC_ERR_BAD_ARG;
  if (d.bc != 0 && d.bc != 1) return NMPC_ERR_BAD_ARG;
  if (d.m < (d.bc == 0 ? 3 : 1)) return NMPC_ERR_BAD_ARG;
  const long long ng = d.dim == 2 ? (long long)d.m * d.m : d.m;
  if (ng > NMPC_WAVE_MAX_POINTS || d.n_u > wave_dev::MAX_NU) return NMPC_ERR_UNSUPPORTED;
  std::vector<char> seen(ng, 0);
  for (int a = 0; a < d.n_u; ++a) {
    if (d.act_cell[a] < 0 || d.act_cell[a] >= ng || seen[d.act_cell[a]]) return NMPC_ERR_BAD_ARG;
    seen[d.act_cell[a]] = 1;
  }
  if (!(d.h > 0) || !(d.a > 0) || !std::isfinite(d.b) || !std::isfinite(d.c) ||
      !std::isfinite(d.kappa) || !std::isfinite(d.gain) || !(d.q >= 0) || !(d.qv >= 0) ||
      !(d.r > 0) || !(d.qf >= 0) || !(d.gamma >= 0))
    return NMPC_ERR_BAD_ARG;
  return NMPC_OK;
}

WArgs make_args(const nmpc_wave* h) {
  WArgs A{};
  A.inst = h->inst_d;
  A.act_of = h->act_of;
  A.x0 = h->drv.x0;
  A.wref = h->wref;
  A.uref = h->uref;
  A.n_lo = h->opts.n_lo;
  A.n_u_it = h->opts.n_u_it;
  A.rb = (h->opts.variant == NMPC_VARIANT_REDBLACK) ? 1 : 0;
  return A;
}

// k_wave_dir for a group of stages.
using DirKernel = void (*)(WArgs, stage_drv::Ctl, stage_drv::Iter, stage_drv::Range);
template <typename T, int PPT>
DirKernel dir_kernel_of(bool neu, bool d2) {
  if (neu) return d2 ? wave_dev::k_wave_dir<T, PPT, true, true> : wave_dev::k_wave_dir<T, PPT, true, false>;
  return d2 ? wave_dev::k_wave_dir<T, PPT, false, true> : wave_dev::k_wave_dir<T, PPT, false, false>;
}
DirKernel dir_kernel(bool mixed, const stage_drv::Group& g) {
  if (mixed) return g.ppt == 1 ? dir_kernel_of<float, 1>(g.neu, g.d2) : dir_kernel_of<float, 2>(g.neu, g.d2);
  return g.ppt == 1 ? dir_kernel_of<double, 1>(g.neu, g.d2) : dir_kernel_of<double, 2>(g.neu, g.d2);
}
size_t stage_smem(bool mixed, const stage_drv::Group& g) {
  return mixed ? wave_dev::stage_bytes<float>(g.ng_max) : wave_dev::stage_bytes<double>(g.ng_max);
}

struct WaveDir {
  const nmpc_wave* h;
  cudaStream_t st;
  cudaError_t operator()(const stage_drv::Ctl& C, const stage_drv::Iter& S) const {
    WArgs A = make_args(h);
    const bool mixed = h->opts.precision == NMPC_MIXED;
    for (int half = 0; half < (A.rb ? 2 : 1); ++half) {
      A.half = half;
      for (const stage_drv::Group& g : h->drv.groups) {
        const cudaError_t e =
            stage_drv::launch_stages(dir_kernel(mixed, g), stage_smem(mixed, g),
                                     stage_drv::range_of(g, A.rb != 0, half), A, C, S, st);
        if (e != cudaSuccess) return e;
      }
    }
    return cudaSuccess;
  }
};

int copy_problem(nmpc_wave* h, const double* x0, const double* w_ref, const double* u_ref,
                 cudaStream_t st) {
  SDRV_CHECK(cudaMemcpyAsync(h->drv.x0, x0, h->drv.n_g * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SDRV_CHECK(cudaMemcpyAsync(h->wref, w_ref, h->n_w * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SDRV_CHECK(cudaMemcpyAsync(h->uref, u_ref, h->n_a * sizeof(double), cudaMemcpyDeviceToDevice, st));
  return NMPC_OK;
}

}  // namespace

extern "C" {

void nmpc_wave_default_opts(nmpc_wave_opts* o) {
  if (!o) return;
  o->tol = 1e-6;
  o->max_iter = 5000;
  o->n_lo = 2;
  o->n_u_it = 2;
  o->variant = NMPC_VARIANT_JACOBI;
  o->check_every = 16;
  o->precision = NMPC_FP64;
}

int nmpc_wave_setup(const nmpc_wave_desc* descs, int n, const nmpc_wave_opts* opts, nmpc_wave** out) {
  if (!descs || n < 1 || !out) return NMPC_ERR_BAD_ARG;
  *out = nullptr;
  nmpc_wave_opts o;
  nmpc_wave_default_opts(&o);
  if (opts) o = *opts;
  if (!(o.tol >= 0) || o.max_iter < 0 || o.n_lo < 1 || o.n_u_it < 0 || o.check_every < 1 ||
      (o.variant != NMPC_VARIANT_JACOBI && o.variant != NMPC_VARIANT_REDBLACK) ||
      (o.precision != NMPC_FP64 && o.precision != NMPC_MIXED))
    return NMPC_ERR_BAD_ARG;
  for (int b = 0; b < n; ++b) {
    const int rc = validate(descs[b]);
    if (rc != NMPC_OK) return rc;
  }
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) return NMPC_ERR_NO_DEVICE;
  nmpc_wave* h = new (std::nothrow) nmpc_wave();
  if (!h) return NMPC_ERR_CUDA;
  h->opts = o;
  std::vector<int> act_of;
  std::vector<stage_drv::GridKind> grid;
  long long n_pts = 0;
  for (int b = 0; b < n; ++b) {
    const nmpc_wave_desc& d = descs[b];
    WInst I{};
    I.dim = d.dim;
    I.m = d.m;
    I.ng = d.dim == 2 ? d.m * d.m : d.m;
    I.nu = d.n_u;
    I.N = d.horizon;
    I.w_off = h->n_w;
    I.a_off = h->n_a;
    I.t_off = n_pts;
    I.h = d.h;
    I.a = d.a;
    I.b = d.b;
    I.c = d.c;
    I.kappa = d.kappa;
    I.gain = d.gain;
    I.q = d.q;
    I.qv = d.qv;
    I.r = d.r;
    I.qf = d.qf;
    I.gamma = d.gamma;
    I.neu = d.bc == 0 ? 1 : 0;
    I.lw = stage_drv::neighbour_weight(d.m, d.bc);
    wave_dev::derive(I);
    const std::vector<int> ao = stage_drv::actuator_map(d.dim, d.m, d.n_u, d.act_cell);
    act_of.insert(act_of.end(), ao.begin(), ao.end());
    grid.push_back(stage_drv::GridKind{d.dim, d.m, I.ng, d.bc == 0});
    stage_drv::Layout L{};
    L.N = I.N;
    L.nx = 2 * I.ng;
    L.nu = I.nu;
    L.u_cold = 0.0;
    h->drv.lay_h.push_back(L);
    h->n_a += I.nu;
    h->n_w += I.ng;
    n_pts += I.ng;
    h->ng_max = std::max(h->ng_max, I.ng);
    h->inst_h.push_back(I);
  }
  cudaError_t e = stage_drv::driver_alloc(h->drv, grid, false);
  auto A = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  A(stage_drv::dalloc(&h->inst_d, n));
  A(stage_drv::dalloc(&h->act_of, act_of.size()));
  A(stage_drv::dalloc(&h->wref, h->n_w));
  A(stage_drv::dalloc(&h->uref, h->n_a));
  A(stage_drv::upload(h->inst_d, h->inst_h));
  A(stage_drv::upload(h->act_of, act_of));
  if (e != cudaSuccess) {
    fprintf(stderr, "nmpc_wave_setup: %s\n", cudaGetErrorString(e));
    free_wave(h);
    delete h;
    return NMPC_ERR_CUDA;
  }
  *out = h;
  return NMPC_OK;
}

int nmpc_wave_sizes(const nmpc_wave* h, int64_t* out) {
  if (!h || !out) return NMPC_ERR_BAD_ARG;
  out[0] = h->drv.n_g;
  out[1] = h->drv.n_x;
  out[2] = h->drv.n_u;
  out[3] = h->n_a;
  out[4] = h->n_w;
  return NMPC_OK;
}

int nmpc_wave_solve(nmpc_wave* h, const double* x0, const double* w_ref, const double* u_ref,
                    int init, double* u_out, nmpc_stats* stats, void* stream) {
  if (!h || !x0 || !w_ref || !u_ref) return NMPC_ERR_BAD_ARG;
  if (init != NMPC_INIT_COLD && init != NMPC_INIT_WARM && init != NMPC_INIT_SHIFT)
    return NMPC_ERR_BAD_ARG;
  if (init != NMPC_INIT_COLD && !h->drv.has_state) return NMPC_ERR_BAD_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int rc = copy_problem(h, x0, w_ref, u_ref, st);
  if (rc != NMPC_OK) return rc;
  WaveDir dir{h, st};
  return stage_drv::solve(h->drv, init, h->opts.max_iter, h->opts.tol, h->opts.check_every, dir,
                          u_out, stats, st);
}

int nmpc_wave_iterate(nmpc_wave* h, const double* x0, const double* w_ref, const double* u_ref,
                      const double* x_in, const double* u_in, const double* lam_in, double* x_out,
                      double* u_out, double* lam_out, int n_iter, double* out, void* stream) {
  if (!h || !x0 || !w_ref || !u_ref || !x_in || !u_in || !lam_in || !x_out || !u_out || !lam_out ||
      n_iter < 1)
    return NMPC_ERR_BAD_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int rc = copy_problem(h, x0, w_ref, u_ref, st);
  if (rc != NMPC_OK) return rc;
  WaveDir dir{h, st};
  return stage_drv::iterate(h->drv, x_in, u_in, lam_in, x_out, u_out, lam_out, n_iter, out, dir, st);
}

int nmpc_wave_get_state(nmpc_wave* h, double* x, double* u, double* lam, void* stream) {
  if (!h) return NMPC_ERR_BAD_ARG;
  return stage_drv::get_state(h->drv, x, u, lam, (cudaStream_t)stream);
}

namespace {
int plant(nmpc_wave* h, double* x, double dt, int n_sub, void* stream) {
  wave_dev::k_wave_plant<<<h->drv.n, wave_dev::THREADS, 3 * h->ng_max * sizeof(double),
                           (cudaStream_t)stream>>>(make_args(h), h->drv.lay, x, h->drv.ub[2], dt,
                                                   n_sub);
  SDRV_CHECK(cudaGetLastError());
  return NMPC_OK;
}
}  // namespace

int nmpc_wave_plant_step(nmpc_wave* h, double* x, double dt, int n_sub, void* stream) {
  if (!h || !x || !(dt >= 0) || n_sub < 1 || !h->drv.has_state) return NMPC_ERR_BAD_ARG;
  return plant(h, x, dt, n_sub, stream);
}

int nmpc_wave_closed_loop(nmpc_wave* h, double* x, const double* w_ref, const double* u_ref,
                          int steps, int n_sub, double* u_hist, int* iters_hist, double* res_hist,
                          void* stream) {
  if (!h || !x || !w_ref || !u_ref || steps < 1 || n_sub < 1) return NMPC_ERR_BAD_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int n = h->drv.n;
  std::vector<nmpc_stats> stats(n);
  int rc_all = NMPC_OK;
  for (int t = 0; t < steps; ++t) {
    const int init = (t == 0 && !h->drv.has_state) ? NMPC_INIT_COLD : NMPC_INIT_SHIFT;
    const int rc = nmpc_wave_solve(h, x, w_ref, u_ref, init, nullptr, stats.data(), stream);
    if (rc == NMPC_ERR_BAD_ARG || rc == NMPC_ERR_CUDA) return rc;
    if (rc != NMPC_OK && rc_all == NMPC_OK) rc_all = rc;
    for (int b = 0; b < n; ++b) {
      if (iters_hist) iters_hist[(size_t)t * n + b] = stats[b].iters;
      if (res_hist) res_hist[(size_t)t * n + b] = stats[b].res_inf;
    }
    if (u_hist) {
      // u_1 of every instance (stage 1 of the packed control trajectory)
      for (int b = 0; b < n; ++b) {
        const WInst& I = h->inst_h[b];
        SDRV_CHECK(cudaMemcpyAsync(u_hist + (size_t)t * h->n_a + I.a_off,
                                   h->drv.ub[2] + h->drv.lay_h[b].u_off, I.nu * sizeof(double),
                                   cudaMemcpyDeviceToDevice, st));
      }
    }
    const int prc = plant(h, x, -1.0, n_sub, stream);  // each instance's own h
    if (prc != NMPC_OK) return prc;
  }
  return rc_all;
}

void nmpc_wave_destroy(nmpc_wave* h) {
  if (!h) return;
  cudaDeviceSynchronize();
  free_wave(h);
  delete h;
}

}  // extern "C"
