// Pinned-actuator solver (include/nmpc_plate.h): the double-layer method on
// the paper's own problem class, the heat plate of Sec. 5.1 whose actuator
// points have their temperatures set directly, with input bounds, the log
// barrier (eq. 8) and the fraction-to-the-boundary step (eq. 11).
//
// One launch of k_plate_dir is one iteration k (two with the red-black upper
// layer: half 0 the even stages; half 1 the odd ones, its right-hand side
// lowered by the even neighbours' directions, M_L Delta x_{i-1} and M_U Delta
// lambda_{i+1}, the form of eq. 18).  A group of threads per (instance,
// stage), one or two grid points a thread (w = x at the state points, u at
// the actuator points; lambda at the state points, zero at the actuators):
// it forms S^k = S^{k-1} - alpha Delta S^{k-1} (the whole instance's step
// alpha_max of eq. 11 is known then) for its own stage, and x_{i-1},
// lambda_{i+1} of the neighbours for itself; evaluates K_i (eq. 9) and its
// norms, the stage's coefficients, and the lower layer (eqs. 21-24 with the
// u-iteration of Sec. 5.2): n_lo pointwise Jacobi sweeps on F_x and F_x^T
// over the state points; stores Delta s_i and the stage's largest admissible
// step (a per-instance atomic minimum).
// The Laplacian of the grid has the mirrored fictitious points of the
// zero-Neumann condition (eqs. 2-3) or the zero Dirichlet ring.
#include <new>

#include "../../include/nmpc_plate.h"
#include "stage_driver.cuh"

namespace plate_dev {

using stage_drv::Ctl;
using stage_drv::Iter;
using stage_drv::Layout;
constexpr int THREADS = 256;
constexpr int MAX_NU = 64;

// Per instance: the grid and the model (packed x, u offsets are the
// driver's Layout; x0 and x_ref share its g_off).
struct PInst {
  int dim, m, ng, ns, nu, N, neu;
  long long a_off;  // u_ref, actuator tables
  long long t_off;  // per-point tables
  double h, k0, k1, beta, ta, gr, q, r, qf, gamma, tau, ulo, uhi;
  double lw;    // the Laplacian's neighbour weight 1 / spacing^2
  double ta4;   // t_amb^4
};

struct PArgs {
  const PInst* inst;
  const int* pt_state;  // [sum ng]: state index, or -1 - a for actuator a
  const int* act_pt;    // [sum nu]: grid point of actuator a
  const double* x0;
  const double* xref;
  const double* uref;
  int n_lo, n_u_it, rb, half;
};

__device__ __forceinline__ double phi(const PInst& I, double w) {
  return I.k0 * (w + 0.5 * I.k1 * w * w);
}
__device__ __forceinline__ double dphi(const PInst& I, double w) {
  return I.k0 * (1.0 + I.k1 * w);
}

// Shared memory of one stage: Phi(w) and the (scaled) lambda in float64, three
// exchange fields of the lower layer's type; each with a zero at index ng.
template <typename T>
__host__ __device__ constexpr size_t stage_bytes(int ng) {
  return (((size_t)(ng + 1) * (2 * sizeof(double) + 3 * sizeof(T))) + 15) & ~size_t(15);
}

// What bounds it: the float64 pipe (2 lanes a clock a SM) on batches, the
// chain of exchanges on one plate.  A thread keeps its points' rows and
// coefficients in registers and exchanges only the field that a stencil reads
// (one barrier each); neighbours are found from the grid (4 additions and one
// multiply-add a stencil, where a table of five weights cost five
// multiply-adds and ten loads); the diagonal's reciprocal is taken once a
// point (a division each sweep before); the actuators' rows, with their
// divisions, sit in the group's first nu threads, so that one or two warps
// execute them and not every warp that owns an actuator point; the maximum
// norm is taken on integers.  1024 plates of 13x13, N = 20, float64: 326 ->
// 144 ms a solve, 140 with the sweeps a constant (float64 pipe 84% busy); one
// plate: 4.8 -> 2.3 ms.  Stages of more than 256 points have two points a thread
// in 64 registers (512 threads, two CTAs a SM) and spill 128 to 276 bytes (412
// with the sweeps read): 64 plates of 24x24, 100 iterations, 46.8 -> 21.2 ms.
// F_x = h (L diag(Phi'(w)) - diag(beta + 4 gr x^3)) - I on the state points;
// v is zero at the actuator points.  The lower layer runs in T (float64, or
// float32 in mixed precision: the residual, the coefficients and the update
// stay float64, so the fixed point is the float64 root).
// NLO: the sweeps per solve as a constant (2, the default), or 0 to read them.
template <typename T, int PPT, bool NEU, bool D2, int NLO>
__global__ void __launch_bounds__(PPT == 1 ? 256 : 512, PPT == 1 ? 3 : 2)
    k_plate_dir(PArgs A, Ctl C, Iter S, stage_drv::Range R) {
  extern __shared__ __align__(16) double smem[];
  __shared__ stage_drv::WarpNorms red[16];
  stage_drv::pdl_trigger();
  const int g = threadIdx.x / R.tps, t = threadIdx.x - g * R.tps;
  const int item = blockIdx.x * R.spc + g;
  stage_drv::pdl_wait();
  if (item >= R.n) return;
  const int2 it = C.work[R.first + item];
  const int b = it.x, s = it.y;
  bool norms_only;
  if (!stage_drv::begin_stage(C, b, s, t, norms_only)) return;
  const PInst& I = A.inst[b];
  const Layout& Ly = C.lay[b];
  const int ng = I.ng, ns = I.ns, nu = I.nu;
  const bool last = (s == I.N - 1);
  double* fA = smem + (size_t)g * (stage_bytes<T>(R.ng_max) / sizeof(double));
  double* fB = fA + (ng + 1);
  T* fC = reinterpret_cast<T*>(fB + (ng + 1));
  T* fD = fC + (ng + 1);
  T* fZ = fD + (ng + 1);  // Phi'(u) v3 at the actuator points, zero elsewhere
  const int* pts = A.pt_state + I.t_off;
  const long long so = Ly.s_off + (long long)s * ns;
  const long long uo = Ly.u_off + (long long)s * nu;
  const double h = I.h, lw = I.lw;
  constexpr double d2 = D2 ? 4.0 : 2.0;  // the Laplacian's centre: -2 dim lw
  const bool first = C.k == 0;           // S^0 is there already
  const double alpha =
      first ? 0.0
            : fmin(1.0, __longlong_as_double(
                            (long long)__ldcg(C.acand + ((C.k - 1) % stage_drv::SLOTS) * C.n_inst + b)));
  // S^k at packed index e of a state array
  auto xk = [&](const double* x, const double* dx, long long e) {
    const double v = __ldcg(x + e);
    return first ? v : v - alpha * __ldcg(dx + e);
  };

  stage_drv::Nbr<NEU, D2> nb[PPT];
  int ts[PPT];  // state index, or negative: an actuator point or none
  if (t == 0) {
    fA[ng] = fB[ng] = 0.0;
    fC[ng] = fD[ng] = fZ[ng] = T(0);
  }
  double w[PPT], lam[PPT];
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    const int p = t + j * R.tps;
    nb[j].set(p, I.m, ng);
    ts[j] = p < ng ? pts[p] : -0x7fffffff;
    w[j] = lam[j] = 0.0;
    if (p < ng) {
      if (ts[j] >= 0) {
        w[j] = xk(S.xin, S.px, so + ts[j]);
        lam[j] = xk(S.lin, S.pl, so + ts[j]);
        if (!first) {
          S.xout[so + ts[j]] = w[j];
          S.lout[so + ts[j]] = lam[j];
        }
      } else {
        w[j] = xk(S.uin, S.pu, uo + (-1 - ts[j]));
        if (!first) S.uout[uo + (-1 - ts[j])] = w[j];
      }
      fA[p] = phi(I, w[j]);
      fB[p] = nb[j].scale(lam[j]);
      fC[p] = fD[p] = fZ[p] = T(0);
    }
  }
  // the first nu threads: an actuator's row each
  const bool act = t < nu;
  stage_drv::Nbr<NEU, D2> na;
  int pa = ng;
  double ua = 0.0;
  if (act) {
    pa = A.act_pt[I.a_off + t];
    ua = xk(S.uin, S.pu, uo + t);
  }
  na.set(pa, I.m, ng);
  stage_drv::group_sync(g, R.tps);

  // K_i (eq. 9), coefficients, norms
  unsigned long long mx = 0ull;
  double sq = 0.0;
  const double d2p = I.k0 * I.k1, hqf = last ? h * I.qf : 0.0;
  T k1[PPT], k3[PPT], rdg[PPT], ax[PPT], dp[PPT];
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    k1[j] = k3[j] = rdg[j] = ax[j] = dp[j] = T(0);
    if (ts[j] < 0) continue;
    const int p = t + j * R.tps, e = ts[j];
    const double x = w[j], lm = lam[j];
    const double xprev = (s == 0) ? A.x0[Ly.g_off + e] : xk(S.xin, S.px, so - ns + e);
    const double dx = x - A.xref[Ly.g_off + e];
    const double lnext = last ? hqf * dx : xk(S.lin, S.pl, so + ns + e);
    const double lph = lw * (nb[j].sum(fA) - d2 * fA[p]);                     // (L Phi)(p)
    const double ltl = lw * (nb[j].unscale(nb[j].sum(fB)) - d2 * lm);         // (L^T lambda)(p)
    const double x2 = x * x, gx3 = 4.0 * I.gr * (x2 * x) + I.beta;
    const double fp = lph - I.beta * (x - I.ta) - I.gr * (x2 * x2 - I.ta4);
    const double K1 = xprev - x + h * fp;
    const double dpx = dphi(I, x);
    const double K3 = lnext - lm + h * (I.q * dx + (dpx * ltl - gx3 * lm));
    mx = max(mx, max(stage_drv::abs_bits(K1), stage_drv::abs_bits(K3)));
    sq += K1 * K1 + K3 * K3;
    // red-black half 1: the right-hand side takes the even neighbours'
    // directions; the norms above stay those of K(S^k)
    double K1r = K1, K3r = K3;
    if (A.rb && A.half == 1) {
      if (s > 0) K1r -= __ldcg(S.dx + so - ns + e);
      if (!last) K3r -= __ldcg(S.dl + so + ns + e);
    }
    k1[j] = (T)K1r;
    k3[j] = (T)K3r;
    dp[j] = (T)dpx;
    rdg[j] = stage_drv::rcp((T)(h * (-d2 * lw * dpx - gx3) - 1.0));
    ax[j] = (T)(h * (I.q + d2p * ltl - 12.0 * I.gr * x2 * lm) + hqf);
  }
  T k2 = T(0), rauu = T(0), dpu = T(0), v3 = T(0);
  double il = 0.0, ih = 0.0;  // 1 / slack to the lower, the upper bound
  if (act) {
    const double ltl = lw * na.unscale(na.sum(fB));  // lambda is zero at the point itself
    double db = 0.0, d2b = 0.0;
    if (I.tau > 0.0) {
      il = 1.0 / (ua - I.ulo);
      ih = 1.0 / (I.uhi - ua);
      db = I.tau * (ih - il);
      d2b = I.tau * (il * il + ih * ih);
    }
    const double dpx = dphi(I, ua);
    const double K2 = h * (I.r * (ua - A.uref[I.a_off + t]) + db + dpx * ltl);
    mx = max(mx, stage_drv::abs_bits(K2));
    sq += K2 * K2;
    k2 = (T)K2;
    rauu = stage_drv::rcp((T)(h * (I.r + d2b + d2p * ltl) + I.gamma));
    dpu = (T)dpx;
  }
  stage_drv::warp_norms(mx, sq, red);

  // u fixed-point iteration (Sec. 5.2) on the direction y = P^{-1}(K_1 - F_u
  // v3, K_3): v3 = (K_2 - F_u^T y_lambda) / A_uu from v3 = 0, then the last y.
  // F_u v3 = h L Z, Z = Phi'(u) v3 at the actuator points.
  const T hw = (T)(h * lw);
  T v5[PPT], v4[PPT];
#pragma unroll
  for (int j = 0; j < PPT; ++j) v5[j] = v4[j] = T(0);
  const int n_lo = NLO > 0 ? NLO : A.n_lo;
  T *ex = fC, *ex2 = fD;  // the next exchange's field, the other one
  for (int itu = 0; itu <= A.n_u_it; ++itu) {
    if (itu > 0) {
      if (act) fZ[pa] = dpu * v3;
      stage_drv::group_sync(g, R.tps);
    }
    T b4[PPT], b5[PPT];
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      b4[j] = itu > 0 ? k1[j] - hw * nb[j].sum(fZ) : k1[j];
      v5[j] = b4[j] * rdg[j];
    }
    for (int sw = 1; sw < n_lo; ++sw) {  // F_x v5 = b4 (rdg is zero off the state points)
#pragma unroll
      for (int j = 0; j < PPT; ++j)
        if (ts[j] >= 0) ex[t + j * R.tps] = dp[j] * v5[j];
      stage_drv::group_sync(g, R.tps);
      if (itu == 0 && sw == 1) {
        if (t == 0) stage_drv::publish_norms(C, b, red, R.tps);
        if (norms_only) return;
      }
#pragma unroll
      for (int j = 0; j < PPT; ++j) v5[j] = (b4[j] - hw * nb[j].sum(ex)) * rdg[j];
      T* x = ex;
      ex = ex2;
      ex2 = x;
    }
    if (itu == 0 && n_lo == 1) {
      stage_drv::group_sync(g, R.tps);
      if (t == 0) stage_drv::publish_norms(C, b, red, R.tps);
      if (norms_only) return;
    }
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      b5[j] = k3[j] - ax[j] * v5[j];
      v4[j] = b5[j] * rdg[j];
    }
    for (int sw = 1; sw < n_lo; ++sw) {  // F_x^T v4 = b5
#pragma unroll
      for (int j = 0; j < PPT; ++j)
        if (ts[j] >= 0) ex[t + j * R.tps] = nb[j].scale(v4[j]);
      stage_drv::group_sync(g, R.tps);
#pragma unroll
      for (int j = 0; j < PPT; ++j)
        v4[j] = (b5[j] - hw * dp[j] * nb[j].unscale(nb[j].sum(ex))) * rdg[j];
      T* x = ex;
      ex = ex2;
      ex2 = x;
    }
    if (itu == A.n_u_it) break;
#pragma unroll
    for (int j = 0; j < PPT; ++j)
      if (ts[j] >= 0) ex[t + j * R.tps] = nb[j].scale(v4[j]);
    stage_drv::group_sync(g, R.tps);
    if (act) v3 = (k2 - hw * dpu * na.unscale(na.sum(ex))) * rauu;
    T* x = ex;
    ex = ex2;
    ex2 = x;
  }
  // direction (Delta x, Delta u, Delta lambda) = (v5, v3, v4); admissible step
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    if (ts[j] >= 0) {
      S.dx[so + ts[j]] = (double)v5[j];
      S.dl[so + ts[j]] = (double)v4[j];
    }
  }
  if ((t & ~31) < nu) {  // the actuators' warps
    double amin = 1.0;
    if (act) {
      const double d = (double)v3;
      S.du[uo + t] = d;
      if (I.tau > 0.0) {
        if (d > 0.0) amin = fmin(amin, 0.995 * (ua - I.ulo) / d);
        if (d < 0.0) amin = fmin(amin, 0.995 * (I.uhi - ua) / (-d));
      }
    }
    stage_drv::publish_step(C, b, amin);
  }
}

// (L v)(p) over a stage's grid, one axis after the other.
__device__ __forceinline__ double lap_at(const PInst& I, const double* v, int p) {
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

// The plant: w (state points) += (dt / n_sub) f(w, u1), n_sub times, with the
// actuator points at the first-stage inputs u1 of the current state; dt < 0
// takes each instance's own stage length h.
__global__ void __launch_bounds__(THREADS) k_plate_plant(PArgs A, const Layout* lay, double* w,
                                                         const double* uc, double dt, int n_sub) {
  const int b = blockIdx.x;
  const PInst I = A.inst[b];
  const Layout Ly = lay[b];
  extern __shared__ double smem[];
  double* W = smem;
  double* PH = W + I.ng;
  const int* pts = A.pt_state + I.t_off;
  for (int p = threadIdx.x; p < I.ng; p += THREADS) {
    const int t = pts[p];
    W[p] = (t >= 0) ? w[Ly.g_off + t] : uc[Ly.u_off + (-1 - t)];
  }
  __syncthreads();
  const double tau = (dt < 0.0 ? I.h : dt) / n_sub;
  for (int k = 0; k < n_sub; ++k) {
    for (int p = threadIdx.x; p < I.ng; p += THREADS) PH[p] = phi(I, W[p]);
    __syncthreads();
    double nw[4];
    int cnt = 0;
    for (int p = threadIdx.x; p < I.ng; p += THREADS, ++cnt) {
      double v = W[p];
      if (pts[p] >= 0) {
        const double lph = lap_at(I, PH, p);
        const double x = v, x4 = x * x * x * x;
        v = x + tau * (lph - I.beta * (x - I.ta) - I.gr * (x4 - I.ta * I.ta * I.ta * I.ta));
      }
      nw[cnt] = v;
    }
    __syncthreads();
    cnt = 0;
    for (int p = threadIdx.x; p < I.ng; p += THREADS, ++cnt) W[p] = nw[cnt];
    __syncthreads();
  }
  for (int p = threadIdx.x; p < I.ng; p += THREADS) {
    const int t = pts[p];
    if (t >= 0) w[Ly.g_off + t] = W[p];
  }
}

}  // namespace plate_dev

using plate_dev::PInst;
using plate_dev::PArgs;

struct nmpc_plate {
  nmpc_plate_opts opts{};
  std::vector<PInst> inst_h;
  stage_drv::Driver drv;     // iterates, direction, control words, layout
  long long n_a = 0;         // sum n_u
  int ng_max = 0;
  PInst* inst_d = nullptr;
  int *pt_state = nullptr, *act_pt = nullptr;
  double *xref = nullptr, *uref = nullptr;
};

namespace {

void free_plate(nmpc_plate* h) {
  stage_drv::driver_free(h->drv);
  void* ptrs[] = {h->inst_d, h->pt_state, h->act_pt, h->xref, h->uref};
  for (void* p : ptrs)
    if (p) cudaFree(p);
}

int validate(const nmpc_plate_desc& d) {
  if ((d.dim != 1 && d.dim != 2) || d.horizon < 1 || d.n_u < 1 || !d.act_cell) return NMPC_ERR_BAD_ARG;
  if (d.bc != 0 && d.bc != 1) return NMPC_ERR_BAD_ARG;
  if (d.m < (d.bc == 0 ? 3 : 1)) return NMPC_ERR_BAD_ARG;
  const long long ng = d.dim == 2 ? (long long)d.m * d.m : d.m;
  if (ng > NMPC_PLATE_MAX_POINTS || d.n_u > plate_dev::MAX_NU) return NMPC_ERR_UNSUPPORTED;
  if (d.n_u >= ng) return NMPC_ERR_BAD_ARG;
  std::vector<char> seen(ng, 0);
  for (int a = 0; a < d.n_u; ++a) {
    if (d.act_cell[a] < 0 || d.act_cell[a] >= ng || seen[d.act_cell[a]]) return NMPC_ERR_BAD_ARG;
    seen[d.act_cell[a]] = 1;
  }
  if (!(d.h > 0) || !(d.k0 > 0) || !std::isfinite(d.k1) || !(d.beta >= 0) || !(d.gamma_r >= 0) ||
      !std::isfinite(d.t_amb) || !(d.q >= 0) || !(d.r > 0) || !(d.qf >= 0) || !(d.gamma >= 0) ||
      !(d.tau >= 0))
    return NMPC_ERR_BAD_ARG;
  if (d.tau > 0 && !(d.u_lo < d.u_hi)) return NMPC_ERR_BAD_ARG;
  return NMPC_OK;
}

PArgs make_args(const nmpc_plate* h) {
  PArgs A{};
  A.inst = h->inst_d;
  A.pt_state = h->pt_state;
  A.act_pt = h->act_pt;
  A.x0 = h->drv.x0;
  A.xref = h->xref;
  A.uref = h->uref;
  A.n_lo = h->opts.n_lo;
  A.n_u_it = h->opts.n_u_it;
  A.rb = (h->opts.variant == NMPC_VARIANT_REDBLACK) ? 1 : 0;
  return A;
}

// k_plate_dir for a group of stages.
using DirKernel = void (*)(PArgs, stage_drv::Ctl, stage_drv::Iter, stage_drv::Range);
template <typename T, int PPT, int NLO>
DirKernel dir_kernel_of(bool neu, bool d2) {
  using namespace plate_dev;
  if (neu) return d2 ? k_plate_dir<T, PPT, true, true, NLO> : k_plate_dir<T, PPT, true, false, NLO>;
  return d2 ? k_plate_dir<T, PPT, false, true, NLO> : k_plate_dir<T, PPT, false, false, NLO>;
}
template <int NLO>
DirKernel dir_kernel_with(bool mixed, const stage_drv::Group& g) {
  if (mixed)
    return g.ppt == 1 ? dir_kernel_of<float, 1, NLO>(g.neu, g.d2) : dir_kernel_of<float, 2, NLO>(g.neu, g.d2);
  return g.ppt == 1 ? dir_kernel_of<double, 1, NLO>(g.neu, g.d2) : dir_kernel_of<double, 2, NLO>(g.neu, g.d2);
}
DirKernel dir_kernel(bool mixed, int n_lo, const stage_drv::Group& g) {
  return n_lo == 2 ? dir_kernel_with<2>(mixed, g) : dir_kernel_with<0>(mixed, g);
}
size_t stage_smem(bool mixed, const stage_drv::Group& g) {
  return mixed ? plate_dev::stage_bytes<float>(g.ng_max) : plate_dev::stage_bytes<double>(g.ng_max);
}

// The direction kernels of one iteration: one launch per group of stages, or
// the two red-black halves.
struct PlateDir {
  const nmpc_plate* h;
  cudaStream_t st;
  cudaError_t operator()(const stage_drv::Ctl& C, const stage_drv::Iter& S) const {
    PArgs A = make_args(h);
    const bool mixed = h->opts.precision == NMPC_MIXED;
    for (int half = 0; half < (A.rb ? 2 : 1); ++half) {
      A.half = half;
      for (const stage_drv::Group& g : h->drv.groups) {
        const cudaError_t e =
            stage_drv::launch_stages(dir_kernel(mixed, A.n_lo, g), stage_smem(mixed, g),
                                     stage_drv::range_of(g, A.rb != 0, half), A, C, S, st);
        if (e != cudaSuccess) return e;
      }
    }
    return cudaSuccess;
  }
};

int copy_problem(nmpc_plate* h, const double* x0, const double* x_ref, const double* u_ref,
                 cudaStream_t st) {
  SDRV_CHECK(cudaMemcpyAsync(h->drv.x0, x0, h->drv.n_g * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SDRV_CHECK(cudaMemcpyAsync(h->xref, x_ref, h->drv.n_g * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SDRV_CHECK(cudaMemcpyAsync(h->uref, u_ref, h->n_a * sizeof(double), cudaMemcpyDeviceToDevice, st));
  return NMPC_OK;
}

int plant(nmpc_plate* h, double* w, double dt, int n_sub, void* stream) {
  plate_dev::k_plate_plant<<<h->drv.n, plate_dev::THREADS, 2 * h->ng_max * sizeof(double),
                             (cudaStream_t)stream>>>(make_args(h), h->drv.lay, w, h->drv.ub[2], dt,
                                                     n_sub);
  SDRV_CHECK(cudaGetLastError());
  return NMPC_OK;
}

}  // namespace

extern "C" {

void nmpc_plate_default_opts(nmpc_plate_opts* o) {
  if (!o) return;
  o->tol = 1e-6;
  o->max_iter = 5000;
  o->n_lo = 2;
  o->n_u_it = 2;
  o->variant = NMPC_VARIANT_JACOBI;
  o->check_every = 16;
  o->precision = NMPC_FP64;
}

int nmpc_plate_setup(const nmpc_plate_desc* descs, int n, const nmpc_plate_opts* opts,
                     nmpc_plate** out) {
  if (!descs || n < 1 || !out) return NMPC_ERR_BAD_ARG;
  *out = nullptr;
  nmpc_plate_opts o;
  nmpc_plate_default_opts(&o);
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
  nmpc_plate* h = new (std::nothrow) nmpc_plate();
  if (!h) return NMPC_ERR_CUDA;
  h->opts = o;
  std::vector<int> pt_state, act_pt;
  std::vector<stage_drv::GridKind> grid;
  long long n_pts = 0;
  for (int b = 0; b < n; ++b) {
    const nmpc_plate_desc& d = descs[b];
    PInst I{};
    I.dim = d.dim;
    I.m = d.m;
    I.ng = d.dim == 2 ? d.m * d.m : d.m;
    I.nu = d.n_u;
    I.ns = I.ng - I.nu;
    I.N = d.horizon;
    I.a_off = h->n_a;
    I.t_off = n_pts;
    I.h = d.h;
    I.k0 = d.k0;
    I.k1 = d.k1;
    I.beta = d.beta;
    I.ta = d.t_amb;
    I.gr = d.gamma_r;
    I.q = d.q;
    I.r = d.r;
    I.qf = d.qf;
    I.gamma = d.gamma;
    I.tau = d.tau;
    I.ulo = d.u_lo;
    I.uhi = d.u_hi;
    I.neu = d.bc == 0 ? 1 : 0;
    I.lw = stage_drv::neighbour_weight(d.m, d.bc);
    I.ta4 = d.t_amb * d.t_amb * d.t_amb * d.t_amb;
    // point -> state index (grid order of the non-actuator points) or -1 - a
    std::vector<int> state_of(I.ng, 0);
    std::vector<char> is_act(I.ng, 0);
    for (int a = 0; a < d.n_u; ++a) {
      state_of[d.act_cell[a]] = -1 - a;
      is_act[d.act_cell[a]] = 1;
    }
    int t = 0;
    for (int p = 0; p < I.ng; ++p)
      if (!is_act[p]) state_of[p] = t++;
    for (int p = 0; p < I.ng; ++p) pt_state.push_back(state_of[p]);
    for (int a = 0; a < d.n_u; ++a) act_pt.push_back(d.act_cell[a]);
    grid.push_back(stage_drv::GridKind{d.dim, d.m, I.ng, d.bc == 0});
    stage_drv::Layout L{};
    L.N = I.N;
    L.nx = I.ns;
    L.nu = I.nu;
    L.u_cold = d.tau > 0.0 ? 0.5 * (d.u_lo + d.u_hi) : 0.0;
    h->drv.lay_h.push_back(L);
    h->n_a += I.nu;
    n_pts += I.ng;
    h->ng_max = std::max(h->ng_max, I.ng);
    h->inst_h.push_back(I);
  }
  cudaError_t e = stage_drv::driver_alloc(h->drv, grid, true);
  auto A = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  A(stage_drv::dalloc(&h->inst_d, n));
  A(stage_drv::dalloc(&h->pt_state, pt_state.size()));
  A(stage_drv::dalloc(&h->act_pt, act_pt.size()));
  A(stage_drv::dalloc(&h->xref, h->drv.n_g));
  A(stage_drv::dalloc(&h->uref, h->n_a));
  A(stage_drv::upload(h->inst_d, h->inst_h));
  A(stage_drv::upload(h->pt_state, pt_state));
  A(stage_drv::upload(h->act_pt, act_pt));
  if (e != cudaSuccess) {
    fprintf(stderr, "nmpc_plate_setup: %s\n", cudaGetErrorString(e));
    free_plate(h);
    delete h;
    return NMPC_ERR_CUDA;
  }
  *out = h;
  return NMPC_OK;
}

int nmpc_plate_sizes(const nmpc_plate* h, int64_t* out) {
  if (!h || !out) return NMPC_ERR_BAD_ARG;
  out[0] = h->drv.n_g;
  out[1] = h->drv.n_x;
  out[2] = h->drv.n_u;
  out[3] = h->n_a;
  return NMPC_OK;
}

int nmpc_plate_solve(nmpc_plate* h, const double* x0, const double* x_ref, const double* u_ref,
                     int init, double* u_out, nmpc_stats* stats, void* stream) {
  if (!h || !x0 || !x_ref || !u_ref) return NMPC_ERR_BAD_ARG;
  if (init != NMPC_INIT_COLD && init != NMPC_INIT_WARM && init != NMPC_INIT_SHIFT)
    return NMPC_ERR_BAD_ARG;
  if (init != NMPC_INIT_COLD && !h->drv.has_state) return NMPC_ERR_BAD_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int rc = copy_problem(h, x0, x_ref, u_ref, st);
  if (rc != NMPC_OK) return rc;
  PlateDir dir{h, st};
  return stage_drv::solve(h->drv, init, h->opts.max_iter, h->opts.tol, h->opts.check_every, dir,
                          u_out, stats, st);
}

int nmpc_plate_iterate(nmpc_plate* h, const double* x0, const double* x_ref, const double* u_ref,
                       const double* x_in, const double* u_in, const double* lam_in,
                       double* x_out, double* u_out, double* lam_out, int n_iter, double* out,
                       void* stream) {
  if (!h || !x0 || !x_ref || !u_ref || !x_in || !u_in || !lam_in || !x_out || !u_out || !lam_out ||
      n_iter < 1)
    return NMPC_ERR_BAD_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int rc = copy_problem(h, x0, x_ref, u_ref, st);
  if (rc != NMPC_OK) return rc;
  PlateDir dir{h, st};
  return stage_drv::iterate(h->drv, x_in, u_in, lam_in, x_out, u_out, lam_out, n_iter, out, dir, st);
}

int nmpc_plate_get_state(nmpc_plate* h, double* x, double* u, double* lam, void* stream) {
  if (!h) return NMPC_ERR_BAD_ARG;
  return stage_drv::get_state(h->drv, x, u, lam, (cudaStream_t)stream);
}

int nmpc_plate_plant_step(nmpc_plate* h, double* w, double dt, int n_sub, void* stream) {
  if (!h || !w || !(dt >= 0) || n_sub < 1 || !h->drv.has_state) return NMPC_ERR_BAD_ARG;
  return plant(h, w, dt, n_sub, stream);
}

int nmpc_plate_closed_loop(nmpc_plate* h, double* w, const double* x_ref, const double* u_ref,
                           int steps, int n_sub, double* u_hist, int* iters_hist,
                           double* res_hist, void* stream) {
  if (!h || !w || !x_ref || !u_ref || steps < 1 || n_sub < 1) return NMPC_ERR_BAD_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int n = h->drv.n;
  std::vector<nmpc_stats> stats(n);
  int rc_all = NMPC_OK;
  for (int t = 0; t < steps; ++t) {
    const int init = (t == 0 && !h->drv.has_state) ? NMPC_INIT_COLD : NMPC_INIT_SHIFT;
    const int rc = nmpc_plate_solve(h, w, x_ref, u_ref, init, nullptr, stats.data(), stream);
    if (rc == NMPC_ERR_BAD_ARG || rc == NMPC_ERR_CUDA) return rc;
    if (rc != NMPC_OK && rc_all == NMPC_OK) rc_all = rc;
    for (int b = 0; b < n; ++b) {
      if (iters_hist) iters_hist[(size_t)t * n + b] = stats[b].iters;
      if (res_hist) res_hist[(size_t)t * n + b] = stats[b].res_inf;
    }
    if (u_hist) {
      // u_1 of every instance (stage 1 of the packed control trajectory)
      for (int b = 0; b < n; ++b) {
        const PInst& I = h->inst_h[b];
        SDRV_CHECK(cudaMemcpyAsync(u_hist + (size_t)t * h->n_a + I.a_off,
                                   h->drv.ub[2] + h->drv.lay_h[b].u_off, I.nu * sizeof(double),
                                   cudaMemcpyDeviceToDevice, st));
      }
    }
    const int prc = plant(h, w, -1.0, n_sub, stream);  // each instance's own h
    if (prc != NMPC_OK) return prc;
  }
  return rc_all;
}

void nmpc_plate_destroy(nmpc_plate* h) {
  if (!h) return;
  cudaDeviceSynchronize();
  free_plate(h);
  delete h;
}

}  // extern "C"
