// The upper-layer driver shared by the stage-parallel solvers (the pinned-
// actuator plate and the second-order wave).  One launch of a problem's
// direction kernel is one iteration k (two, one per stage parity, with the
// red-black order): it decides from iteration k - 1's norms whether the
// instance has finished (Table 2's rule ||K||_inf <= tol), publishes
// ||K(S^k)||_inf, ||K(S^k)||_2^2 and the largest admissible step (eq. 11)
// per instance, and forms S^{k+1} itself (wave: the full step) or leaves
// Delta S^k for the next launch to apply (plate: the step length is known
// once every stage of the instance has published its own).  So an iteration
// costs one launch and no separate pass over the state.  Start iterates
// (cold, warm, shifted by one stage), the returned iterate and the host loops
// of a solve and of a fixed number of iterations live here too.
//
// Arrays are packed per instance: x, lambda [sum N nx] stage-major, u
// [sum N nu] stage-major, x0 [sum nx].  The control words of iteration k are
// in slot k % SLOTS: k - 1's is read while k's accumulates and k + 1's is
// cleared, and launches may overlap their start with the previous launch's
// end (programmatic dependent launch).
#pragma once

#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../include/nmpc.h"

namespace stage_drv {

enum { ST_RUNNING = 0, ST_CONVERGED = 1, ST_DIVERGED = 2, ST_MAX_ITER = 3 };
enum { MODE_SOLVE = 0, MODE_ONESHOT = 1 };
constexpr int SLOTS = 4;  // iterations k - 1, k, k + 1 in use at once

struct Layout {
  int N, nx, nu;     // stages, state entries per stage, inputs per stage
  long long s_off;   // packed x, lambda: stage 1 of this instance
  long long u_off;   // packed u
  long long g_off;   // packed x0
  double u_cold;     // the cold start's input
};

struct Ctl {
  const Layout* lay;
  const int2* work;            // (instance, stage), one thread group each
  unsigned long long* rmax;    // [SLOTS][n] bits of ||K||_inf (non-negative doubles order as integers)
  double* rsq;                 // [SLOTS][n] ||K||_2^2
  unsigned long long* acand;   // [SLOTS][n] bits of the admissible step
  int* status;
  int* iters;
  int* final_buf;
  double* fin;                 // [2][n] final (||K||_inf, ||K||_2)
  int* n_active;
  int n_inst, k, mode, max_iter;
  double tol;
};

// The state arrays of one launch: xin, uin, lin hold the iterate that the
// launch reads, xout, uout, lout the one it writes; the plate's launch k also
// reads Delta S^{k-1} (px, pu, pl) and writes Delta S^k (dx, du, dl).
struct Iter {
  const double* xin;
  const double* uin;
  const double* lin;
  double* xout;
  double* uout;
  double* lout;
  const double* px;
  const double* pu;
  const double* pl;
  double* dx;
  double* du;
  double* dl;
};

// The work items that one launch shape covers: the stages of the instances of
// one grid kind (dimension, boundary condition; see driver_alloc), even stages
// first.  A stage
// is a group of tps threads (a multiple of 32) with ppt points each, spc
// groups to a CTA: a 64-point string on a 256-thread CTA of its own left six
// of eight warps idle, four of them share one now.  More than 256 points take
// two a thread (at most 512 threads).  Few stages stay one to a CTA so that a
// single instance still spreads over the SMs.
struct Group {
  int first, n, n_even;
  int tps, spc, ppt;
  bool neu, d2;
  int ng_max;
};
struct Range {  // the items of one launch
  int first, n, tps, spc, ng_max;
};

// A group's items in one launch: all of them, or one parity's (red-black).
inline Range range_of(const Group& g, bool rb, int half) {
  Range r{g.first, g.n, g.tps, g.spc, g.ng_max};
  if (rb) {
    r.first += half ? g.n_even : 0;
    r.n = half ? g.n - g.n_even : g.n_even;
  }
  return r;
}

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Barrier of thread group g of a CTA (tps threads, a multiple of 32).
__device__ __forceinline__ void group_sync(int g, int tps) {
  if (tps == 32)
    __syncwarp();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(tps) : "memory");
}

// The grid neighbours of point p among m (or m x m) points, as indices into a
// field of ng values with a zero at index ng: outside a Dirichlet grid the
// zero, outside a Neumann grid the mirrored point (eq. 3).
template <bool NEU, bool D2>
struct Nbr {
  unsigned lr, ud;  // left | right << 16, above | below << 16 (fields hold at most 1025 values)
  float di;         // NEU: 2 per axis on whose boundary p lies, else 1 (L^T below)
  __device__ __forceinline__ void set(int p, int m, int ng) {
    if (p >= ng) {  // no point: reads the zero
      lr = ud = (unsigned)ng | ((unsigned)ng << 16);
      di = 1.0f;
      return;
    }
    const int iy = D2 ? p / m : 0, ix = p - iy * m;
    const int l = ix > 0 ? p - 1 : (NEU ? p + 1 : ng);
    const int r = ix < m - 1 ? p + 1 : (NEU ? p - 1 : ng);
    lr = (unsigned)l | ((unsigned)r << 16);
    ud = 0u;
    if constexpr (D2) {
      const int u = iy > 0 ? p - m : (NEU ? p + m : ng);
      const int d = iy < m - 1 ? p + m : (NEU ? p - m : ng);
      ud = (unsigned)u | ((unsigned)d << 16);
    }
    di = 1.0f;
    if constexpr (NEU) {
      if (ix == 0 || ix == m - 1) di *= 2.0f;
      if (D2 && (iy == 0 || iy == m - 1)) di *= 2.0f;
    }
  }
  // sum over the neighbours of v: (L v)(p) = lw (sum - 2 dim v(p))
  template <typename V>
  __device__ __forceinline__ V sum(const V* v) const {
    V s = v[lr & 0xffffu] + v[lr >> 16];
    if constexpr (D2) s += v[ud & 0xffffu] + v[ud >> 16];
    return s;
  }
  // The mirrored Laplacian is D^{-1} S with S symmetric and D = diag(1 / di),
  // so (L^T v)(p) = (L (di v))(p) / di: a field read through the transpose is
  // stored as scale(v), its neighbour sum taken through unscale().  Both are
  // exact (powers of two); on a Dirichlet grid L is symmetric.
  template <typename V>
  __device__ __forceinline__ V scale(V v) const {
    return NEU ? v * (V)di : v;
  }
  template <typename V>
  __device__ __forceinline__ V unscale(V v) const {
    return NEU ? v * (V)(di == 1.0f ? 1.0f : (di == 2.0f ? 0.5f : 0.25f)) : v;
  }
};

// 1 / v rounded to nearest
__device__ __forceinline__ float rcp(float v) { return __frcp_rn(v); }
__device__ __forceinline__ double rcp(double v) { return __drcp_rn(v); }

// b / d from r = 1 / d rounded: the product and its correction, one rounding as
// in a division.
template <typename T>
__device__ __forceinline__ T quot(T b, T d, T r) {
  const T q = b * r;
  return fma(fma(-q, d, b), r, q);
}

// Bits of |v|: non-negative doubles order as integers, NaN above infinity, so
// that a maximum costs the integer pipe and not the two-lane float64 one and
// keeps a NaN.
__device__ __forceinline__ unsigned long long abs_bits(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// The warp's norms (max bits, sum of squares) into red[warp] (lane 0).
struct WarpNorms {
  unsigned long long mx;
  double sq;
};
__device__ __forceinline__ void warp_norms(unsigned long long mx, double sq, WarpNorms* red) {
  for (int o = 16; o > 0; o >>= 1) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    sq += __shfl_xor_sync(0xffffffffu, sq, o);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = WarpNorms{mx, sq};
}

// After a group barrier, by the group's thread 0: its warps' norms into the
// instance's slot of iteration k.
__device__ __forceinline__ void publish_norms(const Ctl& C, int b, const WarpNorms* red, int tps) {
  const int w0 = threadIdx.x >> 5;
  unsigned long long mx = red[w0].mx;
  double sq = red[w0].sq;
  for (int w = 1; w < tps / 32; ++w) {
    mx = max(mx, red[w0 + w].mx);
    sq += red[w0 + w].sq;
  }
  const int slot = (C.k % SLOTS) * C.n_inst + b;
  atomicMax(&C.rmax[slot], mx);
  atomicAdd(&C.rsq[slot], sq);
}

// A warp's smallest admissible step (amin in (0, 1]) into the instance's slot.
__device__ __forceinline__ void publish_step(const Ctl& C, int b, double amin) {
  for (int o = 16; o > 0; o >>= 1) amin = fmin(amin, __shfl_xor_sync(0xffffffffu, amin, o));
  if ((threadIdx.x & 31) == 0 && amin < 1.0)
    atomicMin(&C.acand[(C.k % SLOTS) * C.n_inst + b],
              (unsigned long long)__double_as_longlong(amin));
}

// Records that instance b stopped with iterate kf.
__device__ __forceinline__ void record_stop(const Ctl& C, int b, int kf, int status, double r) {
  C.status[b] = status;
  C.iters[b] = kf;
  C.final_buf[b] = kf & 1;
  C.fin[b] = r;
  C.fin[C.n_inst + b] = sqrt(__ldcg(C.rsq + (kf % SLOTS) * C.n_inst + b));
  atomicSub(C.n_active, 1);
}

// What iteration k does for a stage's group: nothing (returns false: the
// instance has stopped, now or before), the norms only (the last iteration a
// solve allows) or all of it.  Every thread of every group of the instance
// reads the same norms and so decides alike (a status written meanwhile by
// the book-keeper, stage 0's thread 0, says the same).
__device__ __forceinline__ bool begin_stage(const Ctl& C, int b, int s, int t, bool& norms_only) {
  norms_only = false;
  const bool books = s == 0 && t == 0;
  if (C.mode == MODE_SOLVE) {
    const int status = __ldcg(C.status + b);
    const double r =
        C.k > 0 ? __longlong_as_double((long long)__ldcg(C.rmax + ((C.k - 1) % SLOTS) * C.n_inst + b))
                : CUDART_INF;
    if (status != ST_RUNNING) return false;
    if (C.k > 0 && (!(r <= 1.79e308) || r <= C.tol)) {
      if (books) record_stop(C, b, C.k - 1, !(r <= 1.79e308) ? ST_DIVERGED : ST_CONVERGED, r);
      return false;
    }
    norms_only = C.k >= C.max_iter;
  }
  if (books) {
    const int nslot = ((C.k + 1) % SLOTS) * C.n_inst + b;
    C.rmax[nslot] = 0ull;
    C.rsq[nslot] = 0.0;
    C.acand[nslot] = (unsigned long long)__double_as_longlong(1.0);
  }
  return true;
}

// The decision of iteration C.k for the instances still running, once its
// launches are done (the host polls the running count after it).
static __global__ void k_settle(Ctl C) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= C.n_inst || C.status[b] != ST_RUNNING) return;
  const double r = __longlong_as_double((long long)C.rmax[(C.k % SLOTS) * C.n_inst + b]);
  if (!(r <= 1.79e308) || r <= C.tol || C.k >= C.max_iter)
    record_stop(C, b, C.k, !(r <= 1.79e308) ? ST_DIVERGED : (r <= C.tol ? ST_CONVERGED : ST_MAX_ITER),
                r);
}

// S_out = S_in - alpha Delta S with iteration C.k's step, one CTA per
// (instance, stage): the last iterate of a fixed number of iterations whose
// directions wait for the step (plate).
static __global__ void __launch_bounds__(256) k_apply(Ctl C, Iter S) {
  const int2 it = C.work[blockIdx.x];
  const int b = it.x, s = it.y;
  const Layout L = C.lay[b];
  const double alpha =
      fmin(1.0, __longlong_as_double((long long)C.acand[(C.k % SLOTS) * C.n_inst + b]));
  const long long so = L.s_off + (long long)s * L.nx;
  const long long uo = L.u_off + (long long)s * L.nu;
  for (int t = threadIdx.x; t < L.nx; t += blockDim.x) {
    S.xout[so + t] = S.xin[so + t] - alpha * S.px[so + t];
    S.lout[so + t] = S.lin[so + t] - alpha * S.pl[so + t];
  }
  for (int a = threadIdx.x; a < L.nu; a += blockDim.x)
    S.uout[uo + a] = S.uin[uo + a] - alpha * S.pu[uo + a];
}

// Start iterate into buffer 0 (mode 0 cold, 1 a copy of the current state,
// 2 the current state shifted by one stage, the last repeated) and the
// control words.  Grid (x, instances).
static __global__ void k_init(const Layout* lay, int n_inst, int mode, const double* x0,
                              const double* xc, const double* uc, const double* lc, double* x,
                              double* u, double* lam, unsigned long long* rmax, double* rsq,
                              unsigned long long* acand, int* status, int* n_active) {
  const int b = blockIdx.y;
  const Layout L = lay[b];
  const long long nxs = (long long)L.N * L.nx, nus = (long long)L.N * L.nu;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nxs;
       e += (long long)gridDim.x * blockDim.x) {
    const int s = (int)(e / L.nx), t = (int)(e - (long long)s * L.nx);
    const int ss = (mode == 2) ? min(s + 1, L.N - 1) : s;
    const long long src = L.s_off + (long long)ss * L.nx + t;
    x[L.s_off + e] = (mode == 0) ? x0[L.g_off + t] : xc[src];
    lam[L.s_off + e] = (mode == 0) ? 0.0 : lc[src];
  }
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nus;
       e += (long long)gridDim.x * blockDim.x) {
    const int s = (int)(e / L.nu), a = (int)(e - (long long)s * L.nu);
    const int ss = (mode == 2) ? min(s + 1, L.N - 1) : s;
    u[L.u_off + e] = (mode == 0) ? L.u_cold : uc[L.u_off + (long long)ss * L.nu + a];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    for (int q = 0; q < SLOTS; ++q) {
      rmax[q * n_inst + b] = 0ull;
      rsq[q * n_inst + b] = 0.0;
      acand[q * n_inst + b] = (unsigned long long)__double_as_longlong(1.0);
    }
    status[b] = ST_RUNNING;
    if (b == 0) *n_active = n_inst;
  }
}

// The control words of every slot, cleared.
static __global__ void k_reset(int n, unsigned long long* rmax, double* rsq,
                               unsigned long long* acand) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rmax[i] = 0ull;
  rsq[i] = 0.0;
  acand[i] = (unsigned long long)__double_as_longlong(1.0);
}

// The returned iterate (buffer final_buf[b]) into the current state.
static __global__ void k_gather(const Layout* lay, const int* final_buf, const double* x0b,
                                const double* x1b, const double* u0b, const double* u1b,
                                const double* l0b, const double* l1b, double* xc, double* uc,
                                double* lc, double* u_out) {
  const int b = blockIdx.y;
  const Layout L = lay[b];
  const int fb = final_buf[b];
  const double* xs = fb ? x1b : x0b;
  const double* us = fb ? u1b : u0b;
  const double* ls = fb ? l1b : l0b;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)L.N * L.nx;
       e += (long long)gridDim.x * blockDim.x) {
    xc[L.s_off + e] = xs[L.s_off + e];
    lc[L.s_off + e] = ls[L.s_off + e];
  }
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)L.N * L.nu;
       e += (long long)gridDim.x * blockDim.x) {
    uc[L.u_off + e] = us[L.u_off + e];
    if (u_out) u_out[L.u_off + e] = us[L.u_off + e];
  }
}

#define SDRV_CHECK(call)                                                    \
  do {                                                                      \
    cudaError_t e_ = (call);                                                \
    if (e_ != cudaSuccess) {                                                \
      fprintf(stderr, "nmpc: %s failed: %s\n", #call, cudaGetErrorString(e_)); \
      return NMPC_ERR_CUDA;                                                 \
    }                                                                       \
  } while (0)

template <typename T>
cudaError_t dalloc(T** p, size_t n) {
  *p = nullptr;
  return cudaMalloc((void**)p, std::max<size_t>(n, 1) * sizeof(T));
}

template <typename T>
cudaError_t upload(T* d, const std::vector<T>& v) {
  if (v.empty()) return cudaSuccess;
  return cudaMemcpy(d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
}

// Device state of the driver: three iterate buffers (two ping-pong, one
// current state), two directions (where the problem asks for them), the
// control words and the instance layout.
struct Driver {
  int n = 0;
  std::vector<Layout> lay_h;
  long long n_g = 0, n_x = 0, n_u = 0;  // sum nx (x0), sum N nx, sum N nu
  Layout* lay = nullptr;
  std::vector<Group> groups;
  int2* work = nullptr;
  int n_work = 0;
  double* x0 = nullptr;  // the solve's start state [n_g]
  double* xb[3] = {nullptr, nullptr, nullptr};
  double* ub[3] = {nullptr, nullptr, nullptr};
  double* lb[3] = {nullptr, nullptr, nullptr};
  double *dx[2] = {nullptr, nullptr}, *du[2] = {nullptr, nullptr}, *dl[2] = {nullptr, nullptr};
  unsigned long long *rmax = nullptr, *acand = nullptr;
  double *rsq = nullptr, *fin = nullptr;
  int *status = nullptr, *iters = nullptr, *final_buf = nullptr, *n_active = nullptr;
  bool has_state = false;
};

// An instance's grid: dimension, points per axis and in all, Neumann or not.
struct GridKind {
  int dim, m, ng;
  bool neu;
};

// The thread groups' shape for stages of ng points, n of them in all.
inline void shape_group(Group& g, int sms) {
  g.ppt = g.ng_max > 256 ? 2 : 1;
  g.tps = 32 * ((g.ng_max + 32 * g.ppt - 1) / (32 * g.ppt));
  // at most 256 threads a CTA (8 named barriers); two CTAs' worth of stages
  // for each SM before stages share a CTA
  g.spc = std::max(1, std::min(256 / g.tps, g.n / (2 * sms)));
}

// Offsets from lay_h[b].{N, nx, nu}; the work items (instance, stage) by
// group, even stages first.
inline cudaError_t driver_alloc(Driver& d, const std::vector<GridKind>& grid, bool directions) {
  d.n = (int)d.lay_h.size();
  d.n_g = d.n_x = d.n_u = 0;
  std::vector<int2> work;
  for (int b = 0; b < d.n; ++b) {
    Layout& L = d.lay_h[b];
    L.s_off = d.n_x;
    L.u_off = d.n_u;
    L.g_off = d.n_g;
    d.n_x += (long long)L.N * L.nx;
    d.n_u += (long long)L.N * L.nu;
    d.n_g += L.nx;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  sms = std::max(1, sms);
  // One group per grid kind; where a kind has stages of up to 256 points beside
  // larger ones and more of both than run at once with the larger ones' threads
  // (two CTAs a SM), the smaller ones are a group of their own: a launch more
  // per iteration, but they need not have two points a thread and 288 to 512
  // threads a stage (one 24x24 plate and 511 of 5x5, N = 20, float64: 118 ms a
  // solve in one group, 49 in two).
  for (int kind = 0; kind < 4; ++kind) {
    long long n[2] = {0, 0};  // stages of up to 256 points, of more
    auto of_kind = [&](int b) {
      return grid[b].neu == ((kind & 1) != 0) && (grid[b].dim == 2) == ((kind & 2) != 0);
    };
    for (int b = 0; b < d.n; ++b)
      if (of_kind(b)) n[grid[b].ng > 256] += d.lay_h[b].N;
    const bool split = n[0] > 0 && n[1] > 0 && n[0] + n[1] > 2 * sms;
    for (int large = 0; large < (split ? 2 : 1); ++large) {
      Group g{};
      g.neu = kind & 1;
      g.d2 = kind & 2;
      g.first = (int)work.size();
      for (int par = 0; par < 2; ++par) {
        for (int b = 0; b < d.n; ++b) {
          if (!of_kind(b) || (split && (grid[b].ng > 256) != (large == 1))) continue;
          g.ng_max = std::max(g.ng_max, grid[b].ng);
          for (int s = par; s < d.lay_h[b].N; s += 2) work.push_back(make_int2(b, s));
        }
        if (par == 0) g.n_even = (int)work.size() - g.first;
      }
      g.n = (int)work.size() - g.first;
      if (g.n == 0) continue;
      shape_group(g, sms);
      d.groups.push_back(g);
    }
  }
  d.n_work = (int)work.size();
  cudaError_t e = cudaSuccess;
  auto A = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  A(dalloc(&d.lay, d.n));
  A(dalloc(&d.work, work.size()));
  A(dalloc(&d.x0, d.n_g));
  for (int q = 0; q < 3; ++q) {
    A(dalloc(&d.xb[q], d.n_x));
    A(dalloc(&d.ub[q], d.n_u));
    A(dalloc(&d.lb[q], d.n_x));
  }
  for (int q = 0; directions && q < 2; ++q) {
    A(dalloc(&d.dx[q], d.n_x));
    A(dalloc(&d.du[q], d.n_u));
    A(dalloc(&d.dl[q], d.n_x));
  }
  A(dalloc(&d.rmax, SLOTS * d.n));
  A(dalloc(&d.acand, SLOTS * d.n));
  A(dalloc(&d.rsq, SLOTS * d.n));
  A(dalloc(&d.fin, 2 * d.n));
  A(dalloc(&d.status, d.n));
  A(dalloc(&d.iters, d.n));
  A(dalloc(&d.final_buf, d.n));
  A(dalloc(&d.n_active, 1));
  A(upload(d.lay, d.lay_h));
  A(upload(d.work, work));
  return e;
}

inline void driver_free(Driver& d) {
  void* ptrs[] = {d.lay, d.work, d.x0, d.xb[0], d.xb[1], d.xb[2], d.ub[0], d.ub[1], d.ub[2],
                  d.lb[0], d.lb[1], d.lb[2], d.dx[0], d.dx[1], d.du[0], d.du[1], d.dl[0], d.dl[1], d.rmax, d.acand, d.rsq, d.fin,
                  d.status, d.iters, d.final_buf, d.n_active};
  for (void* p : ptrs)
    if (p) cudaFree(p);
}

inline Ctl make_ctl(const Driver& d, int k, int mode, int max_iter, double tol) {
  Ctl C{};
  C.lay = d.lay;
  C.work = d.work;
  C.rmax = d.rmax;
  C.rsq = d.rsq;
  C.acand = d.acand;
  C.status = d.status;
  C.iters = d.iters;
  C.final_buf = d.final_buf;
  C.fin = d.fin;
  C.n_active = d.n_active;
  C.n_inst = d.n;
  C.k = k;
  C.mode = mode;
  C.max_iter = max_iter;
  C.tol = tol;
  return C;
}

// Launch k's arrays.  Without directions it reads S^k and writes S^{k+1};
// with them it reads S^{k-1} and Delta S^{k-1} (k = 0: S^0), writes S^k and
// Delta S^k.  Iterate k is in buffer k & 1 either way.
inline Iter make_iter(const Driver& d, int k) {
  const bool dir = d.dx[0] != nullptr;
  const int rd = dir ? (k > 0 ? (k - 1) & 1 : 0) : k & 1, wr = dir ? k & 1 : (k + 1) & 1;
  Iter S{};
  S.xin = d.xb[rd];
  S.uin = d.ub[rd];
  S.lin = d.lb[rd];
  S.xout = d.xb[wr];
  S.uout = d.ub[wr];
  S.lout = d.lb[wr];
  S.px = d.dx[rd];
  S.pu = d.du[rd];
  S.pl = d.dl[rd];
  S.dx = d.dx[k & 1];
  S.du = d.du[k & 1];
  S.dl = d.dl[k & 1];
  return S;
}

inline dim3 inst_grid(const Driver& d) { return dim3(8, (unsigned)d.n); }

// A direction kernel over one range of items, overlapping its start with the
// previous launch's end.
template <typename K, typename Args>
cudaError_t launch_stages(K kernel, size_t smem_per_group, const Range& r, const Args& A,
                          const Ctl& C, const Iter& S, cudaStream_t st) {
  if (r.n == 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((r.n + r.spc - 1) / r.spc));
  cfg.blockDim = dim3((unsigned)(r.tps * r.spc));
  cfg.dynamicSmemBytes = smem_per_group * r.spc;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, A, C, S, r);
}

// A solve from d.x0 (already on the device): init NMPC_INIT_*; host polls of
// the running count every check_every iterations.  Fills stats (host, [n])
// and u_out (device or NULL); returns NMPC_OK or the first of NOT_CONVERGED /
// DIVERGED met.
template <class Dir>
int solve(Driver& d, int init, int max_iter, double tol, int check_every, Dir& dir, double* u_out,
          nmpc_stats* stats, cudaStream_t st) {
  if (init != NMPC_INIT_COLD && init != NMPC_INIT_WARM && init != NMPC_INIT_SHIFT)
    return NMPC_ERR_BAD_ARG;
  if (init != NMPC_INIT_COLD && !d.has_state) return NMPC_ERR_BAD_ARG;
  const int mode = init == NMPC_INIT_COLD ? 0 : (init == NMPC_INIT_WARM ? 1 : 2);
  k_init<<<inst_grid(d), 256, 0, st>>>(d.lay, d.n, mode, d.x0, d.xb[2], d.ub[2], d.lb[2], d.xb[0],
                                       d.ub[0], d.lb[0], d.rmax, d.rsq, d.acand, d.status,
                                       d.n_active);
  SDRV_CHECK(cudaGetLastError());
  int active = d.n;
  for (int k = 0; k <= max_iter;) {
    for (int c = 0; c < check_every && k <= max_iter; ++c, ++k)
      SDRV_CHECK(dir(make_ctl(d, k, MODE_SOLVE, max_iter, tol), make_iter(d, k)));
    k_settle<<<(d.n + 127) / 128, 128, 0, st>>>(make_ctl(d, k - 1, MODE_SOLVE, max_iter, tol));
    SDRV_CHECK(cudaGetLastError());
    SDRV_CHECK(cudaMemcpyAsync(&active, d.n_active, sizeof(int), cudaMemcpyDeviceToHost, st));
    SDRV_CHECK(cudaStreamSynchronize(st));
    if (active == 0) break;
  }
  k_gather<<<inst_grid(d), 256, 0, st>>>(d.lay, d.final_buf, d.xb[0], d.xb[1], d.ub[0], d.ub[1],
                                         d.lb[0], d.lb[1], d.xb[2], d.ub[2], d.lb[2], u_out);
  SDRV_CHECK(cudaGetLastError());
  d.has_state = true;
  std::vector<int> status(d.n), iters(d.n);
  std::vector<double> fin(2 * d.n);
  SDRV_CHECK(cudaMemcpyAsync(status.data(), d.status, d.n * sizeof(int), cudaMemcpyDeviceToHost, st));
  SDRV_CHECK(cudaMemcpyAsync(iters.data(), d.iters, d.n * sizeof(int), cudaMemcpyDeviceToHost, st));
  SDRV_CHECK(cudaMemcpyAsync(fin.data(), d.fin, 2 * d.n * sizeof(double), cudaMemcpyDeviceToHost, st));
  SDRV_CHECK(cudaStreamSynchronize(st));
  int rc = NMPC_OK;
  for (int b = 0; b < d.n; ++b) {
    if (stats) {
      stats[b].status = status[b];
      stats[b].iters = iters[b];
      stats[b].res_inf = fin[b];
      stats[b].res_2 = fin[d.n + b];
      stats[b].f64_iters = iters[b] + 1;  // every residual is evaluated in float64
    }
    if (rc == NMPC_OK) {
      if (status[b] == ST_DIVERGED) rc = NMPC_ERR_DIVERGED;
      else if (status[b] != ST_CONVERGED) rc = NMPC_ERR_NOT_CONVERGED;
    }
  }
  return rc;
}

// n_iter iterations from (x_in, u_in, lam_in) (device, packed) into the
// output arrays, no convergence test; out: NULL or host [n][3] = (||K||_inf,
// ||K||_2, alpha) of the last iteration.
template <class Dir>
int iterate(Driver& d, const double* x_in, const double* u_in, const double* lam_in, double* x_out,
            double* u_out, double* lam_out, int n_iter, double* out, Dir& dir, cudaStream_t st) {
  SDRV_CHECK(cudaMemcpyAsync(d.xb[0], x_in, d.n_x * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SDRV_CHECK(cudaMemcpyAsync(d.ub[0], u_in, d.n_u * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SDRV_CHECK(cudaMemcpyAsync(d.lb[0], lam_in, d.n_x * sizeof(double), cudaMemcpyDeviceToDevice, st));
  k_reset<<<(SLOTS * d.n + 127) / 128, 128, 0, st>>>(SLOTS * d.n, d.rmax, d.rsq, d.acand);
  SDRV_CHECK(cudaGetLastError());
  for (int k = 0; k < n_iter; ++k)
    SDRV_CHECK(dir(make_ctl(d, k, MODE_ONESHOT, 0, 0.0), make_iter(d, k)));
  if (d.dx[0]) {
    k_apply<<<d.n_work, 256, 0, st>>>(make_ctl(d, n_iter - 1, MODE_ONESHOT, 0, 0.0),
                                      make_iter(d, n_iter));
    SDRV_CHECK(cudaGetLastError());
  }
  const int fb = n_iter & 1, slot = (n_iter - 1) % SLOTS;
  SDRV_CHECK(cudaMemcpyAsync(x_out, d.xb[fb], d.n_x * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SDRV_CHECK(cudaMemcpyAsync(u_out, d.ub[fb], d.n_u * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SDRV_CHECK(cudaMemcpyAsync(lam_out, d.lb[fb], d.n_x * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (out) {
    std::vector<unsigned long long> rm(d.n), ac(d.n);
    std::vector<double> rs(d.n);
    SDRV_CHECK(cudaMemcpyAsync(rm.data(), d.rmax + (size_t)slot * d.n, d.n * sizeof(unsigned long long),
                               cudaMemcpyDeviceToHost, st));
    SDRV_CHECK(cudaMemcpyAsync(rs.data(), d.rsq + (size_t)slot * d.n, d.n * sizeof(double), cudaMemcpyDeviceToHost, st));
    SDRV_CHECK(cudaMemcpyAsync(ac.data(), d.acand + (size_t)slot * d.n, d.n * sizeof(unsigned long long),
                               cudaMemcpyDeviceToHost, st));
    SDRV_CHECK(cudaStreamSynchronize(st));
    for (int b = 0; b < d.n; ++b) {
      double r, a;
      std::memcpy(&r, &rm[b], sizeof(r));
      std::memcpy(&a, &ac[b], sizeof(a));
      out[3 * b] = r;
      out[3 * b + 1] = std::sqrt(rs[b]);
      out[3 * b + 2] = std::min(1.0, a);
    }
  }
  return NMPC_OK;
}

inline int get_state(const Driver& d, double* x, double* u, double* lam, cudaStream_t st) {
  if (x) SDRV_CHECK(cudaMemcpyAsync(x, d.xb[2], d.n_x * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (u) SDRV_CHECK(cudaMemcpyAsync(u, d.ub[2], d.n_u * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (lam) SDRV_CHECK(cudaMemcpyAsync(lam, d.lb[2], d.n_x * sizeof(double), cudaMemcpyDeviceToDevice, st));
  return NMPC_OK;
}

// The grid Laplacian's neighbour weight, 1 / spacing^2: zero Neumann grids
// (bc 0) include the boundary (spacing 1 / (m - 1)), zero Dirichlet ones hold
// the interior points (spacing 1 / (m + 1)).
inline double neighbour_weight(int m, int bc) {
  const double dp = bc == 0 ? 1.0 / (m - 1) : 1.0 / (m + 1);
  return 1.0 / (dp * dp);
}

// Per grid point the actuator on it, or minus the number of grid steps to the
// nearest one.
inline std::vector<int> actuator_map(int dim, int m, int n_u, const int* act_cell) {
  const int ng = dim == 2 ? m * m : m;
  std::vector<int> of(ng, 0), front;
  for (int a = 0; a < n_u; ++a) front.push_back(act_cell[a]);
  std::vector<char> seen(ng, 0);
  for (int p : front) seen[p] = 1;
  for (int dist = 1; !front.empty(); ++dist) {
    std::vector<int> next;
    for (int p : front) {
      const int ix = p % m, iy = p / m;
      const int q[4] = {ix > 0 ? p - 1 : -1, ix < m - 1 ? p + 1 : -1,
                        dim == 2 && iy > 0 ? p - m : -1, dim == 2 && iy < m - 1 ? p + m : -1};
      for (int c : q)
        if (c >= 0 && !seen[c]) {
          seen[c] = 1;
          of[c] = -dist;
          next.push_back(c);
        }
    }
    front = next;
  }
  for (int a = 0; a < n_u; ++a) of[act_cell[a]] = a;
  return of;
}

}  // namespace stage_drv
