// Types, control words and device helpers shared by the heat solver's kernels:
// the instance table, the iteration's arguments, the slab geometry, float64 /
// float32 conversions, the decision of an iteration, the split residual's
// rounding bound and the publication of its norms.
#pragma once

#include <cooperative_groups.h>
#include <type_traits>
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stddef.h>
#include <stdint.h>

namespace nmpc_dev {

namespace cg = cooperative_groups;

constexpr int RES_SLOTS = 16;    // rolling residual history per instance
// iterations over which a split residual r with r - e <= threshold (e its
// rounding bound) that has not decreased hands over to the float64 residual
// although r itself stays above the threshold (its rounding floor)
constexpr int SPLIT_PATIENCE = 12;
static_assert(SPLIT_PATIENCE + 2 < RES_SLOTS, "history slots read by decide()");
// res_err of an iteration that evaluated the float64 residual (above the bits
// of every non-negative double or NaN, so atomicMax keeps it)
constexpr unsigned long long RES_FULL_MARK = 0xfff0000000000000ull;
constexpr int MAX_NU = 64;

struct InstDev {
  int dim, mx, my, ng;
  int N, nu, act_off;
  int dist_off;  // where in act (in ints) a byte per cell says how many grid
                 // steps the nearest actuator is away, 255 beyond 2; 0: nowhere
  long long s_off;  // offset of stage 1 in packed x / lam
  long long u_off;  // offset in packed u
  long long g_off;  // offset in packed x0 / ref
  double h, q, r, qf, gamma, k0, k1, b0, cx, cy;
  // derived (derive()): float64 2 (cx + cy), h qf, h r + gamma; float32 copies
  double dcoef, hqf, auu;
  float fh, fcx, fcy, fdc, fk0, fk1, fk1h, fk01, fq, fb0, fhqf, fauu;
};

// Fill the derived fields of an instance from its parameters.
__host__ __device__ inline void derive(InstDev& I) {
  I.dcoef = 2.0 * (I.cx + I.cy);
  I.hqf = I.h * I.qf;
  I.auu = I.h * I.r + I.gamma;
  I.fh = (float)I.h;
  I.fcx = (float)I.cx;
  I.fcy = (float)I.cy;
  I.fdc = (float)I.dcoef;
  I.fk0 = (float)I.k0;
  I.fk1 = (float)I.k1;
  I.fk1h = (float)(0.5 * I.k1);
  I.fk01 = (float)(I.k0 * I.k1);
  I.fq = (float)I.q;
  I.fb0 = (float)I.b0;
  I.fhqf = (float)I.hqf;
  I.fauu = (float)I.auu;
}

enum { MODE_SOLVE = 0, MODE_ONESHOT = 1 };
enum { ST_RUNNING = 0, ST_CONVERGED = 1, ST_DIVERGED = 2, ST_MAX_ITER = 3 };

struct IterArgs {
  const InstDev* inst;
  const int2* work;  // (instance, 0-based stage)
  int n_work;
  int n_inst;
  const int* act;
  const double* x0;
  const double* ref;
  // state buffers: solve mode reads [k & 1] and writes [(k + 1) & 1];
  // one-shot mode reads [0] and writes [1]
  const double* xin[2];
  const double* uin[2];
  const double* lin[2];
  double* xout[2];
  double* uout[2];
  double* lout[2];
  // control (solve mode)
  int* iter_k;
  unsigned long long* res_inf;   // [RES_SLOTS][n_inst], bits of non-negative doubles
  unsigned long long* res_err;   // [RES_SLOTS][n_inst] bound on a split residual's rounding error
  double* res_sq;                // [RES_SLOTS][n_inst]
  unsigned long long* res_first; // [n_inst] ||K(S^0)||_inf
  int* status;
  int* iters;
  int* final_buf;
  double* fin_inf;
  double* fin_2;
  int* f64_count;  // [n_inst] iterations that evaluated the float64 residual
  int* full0;      // [n_inst] 1: iteration 0 does (warm starts)
  int* n_active;
  // persistent launch: [0] barrier arrivals, [1] barrier generation, [2] stop
  // (no instance running), [3] a wait ran out of time
  unsigned* gsync;
  double tol, div_limit, alpha;
  double split_min;  // below max(tol, split_min) iterations use the float64 residual
  int max_iter, n_lo, n_u_it;
  // upper-layer variant: 0 Jacobi (eq. 15, every stage from iterate k);
  // 1 red-black Gauss-Seidel (the stage-block form of eq. 18 in the order
  // even stages, then odd stages): an iteration is two launches, half 0
  // updating the even 0-based stages from iterate k, half 1 the odd ones
  // with x_{i-1}, lambda_{i+1} already updated (launch index j = 2 i + half)
  int rb;
  // red-black: the cluster, strip and patch lists hold the items of even
  // stages first (this many), then those of odd stages; a half-sweep
  // launch covers its own range only
  int n_work_even, n_strips_even, n_patches_even;
  long long grid_wait;  // spin budget of one grid-barrier wait (SM clock cycles)
  int resid_only;  // one-shot: residual norms only (float64)
  int full_all;    // every residual in float64 (FP64 precision)
  int csize;       // CTAs per work item (cluster size)
  int stage;       // float64 slab inputs staged in shared memory (1) or read in place
  int local_u;     // u-iteration through the actuators' local responses (1) or full sweeps
  int box_r;       // half-width of a local-response box, 2 (n_lo - 1)
  int slab_max;    // records per slab (padded positions, halo rows and pads included)
  // lower-layer work arrays: shared memory (scratch == nullptr) or a global
  // slab of scratch_stride bytes per CTA
  char* scratch;
  long long scratch_stride;
  // strip path (k_strip): (instance, stage, first own column, first own row)
  // per strip
  const int4* strips;
  int n_strips;
  int strip_x, strip_y;  // own columns and rows per strip
  const float* ref_f;    // ref truncated to float32 (d2f) for k_strip2's split residual
  // the tail plan (k_strip2, solves): strips of tail_y own rows, taken by a
  // launch when the running-instance count that k_patch recorded before it
  // (*strip_run) is at most tail_below (n_tail = 0: no tail plan)
  const int4* tail;
  int n_tail, n_tail_even, tail_y, tail_below;
  int* strip_run;
  // k_patch: (instance, stage, actuator) per warp; v3 per control (float64)
  const int4* patches;
  int n_patches;
  double* v3g;
  // line path (k_line): (instance, stage, cells per lane, 0) per 1D stage;
  // solve mode walks the items of running instances (k_compact_lines)
  const int4* lines;
  int n_lines;
  int4* lines_act;
  int* n_lines_act;
};

struct Cl {
  int C, rank;
  __device__ __forceinline__ void sync() const {
    if (C > 1) cg::this_cluster().sync();
    else __syncthreads();
  }
  template <typename T>
  __device__ __forceinline__ T* map(T* p, int r) const {
    return cg::this_cluster().map_shared_rank(p, r);
  }
};

// Quotient q / d for 0 <= q < 2^22, d >= 1, inv = 1.0f / d: the float
// estimate is off by at most one and is corrected.
__device__ __forceinline__ int fdiv(int q, int d, float inv) {
  const int j = __float2int_rz(__int2float_rz(q) * inv);
  const int r = q - j * d;
  return j + (r >= d ? 1 : 0) - (r < 0 ? 1 : 0);
}

// ---------------------------------------------------------------------------
// Work-item slab in shared memory (or a global scratch slab).
//
// The stage grid is split across the C cluster ranks in whole rows (2D) or
// segments (1D), `per` rows or cells per rank (the last non-empty rank may
// hold fewer, later ranks none).  2D: a rank's slab is a padded layout of
// (rows + 2) x W positions, W = mx + 2, interior cell (row j, column i) at
// p = (j + 1) W + i + 1; padded rows 0 and rows + 1 hold the neighbouring
// ranks' boundary rows (the halo) or zeros at the grid's Dirichlet ring,
// columns 0 and W - 1 are zero.  1D: one padded row, cell q at p = q + 1,
// positions 0 and n + 1 the halo or zero.  The five-point stencil reads
// p +- 1 and p +- Wv with Wv = W in 2D and Wv = 0 in 1D (the cell itself,
// under the zero vertical weight).  Each position holds one record of
// NUM_FIELDS values of T (work record) and, when the float64 inputs are
// staged, one record of NUM_SFIELDS doubles: a field access is one
// shared-memory access at a fixed offset from the record.  A rank that writes
// a boundary value also stores it into the neighbour's halo record.
enum WField { F_B2 = 0, F_DP, F_AX, F_RG, F_V1, F_P1, F_Y5, F_W1, F_Y4, F_E1, F_E2, NUM_FIELDS };
// NUM_FIELDS is odd: consecutive records start in distinct banks.
// Split residual: float copies of x, lambda and Phi(x) in the F_Y5, F_W1 and
// F_Y4 fields (dead before those are written).
enum SField { S_X = 0, S_L, S_XP, S_LN, S_RF, S_PH };
constexpr int NUM_SFIELDS = 7;  // 14 words per record: 16 consecutive records hit distinct bank pairs

struct Geo {
  int n;       // cells of this rank
  int cols;    // cells per interior row: 2D mx, 1D n
  int rows;    // interior rows: 2D slab rows, 1D 1
  int W;       // padded row length
  int Wv;      // position distance of the vertical stencil neighbours: 2D W, 1D 0
  int p0;      // position of the first cell: 2D W + 1, 1D 1
  int plen;    // padded positions: 2D (rows + 2) W, 1D n + 2
  int lo;      // first grid cell of the slab
  int r0;      // first grid row (2D) / cell (1D) of the slab
  int per;     // rows (2D) / cells (1D) per rank
  int edge;    // cells of the first (last) row: 2D mx, 1D 1
  int up_off;  // position shift into rank - 1's layout (its bottom / right halo)
  int dn_off;  // position shift back into rank + 1's layout (its top / left halo)
  bool d2;     // 2D grid
  bool up, dn; // rank - 1 / rank + 1 hold cells and exchange halos with this rank
};

__device__ __forceinline__ Geo geo_of(const InstDev& I, int C, int rank) {
  Geo g;
  g.d2 = (I.dim == 2);
  const int nun = g.d2 ? I.my : I.mx;
  g.per = (nun + C - 1) / C;
  const int a = min(rank * g.per, nun), b = min(a + g.per, nun);
  g.r0 = a;
  g.n = g.d2 ? (b - a) * I.mx : b - a;
  g.cols = g.d2 ? I.mx : b - a;
  g.rows = g.d2 ? b - a : 1;
  g.W = g.d2 ? I.mx + 2 : g.per + 2;
  g.Wv = g.d2 ? g.W : 0;
  g.p0 = g.d2 ? g.W + 1 : 1;
  g.plen = g.d2 ? (g.rows + 2) * g.W : g.n + 2;
  g.lo = g.d2 ? a * I.mx : a;
  g.edge = g.d2 ? I.mx : 1;
  g.up_off = g.d2 ? g.per * g.W : g.per;
  g.dn_off = g.d2 ? (b - a) * g.W : (b - a);
  g.up = (rank > 0) && (b > a);
  g.dn = (b < nun) && (b > a);
  return g;
}

// The NC cells a thread carries through a pass: positions, and bit masks of
// the slots that hold a cell and of those whose value also goes to
// rank - 1's / rank + 1's halo.  Slot k holds cell q = first + k blockDim.  A
// slot past the slab gets position p0, whose stencil neighbours lie inside
// every rank's records: its loads are harmless, its stores are skipped.
template <int NC>
struct Cells {
  int p[NC];
  unsigned valid, pu, pd;
};

template <int NC>
__device__ __forceinline__ Cells<NC> cells_of(const Geo& g, int first) {
  Cells<NC> cs;
  cs.valid = 0u;
  cs.pu = 0u;
  cs.pd = 0u;
  const int bd = blockDim.x;
  const int cols = max(g.cols, 1);
  int j = first / cols, i = first - j * cols;
  const int dj = bd / cols, di = bd - dj * cols;
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    const int q = first + k * bd;
    const bool v = q < g.n;
    cs.p[k] = v ? g.p0 + j * g.W + i : g.p0;
    cs.valid |= (v ? 1u : 0u) << k;
    cs.pu |= ((v && g.up && q < g.edge) ? 1u : 0u) << k;
    cs.pd |= ((v && g.dn && q >= g.n - g.edge) ? 1u : 0u) << k;
    i += di;
    j += dj;
    if (i >= cols) {
      i -= cols;
      ++j;
    }
  }
  return cs;
}

// Slot of a pass: mask bit (round * NC + k), slot k, cell q, position p, and
// whether it holds a cell.
struct Slot {
  int kk, k, q, p;
  bool v;
};

// One pass over the rank's cells.  Rounds of NC cells per thread (one round
// for shared-memory slabs, whose cells the host sizes to fit; several for
// global slabs); within a round, groups of G slots: every slot's loads and
// arithmetic (ld) come before the group's stores (st), so a group forms G
// independent dependency chains.
template <int NC, int G, bool MULTI, typename V, typename LD, typename ST>
__device__ __forceinline__ void pass(const Geo& g, const Cells<NC>& c0, LD ld, ST st) {
  static_assert(NC % G == 0, "group size must divide the cells per thread");
  const int rounds = MULTI ? (g.n + NC * (int)blockDim.x - 1) / (NC * (int)blockDim.x) : 1;
  for (int r = 0; r < rounds; ++r) {
    Cells<NC> cs = c0;
    if (MULTI && r > 0) cs = cells_of<NC>(g, threadIdx.x + r * NC * blockDim.x);
#pragma unroll
    for (int k0 = 0; k0 < NC; k0 += G) {
      V v[G];
#pragma unroll
      for (int k = 0; k < G; ++k) {
        const Slot sl{r * NC + k0 + k, k0 + k, (int)threadIdx.x + (r * NC + k0 + k) * (int)blockDim.x,
                      cs.p[k0 + k], ((cs.valid >> (k0 + k)) & 1u) != 0u};
        v[k] = ld(sl, cs);
      }
#pragma unroll
      for (int k = 0; k < G; ++k) {
        const Slot sl{r * NC + k0 + k, k0 + k, (int)threadIdx.x + (r * NC + k0 + k) * (int)blockDim.x,
                      cs.p[k0 + k], ((cs.valid >> (k0 + k)) & 1u) != 0u};
        st(sl, cs, v[k]);
      }
    }
  }
}

// Shared-memory address of a generic pointer into this CTA's shared memory,
// and the same location in cluster rank r's shared memory.
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned map_rank(unsigned a, int r) {
  unsigned out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(a), "r"(r));
  return out;
}
// Store v to a cluster shared-memory address when flag != 0 (predicated, no branch).
__device__ __forceinline__ void push_if(unsigned addr, float v, unsigned flag) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.shared::cluster.f32 [%0], %1;\n}"
               :: "r"(addr), "f"(v), "r"(flag) : "memory");
}
__device__ __forceinline__ void push_if(unsigned addr, double v, unsigned flag) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.shared::cluster.f64 [%0], %1;\n}"
               :: "r"(addr), "d"(v), "r"(flag) : "memory");
}

// Programmatic dependent launch: let the next launch in the stream start its
// CTAs now, and wait until the previous launch has finished and its writes
// are visible (both no-ops for launches without the attribute).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Rank owning grid cell c and its padded position there.
__device__ __forceinline__ int owner_of(int c, const Geo& g, int mx, int& p) {
  if (g.d2) {
    const int row = c / mx, col = c - row * mx;
    const int r = row / g.per;
    p = (row - r * g.per + 1) * g.W + col + 1;
    return r;
  }
  const int r = c / g.per;
  p = c - r * g.per + 1;
  return r;
}

__device__ __forceinline__ double phi_d(double w, double k0, double k1) {
  return k0 * (w + 0.5 * k1 * w * w);
}

__device__ __forceinline__ double abs_or_inf(double v) {
  const double a = fabs(v);
  return (a <= 1.79e308) ? a : CUDART_INF;  // NaN and Inf count as +Inf
}

// Bits of |v|: non-negative doubles order as integers, NaN above infinity.
__device__ __forceinline__ unsigned long long abs_bits(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// max(a, b) that returns NaN when either is NaN (one instruction)
__device__ __forceinline__ float fmax_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ double dmax_nan(double a, double b) {
  return (a != a) ? a : ((b != b || b > a) ? b : a);
}

// float64 <-> float32 by IEEE-754 bit manipulation on the integer ALUs (the
// float64 pipe issues 2 lanes per clock per SM on this part).  d2f truncates
// toward zero (relative error < 2^-23) for magnitudes in [2^-126, 2^128);
// the magnitude's high word is clamped to that range first (two min/max
// instructions instead of two compare/select pairs), so +-0 stays +-0,
// smaller magnitudes become floats below 2^-146 (of the right sign), and
// 2^128 and beyond, Inf and NaN become Inf or NaN (never a finite value).
// f2d is exact for normal floats; subnormal floats become +-0.
__device__ __forceinline__ float d2f(double d) {
  const unsigned hi = (unsigned)__double2hiint(d);
  const unsigned lo = (unsigned)__double2loint(d);
  const unsigned a = min(hi & 0x7fffffffu, 0x47f00000u);
  // exponent rebiased (1023 -> 127) and the top 23 mantissa bits, in one funnel shift
  const unsigned bits = __funnelshift_l(lo, max(a, 0x38000000u) - 0x38000000u, 3);
  return __uint_as_float(bits | (hi & 0x80000000u));
}

__device__ __forceinline__ double f2d(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned a = b & 0x7fffffffu;
  unsigned hi = (a >> 3) + 0x38000000u;  // exponent rebiased (127 -> 1023)
  unsigned lo = a << 29;
  hi = (a < 0x00800000u) ? 0u : hi;  // zero or subnormal
  lo = (a < 0x00800000u) ? 0u : lo;
  hi = (a >= 0x7f800000u) ? (0x7ff00000u | (a >> 3)) : hi;  // Inf, NaN
  return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)lo);
}

// Sum of the stencil neighbours' values, each weighted by its axis
// coefficient; cells outside the interior grid are zero (Dirichlet ring).
template <typename V, typename G>
__device__ __forceinline__ V nbr_sum(int c, int ix, int iy, int mx, int my, V cx, V cy, G g) {
  V sx = V(0), sy = V(0);
  if (ix > 0) sx += g(c - 1);
  if (ix < mx - 1) sx += g(c + 1);
  if (iy > 0) sy += g(c - mx);
  if (iy < my - 1) sy += g(c + mx);
  return cx * sx + cy * sy;
}

struct BlockRed {
  double mx[32];
  double sq[32];
  float4 mg[32];
};

__device__ __forceinline__ void block_reduce_store(double vmax, double vsq, BlockRed* red,
                                                   double* out_max, double* out_sq) {
  for (int o = 16; o > 0; o >>= 1) {
    vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    vsq += __shfl_xor_sync(0xffffffffu, vsq, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    red->mx[wid] = vmax;
    red->sq[wid] = vsq;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0, s = 0.0;
    const int nw = (blockDim.x + 31) >> 5;
    for (int w = 0; w < nw; ++w) {
      m = fmax(m, red->mx[w]);
      s += red->sq[w];
    }
    *out_max = m;
    *out_sq = s;
  }
}

// Split residual: float32 partial norms (max, sum of squares) and the four
// magnitude maxima of its rounding bound, block-reduced; thread 0 receives the
// norms in float64 and the maxima in mags[4].
__device__ __forceinline__ void block_reduce_store_f(float vmax, float vsq, float4 mg,
                                                     BlockRed* red, double* out_max,
                                                     double* out_sq, float* mags) {
  for (int o = 16; o > 0; o >>= 1) {
    vmax = fmax_nan(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    vsq += __shfl_xor_sync(0xffffffffu, vsq, o);
    mg.x = fmaxf(mg.x, __shfl_xor_sync(0xffffffffu, mg.x, o));
    mg.y = fmaxf(mg.y, __shfl_xor_sync(0xffffffffu, mg.y, o));
    mg.z = fmaxf(mg.z, __shfl_xor_sync(0xffffffffu, mg.z, o));
    mg.w = fmaxf(mg.w, __shfl_xor_sync(0xffffffffu, mg.w, o));
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    red->mx[wid] = f2d(vmax);
    red->sq[wid] = f2d(vsq);
    red->mg[wid] = mg;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0, s = 0.0;
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    const int nw = (blockDim.x + 31) >> 5;
    for (int w = 0; w < nw; ++w) {
      m = dmax_nan(m, red->mx[w]);
      s += red->sq[w];
      g.x = fmaxf(g.x, red->mg[w].x);
      g.y = fmaxf(g.y, red->mg[w].y);
      g.z = fmaxf(g.z, red->mg[w].z);
      g.w = fmaxf(g.w, red->mg[w].w);
    }
    *out_max = m;
    *out_sq = s;
    mags[0] = g.x;
    mags[1] = g.y;
    mags[2] = g.z;
    mags[3] = g.w;
  }
}

// Per-work-item shared scalars (the slab records follow).
template <typename T>
struct SmallShared {
  unsigned long long amask[512];  // per thread: which of its cells carry an actuator
  BlockRed red;
  double red_out[2];
  double u[MAX_NU];
  T b3[MAX_NU];
  T v3[MAX_NU];
  T b1a[MAX_NU];  // state-equation row K1 at each actuator cell (owner rank only)
  T y4a[MAX_NU];  // lambda-part of Y(0) at each actuator cell
  T v3n[MAX_NU];
  int act[MAX_NU];
  double lact[MAX_NU];  // lambda at the actuator cells
  int bar_code;         // persistent launch: the grid barrier's stop / error bits
  int skip;
  int full;
};

__device__ __forceinline__ double to_double(float v) { return f2d(v); }
__device__ __forceinline__ double to_double(double v) { return v; }

// float64 -> T off the float64 pipe (truncating for float)
template <typename T>
__device__ __forceinline__ T to_T(double v);
template <>
__device__ __forceinline__ float to_T<float>(double v) { return d2f(v); }
template <>
__device__ __forceinline__ double to_T<double>(double v) { return v; }

// The float64 or the float32 copy of a constant, for arithmetic in T.
template <typename T>
__device__ __forceinline__ T pick(double d, float f);
template <>
__device__ __forceinline__ float pick<float>(double, float f) { return f; }
template <>
__device__ __forceinline__ double pick<double>(double d, float) { return d; }

// 1 / v rounded to nearest (the same value as the IEEE division)
__device__ __forceinline__ float rcp_T(float v) { return __frcp_rn(v); }
__device__ __forceinline__ double rcp_T(double v) { return __drcp_rn(v); }

__device__ __forceinline__ void cp_async8(void* dst_smem, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src));
}

// cp_async8 that writes zeros instead when `valid` is false (source size 0:
// nothing is read; src must still be a valid address)
__device__ __forceinline__ void cp_async8_zfill(void* dst_smem, const void* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src),
               "r"(valid ? 8 : 0));
}

// Iteration index (relative to *iter_k) and half-sweep of launch j.
__device__ __forceinline__ int launch_iter(const IterArgs& A, int j) { return A.rb ? (j >> 1) : j; }
__device__ __forceinline__ int launch_half(const IterArgs& A, int j) { return A.rb ? (j & 1) : 0; }
// Whether stage s is updated by half-sweep `half` (every stage under Jacobi).
__device__ __forceinline__ bool stage_in_half(const IterArgs& A, int s, int half) {
  return !A.rb || ((s & 1) == half);
}

// Whether iteration k >= 1, whose predecessor left the residual r (not yet
// converged or diverged), evaluates the float64 residual: once r (split or
// float64) is at or below T = max(tol, split_min) (it is then expected at or
// below T, or the split residual could not resolve it).  A float64 residual
// above T hands back to the split residual where the split residual itself
// had reached T (the iterates' residual rose again) or the float64 one was
// iteration 0's; a float64 phase that began on the split residual's rounding
// floor or has lasted longer stays.  The floor: a split residual with r - e <=
// T (it can no longer show that the float64 residual is above T) and no lower
// than SPLIT_PATIENCE iterations before.  hist(kk, r, e): iteration kk's
// residual and the bits of its bound (RES_FULL_MARK: float64).
template <typename Hist>
__device__ __forceinline__ bool switch_to_full(const IterArgs& A, int k, double r, bool prev_full,
                                               unsigned long long e_bits, Hist hist) {
  const double T = fmax(A.tol, A.split_min);
  double r2;
  unsigned long long e2;
  if (r <= T) return true;
  if (prev_full) {
    if (k < 2) return false;
    hist(k - 2, r2, e2);
    return e2 == RES_FULL_MARK || !(r2 <= T);
  }
  const double e = __longlong_as_double((long long)e_bits);
  if (r - e <= T && k - 1 - SPLIT_PATIENCE >= 0) {
    hist(k - 1 - SPLIT_PATIENCE, r2, e2);
    return r >= r2;
  }
  return false;
}

// Iteration k's decision for instance b, from its residual history
// (iteration k - 1), with no side effects: skip (finished before, or k past
// max_iter: `before`; or finished now: st != ST_RUNNING) and whether the
// residual is evaluated in float64.  Control words are read around L1 (other
// CTAs write them within a persistent launch).
struct Decision {
  int skip, full, before, st, pslot;
  double r;
};

__device__ __forceinline__ Decision decide(const IterArgs& A, int b, int k) {
  Decision d{0, 1, 0, ST_RUNNING, (k > 0) ? ((k - 1) % RES_SLOTS) * A.n_inst + b : 0, 0.0};
  // every control word the decision reads, loaded at once
  const int status_b = __ldcg(A.status + b);
  const int f0 = __ldcg(A.full0 + b);
  const unsigned long long r_bits = __ldcg(A.res_inf + d.pslot);
  const unsigned long long r0_bits = __ldcg(A.res_first + b);
  const unsigned long long e_bits = __ldcg(A.res_err + d.pslot);
  if (k > A.max_iter || status_b != ST_RUNNING) {
    d.skip = 1;
    d.before = 1;
    return d;
  }
  bool switch_now = false;
  if (k > 0) {
    d.r = __longlong_as_double((long long)r_bits);
    const double r0 = __longlong_as_double((long long)r0_bits);
    const bool prev_full = e_bits == RES_FULL_MARK;
    if (!(d.r <= 1.79e308) || d.r > A.div_limit * fmax(r0, 1e-300)) {
      d.st = ST_DIVERGED;
    } else if (prev_full && d.r <= A.tol) {
      d.st = ST_CONVERGED;
    } else {
      switch_now = switch_to_full(A, k, d.r, prev_full, e_bits, [&](int kk, double& r, unsigned long long& e) {
        const int sl = (kk % RES_SLOTS) * A.n_inst + b;
        r = __longlong_as_double((long long)__ldcg(A.res_inf + sl));
        e = __ldcg(A.res_err + sl);
      });
    }
  }
  if (d.st != ST_RUNNING) {
    d.skip = 1;
  } else {
    d.full = (A.full_all || switch_now || k == A.max_iter || (k == 0 && f0)) ? 1 : 0;
  }
  return d;
}

// decide() for work item (b, s), taken by one thread; the CTA of stage 0,
// cluster rank 0 keeps the books: it records a finished instance (status,
// returned iterate k - 1), counts the float64-residual iterations, and clears
// the residual slot of iteration k + 1.
static __device__ __noinline__ void control_decision(const IterArgs& A, int b, int s, int k, const Cl& cl,
                                              int& skip_out, int& full_out) {
  const Decision d = decide(A, b, k);
  if (!d.before && s == 0 && cl.rank == 0) {
    if (d.st != ST_RUNNING) {
      A.status[b] = d.st;
      A.iters[b] = k - 1;
      A.final_buf[b] = (k - 1) & 1;
      A.fin_inf[b] = d.r;
      A.fin_2[b] = sqrt(__ldcg(A.res_sq + d.pslot));
      atomicSub(A.n_active, 1);
    } else {
      if (d.full) A.f64_count[b] += 1;
      const int nslot = ((k + 1) % RES_SLOTS) * A.n_inst + b;
      A.res_inf[nslot] = 0ull;
      A.res_err[nslot] = 0ull;
      A.res_sq[nslot] = 0.0;
    }
  }
  skip_out = d.skip;
  full_out = d.full;
}

// Rounding bound of the split residual over a set of cells (unit roundoff
// u = 2^-24).  x and lambda are truncated to float32 (2u), Phi, Phi' and the
// five-point sums are evaluated in float32 (a few u each): with X, Lm the
// maxima of |x|, |lambda| over the cells and their stencil neighbours, every
// O(h) term is off by at most 16 u h S, S = 4 (cx + cy) (Phi_max + Phi'_max
// Lm) + b0 sum|u| + (q + qf [last stage]) (X + max|ref|); the float64
// differences and the stage-gradient rows are truncated once (2u) and summed
// (u).  With diff32 the differences are instead taken in float32 from the
// truncated values (2u each, then rounded: u), which adds 4u max(X, Lm) with
// X, Lm covering the neighbouring stages' values as well.  Every cell's
// |K_split - K| is below the bound.  It is evaluated in float32 (its own
// rounding, a few u relative, is far inside the factor 16) and rounded up by
// 1%.  mags: X, Lm, max |difference or K2|, max |ref|; usum: sum over the
// stage's controls of |u| (float32).
// With Gm >= 0 the Laplacian of Phi is instead summed in difference form,
// sum_n c_n k0 (x_n - x_c)(1 + k1/2 (x_n + x_c)), from the truncated values:
// each term is off by k0 (1 + |k1| X)(4u X + 7u Gm), Gm the largest
// neighbour difference, so that part of S is dcoef k0 (1 + |k1| X)(4 X + 7
// Gm) / 8 (no cancellation of the O(dcoef Phi) terms).
__device__ __forceinline__ double split_bound(const InstDev& I, bool last, const float* mags,
                                              float usum, bool diff32 = false, float Gm = -1.0f) {
  const float u32 = 5.9604645e-08f;
  const float Xm = mags[0], Lm = mags[1], Dm = mags[2], Rm = mags[3];
  const float ak0 = fabsf(I.fk0), ak1 = fabsf(I.fk1);
  const float pmax = ak0 * (Xm + 0.5f * ak1 * Xm * Xm);
  const float dpmax = ak0 * (1.0f + ak1 * Xm);
  const float phi_part = (Gm >= 0.0f) ? I.fdc * dpmax * (4.0f * Xm + 7.0f * Gm) * 0.125f
                                      : 2.0f * I.fdc * pmax;
  const float S = phi_part + 2.0f * I.fdc * dpmax * Lm + fabsf(I.fb0) * usum +
                  (I.fq + (last ? I.fhqf / I.fh : 0.0f)) * (Xm + Rm);
  const float Dterm = 3.0f * Dm + (diff32 ? 4.0f * fmaxf(Xm, Lm) : 0.0f);
  return f2d(1.01f * u32 * (Dterm + 16.0f * I.fh * S));
}

// Residual norms of a work item (max, sum of squares) and, for the split
// residual, its rounding bound (else RES_FULL_MARK), into iteration k's slot of
// instance b.
__device__ __forceinline__ void publish_residual(const IterArgs& A, int slot, int b, int k,
                                                 double rmax, double rsq, double e, bool full) {
  atomicMax(&A.res_err[slot], full ? RES_FULL_MARK : (unsigned long long)__double_as_longlong(e));
  atomicMax(&A.res_inf[slot], (unsigned long long)__double_as_longlong(rmax));
  atomicAdd(&A.res_sq[slot], rsq);
  if (k == 0 && A.res_first)
    atomicMax(&A.res_first[b], (unsigned long long)__double_as_longlong(rmax));
}

}  // namespace nmpc_dev
