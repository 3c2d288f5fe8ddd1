// Preconditioner apply z = M M^T r (Sec. 2.8) on per-level vectors, for the
// OrthS factorization (the interpolative variants, whose kept dofs are
// arbitrary subsets, run k_apply of solve_kernels.cuh).
//
// Every elimination step t has its own vector X_t: the values of the step's
// clusters, cluster after cluster (X_1 is the vector in cluster order that the
// apply works on in place).  The coarse values that an interface keeps are
// written straight to their place in X_{t+1} (a parent cluster is its
// children's coarse values in order), so every operand is a contiguous range:
// no index lists.  With Y = U^{-T} (Sec. 2.4, 2.5) and the coarse basis Q_pc
// (Sec. 2.6.1; the fine dofs are identity in M^T A M, so only Q_pc and the
// forward values are needed), per step
//   forward   E_s: y_s = Y x_s; u_s = X_ns y_s
//             S_p: v = x_p - sum of the u's pieces for p (separator order);
//                  y_p = Y v; X_{t+1}(p) = c = Q_pc^T y_p
//   backward  S_p: x_p = Y^T (y_p + Q_pc (X_{t+1}(p) - c)), also copied to p's
//                  piece of the operand of every adjacent separator
//             E_s: x_s = Y^T (y_s - X_ns^T x_n)
// Two dependent products per operation would be two phases.  The combined
// blocks G_ns = X_ns Y and P_p = Q_pc^T Y (formed once per factorization,
// k_combine) make each a single one, [y; u] = [Y; G] x_s and
// [y; c] = [Y; P] v on the way down, x_s = [Y; G]^T [y; -x_n] and
// x_p = [Y; P]^T [y; X_{t+1} - c] on the way back: the same bytes, half the
// phases.  G costs n^2 m operations per separator, next to nothing above the
// leaves; steps where it would be dear (the leaves) keep X_ns and two phases.
//
// GB300 mapping.  The apply is bound by its chain of dependent phases: the
// factor's bytes alone take a fifth to a third of its time.
//  * Work items are warp-sized: 2 to 16 rows of a row product, or 1 to 32
//    columns of a column product, 16-byte loads, 8 in flight per lane,
//    reductions by shuffles, no block barrier inside a phase.  A table per
//    phase lists them; the launch deals them over all its warps.
//  * Every warp copies the descriptors of its first item of every phase to
//    shared memory when the kernel starts, and issues that item's first loads
//    of factor data before it waits for the phase's operands; the descriptors
//    of later items are read one item ahead.
// Every item is computed by one warp in a fixed order whatever the launch
// shape, so z has the same bits for every shape.
//
// Measured, one application, slot-list kernel (nine phases per step) -> this
// one: 64^3 diffusion FP32 (0.46 GB of factor) 0.78 -> 0.46 ms, FP64 1.78 ->
// 1.21; 96^3 FP32 (1.2 GB) 1.59 -> 0.92; 300 x 280 FP32 0.52 -> 0.21; 64 x 64
// FP64 0.31 -> 0.15.  A phase of few items takes 2.5-4 us, most of it L2 round
// trips (operands, stores before the barrier, the barrier itself); the leaf
// phases run at 6-7 TB/s.  Tried and not kept: one cluster (hardware barrier) or
// one CTA (vectors in shared memory) for the steps near the root, no faster
// than the whole grid; double-buffered items with fewer warps, 0.77 ms at
// 64^3 FP32 against 0.46: the number of warps hides the latency better.
#pragma once

#include <algorithm>
#include <type_traits>

#include "dense_tiles.cuh"
#include "solve_kernels.cuh"

namespace spand {

enum LevelPhaseKind : int32_t {
  LP_FE = 0,  // [y; u] = [Y; G] x_s
  LP_FY,      // y = Y x_s
  LP_FU,      // u = X_ns y
  LP_FS,      // [y; c] = [Y; P] (x_p - sum u)
  LP_BS,      // x_p = [Y; P]^T [y; X_{t+1} - c]
  LP_BE,      // x_s = [Y; G]^T [y; -x_n]
  LP_BA,      // z = y - X_ns^T x_n
  LP_BX       // x_s = Y^T z
};

template <typename TF>
struct LevelOp {     // one operation of a step: E_s or S_p
  const TF* A;       // E: G (m x n), or X^T (n x m) for the two-phase form; S: P (m x n), nullptr: not sparsified
  const TF* Y;       // pivot inverse (lower, n x n); nullptr (S only): not scaled, values pass through
  int32_t n, m, lda, ldy;
  int64_t x;         // place in X_t
  int64_t y;         // place of y (kept from the forward to the backward sweep)
  int64_t z;         // E, two-phase form: place of the backward intermediate
  int64_t u;         // E: place of u_s / of the operand x_n; S: place in X_{t+1}
  int64_t c;         // S: place of the forward coarse values
  int32_t l0, nl;    // S: adjacent separators' pieces, list[l0 .. l0 + nl) (places in u)
};
static_assert(sizeof(LevelOp<float>) == 80 && sizeof(LevelOp<double>) == 80, "descriptor copies");

struct LevelItem {
  int32_t op, loc;
};

template <typename TF>
struct LevelPhase {
  const LevelOp<TF>* ops;
  const int64_t* list;
  const LevelItem* items;
  const int32_t* base;   // first item of every operation
  int32_t kind, nitems, nops;
  int32_t first;         // 1: X_t is the vector the apply works on
  int32_t mode, pad;     // LevelMode
};

// The vectors of an apply, in the factor's precision: everything an FP32
// factor's products read is rounded to FP32 on the way in and everything they
// write is an FP32 sum, so FP32 work vectors hold the same values as FP64 ones
// would, and the FP64 unit (1/64 of the FP32 rate) stays out of the way: with
// FP64 work vectors its conversions and additions alone bounded the leaf phases
// (1.13 ms per application against 0.59 at 64^3, the items cut the same way).  Where an FP64 value
// enters, r itself and the sums x_p - sum u, it is carried as an unevaluated
// pair hi + lo of FP32 numbers (TwoSum, Knuth 1969).  The result is written in FP64.
template <typename TF>
struct LevelVecs {
  const TF *xh, *xl;   // X_1 on the way down: hi (all of it for an FP64 factor) and lo
  double* out;         // X_1 on the way back
  TF *xs, *xsl;        // X_t, t > 1, and its lo parts (nullptr: zero, every cluster is scaled)
  TF *y, *c, *z, *u;
};

// r -> hi + lo
__global__ void __launch_bounds__(256) k_split(int64_t n, const double* __restrict__ r, float* __restrict__ hi,
                                               float* __restrict__ lo) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = r[i];
    const float h = (float)v;
    hi[i] = h;
    lo[i] = (float)(v - (double)h);
  }
}

// s + e - u, e collecting the rounding errors of an FP32 s; plain in FP64.
__device__ __forceinline__ void la_less(float& s, float& e, float u) {
  const float t = s - u, b = t - s;
  e += (s - (t - b)) - (u + b);
  s = t;
}
__device__ __forceinline__ void la_less(double& s, double&, double u) { s -= u; }

constexpr int LA_NT = 256;  // threads per CTA (three CTAs per SM: 80 registers a thread)
constexpr int LA_NW = LA_NT / 32;

enum LevelMode : int32_t { LA_FEW = 0, LA_MID, LA_STREAM };

template <typename TF>
struct LaGeom {
  static constexpr int VW = 16 / (int)sizeof(TF);  // rows per 16-byte vector
  // How the items of a phase are cut (LevelPhase::mode):
  //  LA_FEW     few items for the launch's warps: as short as possible;
  //  LA_MID     in between;
  //  LA_STREAM  much factor data: as few bytes wasted and as little fixed cost
  //             as possible.
  // Row products: rows per item, one 16-byte vector, 8 or (FP32) 16: 8 loads in
  // flight then cover 256, 128 or 64 columns (FP64: 256, 64), and a load's
  // pieces of a column are 16, 32 or 64 bytes (a DRAM burst; FP64: 16, 64).
  __host__ __device__ static int rb(int mode) { return mode == LA_FEW ? VW : mode == LA_STREAM && VW == 4 ? 16 : 8; }
  // Column products.  Narrow: 8 lanes down the rows (8 VW rows per load), 4
  // columns per load; wide: 32 lanes down the rows, one column per load.  An
  // item is CG such column groups.  shape = CG (narrow) or -CG (wide) for R rows:
  // as many as 8 loads in flight cover (the taller ones take several rounds);
  // with LA_STREAM narrow items of 8 columns instead of wide ones: the rounds of
  // many warps overlap, and the items' fixed cost (operand loads, shuffles) is
  // spread over more bytes.  One apply at 48^3, 64^3, 96^3 FP32, 64^3, 30^3 FP64:
  // as here 0.279, 0.458, 0.946, 1.166, 0.265 ms; wide items with LA_STREAM too
  // 0.297, 0.510, 1.175, 1.466, 0.281; never wide (2 from 16 VW rows on) 0.309,
  // 0.494, 0.968, 1.238, 0.322.
  __host__ __device__ static int shape(int R, int mode) {
    return R <= 8 * VW ? 8 : R <= 16 * VW ? 4 : R <= 32 * VW || mode == LA_STREAM ? 2 : R <= 64 * VW ? -4 : R <= 128 * VW ? -2 : -1;
  }
  __host__ __device__ static int width(int R, int mode) {
    const int g = shape(R, mode);
    return g > 0 ? 4 * g : -g;
  }
};

// Items of an operation in a phase.
template <typename TF>
__host__ __device__ inline int la_items(int kind, int n, int m, bool hasA, bool hasY, int mode) {
  const int b = LaGeom<TF>::rb(mode), rn = (n + b - 1) / b, rm = (m + b - 1) / b;
  auto cols = [=](int c, int R) {
    const int w = LaGeom<TF>::width(R, mode);
    return (c + w - 1) / w;
  };
  switch (kind) {
    case LP_FE: return rn + rm;
    case LP_FY: return rn;
    case LP_BA: return rn;
    case LP_FU: return cols(m, n);
    case LP_BX: return cols(n, n);
    case LP_BE: return cols(n, n + m);
    case LP_FS: return !hasY ? (n + 31) >> 5 : rn + (hasA ? rm : 0);
    default: return !hasY ? (n + 31) >> 5 : cols(n, n + (hasA ? m : 0));
  }
}

// The item table of every phase: block y fills phase y's, one thread per operation.
template <typename TF>
__global__ void k_level_items(const LevelPhase<TF>* __restrict__ phases) {
  const LevelPhase<TF> P = phases[blockIdx.y];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.nops; i += gridDim.x * blockDim.x) {
    const LevelOp<TF>& o = P.ops[i];
    const int k = la_items<TF>(P.kind, o.n, o.m, o.A != nullptr, o.Y != nullptr, P.mode), b = P.base[i];
    for (int e = 0; e < k; ++e) const_cast<LevelItem*>(P.items)[b + e] = LevelItem{i, e};
  }
}

// G_ns = X_ns Y or P_p = Q_pc^T Y: O (m x n, leading dimension ldo) = A^T Y, A
// n x m, one 64 x 64 tile per CTA; Y is zero above its diagonal, so the sum
// starts at the tile's first column.
template <typename T>
struct CombineTask {
  const T* A;
  const T* Y;
  T* O;
  int32_t n, m, lda, ldy, ldo, pad;
};
struct CombineTile {
  int32_t task, i0, j0;
};
template <typename T>
__global__ void __launch_bounds__(NT) k_combine(const CombineTile* __restrict__ tiles,
                                                const CombineTask<T>* __restrict__ tasks) {
  __shared__ TileSmem<T> sm;
  const CombineTile t = tiles[blockIdx.x];
  const CombineTask<T> d = tasks[t.task];
  const int mi = min(TB, d.m - t.i0), nj = min(TB, d.n - t.j0), k0 = t.j0;
  T acc[4][4];
  zero_acc(acc);
  tn_acc(acc, d.A + k0 + (size_t)t.i0 * d.lda, d.lda, mi, d.Y + k0 + (size_t)t.j0 * d.ldy, d.ldy, nj, d.n - k0, sm);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int jj = 0; jj < 4; ++jj)
#pragma unroll
    for (int ii = 0; ii < 4; ++ii) {
      const int r = tx + 16 * ii, c = ty + 16 * jj;
      if (r < mi && c < nj) d.O[(size_t)(t.i0 + r) + (size_t)(t.j0 + c) * d.ldo] = acc[ii][jj];
    }
}

__device__ __forceinline__ float4 la_zero(float4*) { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ double2 la_zero(double2*) { return make_double2(0.0, 0.0); }

template <typename TF>
using LaVec = typename std::conditional<sizeof(TF) == 4, float4, double2>::type;

// Matrix of a row item and its place.
template <typename TF>
struct LaRow {
  const TF* A;
  int ld, row, K;  // first row of the item, columns (a multiple of RB below)
  bool y;          // rows of Y (else of G / P)
};
template <typename TF>
__device__ __forceinline__ LaRow<TF> la_row_of(int kind, const LevelOp<TF>& o, int loc, int b) {
  LaRow<TF> r;
  const int rn = (o.n + b - 1) / b;
  if (kind == LP_BA) {
    r.A = o.A, r.ld = o.lda, r.row = b * loc, r.K = o.m, r.y = false;
  } else if (loc < rn) {
    r.A = o.Y, r.ld = o.ldy, r.row = b * loc, r.K = min(o.n, b * loc + b), r.y = true;
  } else {
    r.A = o.A, r.ld = o.lda, r.row = b * (loc - rn), r.K = o.n, r.y = false;
  }
  return r;
}

// Eight loads of a row product: columns k0 + cl + CL u (u < 8) of the lane's rows.
template <typename TF, int RB>
__device__ __forceinline__ void la_row_load(LaVec<TF> (&a)[8], const LaRow<TF>& r, int k0) {
  typedef LaVec<TF> V;
  constexpr int VW = LaGeom<TF>::VW, RL = RB / VW, CL = 32 / RL;
  const int lane = threadIdx.x & 31, row = r.row + VW * (lane % RL), k1 = k0 + lane / RL;
  const TF* p = r.A + row + (size_t)k1 * r.ld;
#pragma unroll
  for (int u = 0; u < 8; ++u)
    a[u] = (k1 + CL * u < r.K && row < r.ld) ? __ldg(reinterpret_cast<const V*>(p + (size_t)(CL * u) * r.ld))
                                             : la_zero((V*)0);
}

template <typename TF, int RB>
__device__ __forceinline__ void la_row_run(LaVec<TF> (&a)[8], int kind, const LevelOp<TF>& o, int loc,
                                           const LevelPhase<TF>& P, const LevelVecs<TF>& V) {
  typedef LaVec<TF> VT;
  constexpr int VW = LaGeom<TF>::VW, RL = RB / VW, CL = 32 / RL;
  const LaRow<TF> r = la_row_of(kind, o, loc, RB);
  const int lane = threadIdx.x & 31, cl = lane / RL;
  const TF* x = kind == LP_BA ? V.u + o.u : (P.first ? V.xh : V.xs) + o.x;
  const TF* xl = (P.first ? V.xl : V.xsl);
  const int nl = kind == LP_FS ? o.nl : 0;
  TF s[VW];
#pragma unroll
  for (int w = 0; w < VW; ++w) s[w] = TF(0);
  for (int k0 = 0; k0 < r.K; k0 += 8 * CL) {
    if (k0) la_row_load<TF, RB>(a, r, k0);
    TF v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = k0 + cl + CL * u;
      v[u] = k < r.K ? x[k] : TF(0);
    }
    if (nl) {  // less the separators' pieces, summed in order
      TF e[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = k0 + cl + CL * u;
        e[u] = xl && k < r.K ? xl[o.x + k] : TF(0);
      }
      for (int l = 0; l < nl; ++l) {
        const TF* piece = V.u + P.list[o.l0 + l];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int k = k0 + cl + CL * u;
          if (k < r.K) la_less(v[u], e[u], piece[k]);
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] += e[u];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const VT f = a[u];
      s[0] = fma(f.x, v[u], s[0]);
      s[1] = fma(f.y, v[u], s[1]);
      if constexpr (VW == 4) {
        s[2] = fma(f.z, v[u], s[2]);
        s[3] = fma(f.w, v[u], s[3]);
      }
    }
  }
#pragma unroll
  for (int off = RL; off < 32; off <<= 1)
#pragma unroll
    for (int w = 0; w < VW; ++w) s[w] += __shfl_xor_sync(0xffffffffu, s[w], off);
  TF mine = s[0];  // column lane w stores row w of its vector
#pragma unroll
  for (int w = 1; w < VW; ++w)
    if (cl == w) mine = s[w];
  const int i = r.row + VW * (lane % RL) + cl;
  if (cl < VW) {
    if (kind == LP_BA) {
      if (i < o.n) V.z[o.z + i] = V.y[o.y + i] - mine;
    } else if (r.y) {
      if (i < o.n) {
        V.y[o.y + i] = mine;
        if (kind == LP_FS && !o.A) {
          V.xs[o.u + i] = mine;
          if (V.xsl) V.xsl[o.u + i] = TF(0);
        }
      }
    } else if (i < o.m) {
      if (kind == LP_FE) {
        V.u[o.u + i] = mine;
      } else {
        V.xs[o.u + i] = mine;
        if (V.xsl) V.xsl[o.u + i] = TF(0);
        V.c[o.c + i] = mine;
      }
    }
  }
}

// A column item: its steps of RS rows run down Y (from the multiple of RS at or
// above its first column: Y is zero above its diagonal), then down G or P.
template <typename TF>
struct LaCol {
  const TF *A0, *A1;
  int ld0, ld1, n0, n1, lo, ncol, c0;
};
template <typename TF, int RS>
__device__ __forceinline__ LaCol<TF> la_col_of(int kind, const LevelOp<TF>& o, int loc, int width) {
  LaCol<TF> c;
  c.c0 = loc * width;
  if (kind == LP_FU) {
    c.A0 = o.A, c.ld0 = o.lda, c.n0 = o.n, c.lo = 0, c.ncol = o.m;
  } else {
    c.A0 = o.Y, c.ld0 = o.ldy, c.n0 = o.n, c.lo = c.c0 / RS * RS, c.ncol = o.n;
  }
  const bool two = (kind == LP_BS && o.A) || kind == LP_BE;
  c.A1 = o.A, c.ld1 = o.lda, c.n1 = two ? o.m : 0;
  return c;
}

// Rows of the item's column products: all of Y's, and of G's or P's.
template <typename TF>
__device__ __forceinline__ int la_rows(int kind, const LevelOp<TF>& o) {
  return o.n + ((kind == LP_BS && o.A) || kind == LP_BE ? o.m : 0);
}

// Loads of ST = 8 / CG row steps from step s0, columns c0 + 4 g + cl (WIDE: c0 + g), g < CG.
template <typename TF, int CG, bool WIDE>
__device__ __forceinline__ void la_col_load(LaVec<TF> (&a)[8], const LaCol<TF>& c, int s0) {
  typedef LaVec<TF> V;
  constexpr int VW = LaGeom<TF>::VW, RS = WIDE ? 32 * VW : 8 * VW;
  const int lane = threadIdx.x & 31, rl = WIDE ? lane : lane & 7, cl = WIDE ? 0 : lane >> 3;
  const int S0 = (c.n0 - c.lo + RS - 1) / RS;
#pragma unroll
  for (int s = 0; s < 8 / CG; ++s) {
    const bool seg = s0 + s >= S0;
    const int i = (seg ? (s0 + s - S0) * RS : c.lo + (s0 + s) * RS) + VW * rl;
    const TF* A = seg ? c.A1 : c.A0;
    const int ld = seg ? c.ld1 : c.ld0, n = seg ? c.n1 : c.n0;
#pragma unroll
    for (int g = 0; g < CG; ++g) {
      const int col = c.c0 + (WIDE ? 1 : 4) * g + cl;
      a[s * CG + g] = (i < n && col < c.ncol) ? __ldg(reinterpret_cast<const V*>(A + i + (size_t)col * ld)) : la_zero((V*)0);
    }
  }
}

// One 16-byte vector of a work vector (its places are multiples of 4 elements).
__device__ __forceinline__ void la_vec(float (&v)[4], const float* p) {
  const float4 f = *reinterpret_cast<const float4*>(p);
  v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
}
__device__ __forceinline__ void la_vec(double (&v)[2], const double* p) {
  const double2 f = *reinterpret_cast<const double2*>(p);
  v[0] = f.x, v[1] = f.y;
}

template <typename TF, int CG, bool WIDE>
__device__ __forceinline__ void la_col_run(LaVec<TF> (&a)[8], int kind, const LevelOp<TF>& o, int loc,
                                           const LevelPhase<TF>& P, const LevelVecs<TF>& V) {
  typedef LaVec<TF> VT;
  constexpr int VW = LaGeom<TF>::VW, RS = WIDE ? 32 * VW : 8 * VW, ST = 8 / CG;
  const LaCol<TF> c = la_col_of<TF, RS>(kind, o, loc, WIDE ? CG : 4 * CG);
  const int lane = threadIdx.x & 31, rl = WIDE ? lane : lane & 7, cl = WIDE ? 0 : lane >> 3;
  const int S0 = (c.n0 - c.lo + RS - 1) / RS, S = S0 + (c.n1 + RS - 1) / RS;
  const bool next = kind == LP_BS && !o.A;  // not sparsified: y_p's place is taken by X_{t+1}
  const TF* src0 = kind == LP_BX ? V.z + o.z : V.y + o.y;
  TF acc[CG];
#pragma unroll
  for (int g = 0; g < CG; ++g) acc[g] = TF(0);
  for (int s0 = 0; s0 < S; s0 += ST) {
    if (s0) la_col_load<TF, CG, WIDE>(a, c, s0);
#pragma unroll
    for (int s = 0; s < ST; ++s) {
      const bool seg = s0 + s >= S0;
      const int i = (seg ? (s0 + s - S0) * RS : c.lo + (s0 + s) * RS) + VW * rl;
      const int n = s0 + s >= S ? 0 : seg ? c.n1 : c.n0;
      TF v[VW];
#pragma unroll
      for (int w = 0; w < VW; ++w) v[w] = TF(0);
      if (i < n) {
        if (next || (seg && kind == LP_BS)) {  // X_{t+1} (any alignment)
#pragma unroll
          for (int w = 0; w < VW; ++w) v[w] = i + w < n ? V.xs[o.u + i + w] : TF(0);
          if (!next) {
            TF q[VW];
            la_vec(q, V.c + o.c + i);
#pragma unroll
            for (int w = 0; w < VW; ++w) v[w] -= q[w];
          }
        } else {
          la_vec(v, (seg ? V.u + o.u : src0) + i);
          if (seg) {
#pragma unroll
            for (int w = 0; w < VW; ++w) v[w] = -v[w];
          }
        }
#pragma unroll
        for (int w = 1; w < VW; ++w)
          if (i + w >= n) v[w] = TF(0);
      }
#pragma unroll
      for (int g = 0; g < CG; ++g) {
        VT f = a[s * CG + g];
        if (i + VW > n) {  // rows past the end are padding: never multiplied
          if (i + 1 >= n) f.y = TF(0);
          if constexpr (VW == 4) {
            if (i + 2 >= n) f.z = TF(0);
            if (i + 3 >= n) f.w = TF(0);
          }
        }
        acc[g] = fma(f.x, v[0], acc[g]);
        acc[g] = fma(f.y, v[1], acc[g]);
        if constexpr (VW == 4) {
          acc[g] = fma(f.z, v[2], acc[g]);
          acc[g] = fma(f.w, v[3], acc[g]);
        }
      }
    }
  }
#pragma unroll
  for (int g = 0; g < CG; ++g) {
#pragma unroll
    for (int off = 1; off < (WIDE ? 32 : 8); off <<= 1) acc[g] += __shfl_xor_sync(0xffffffffu, acc[g], off);
  }
  TF mine = acc[0];  // row lane g (of column lane cl) stores group g's column
#pragma unroll
  for (int g = 1; g < CG; ++g)
    if (rl == g) mine = acc[g];
  const int col = c.c0 + (WIDE ? 1 : 4) * rl + cl;
  if (rl < CG && col < c.ncol) {
    if (kind == LP_FU) {
      V.u[o.u + col] = mine;
    } else {
      if (P.first) V.out[o.x + col] = (double)mine;
      else V.xs[o.x + col] = mine;
      if (kind == LP_BS)
        for (int e = 0; e < o.nl; ++e) V.u[P.list[o.l0 + e] + col] = mine;
    }
  }
}

__device__ __forceinline__ bool la_is_row(int kind) {
  return kind == LP_FE || kind == LP_FY || kind == LP_FS || kind == LP_BA;
}

// First loads of an item.
template <typename TF>
__device__ __forceinline__ void la_fetch(LaVec<TF> (&a)[8], int kind, int mode, const LevelOp<TF>& o, int loc) {
  if (!o.Y) return;  // values pass through
  if (la_is_row(kind)) {
    constexpr int F = LaGeom<TF>::VW, S = F == 4 ? 16 : 8;
    if (mode == LA_FEW) la_row_load<TF, F>(a, la_row_of(kind, o, loc, F), 0);
    else if (mode == LA_MID) la_row_load<TF, 8>(a, la_row_of(kind, o, loc, 8), 0);
    else la_row_load<TF, S>(a, la_row_of(kind, o, loc, S), 0);
    return;
  }
  constexpr int N = 8 * LaGeom<TF>::VW, W = 32 * LaGeom<TF>::VW;
  switch (LaGeom<TF>::shape(la_rows(kind, o), mode)) {
    case 8: la_col_load<TF, 8, false>(a, la_col_of<TF, N>(kind, o, loc, 32), 0); break;
    case 4: la_col_load<TF, 4, false>(a, la_col_of<TF, N>(kind, o, loc, 16), 0); break;
    case 2: la_col_load<TF, 2, false>(a, la_col_of<TF, N>(kind, o, loc, 8), 0); break;
    case -4: la_col_load<TF, 4, true>(a, la_col_of<TF, W>(kind, o, loc, 4), 0); break;
    case -2: la_col_load<TF, 2, true>(a, la_col_of<TF, W>(kind, o, loc, 2), 0); break;
    default: la_col_load<TF, 1, true>(a, la_col_of<TF, W>(kind, o, loc, 1), 0);
  }
}

template <typename TF>
__device__ __forceinline__ void la_run(LaVec<TF> (&a)[8], int kind, const LevelOp<TF>& o, int loc,
                                       const LevelPhase<TF>& P, const LevelVecs<TF>& V) {
  const int mode = P.mode;
  if (!o.Y) {  // not scaled: 32 values pass through
    const int i = 32 * loc + (threadIdx.x & 31);
    if (i >= o.n) return;
    if (kind == LP_FS) {
      const TF* xl = P.first ? V.xl : V.xsl;
      TF s = (P.first ? V.xh : V.xs)[o.x + i], e = xl ? xl[o.x + i] : TF(0);
      for (int l = 0; l < o.nl; ++l) la_less(s, e, V.u[P.list[o.l0 + l] + i]);
      const TF h = s + e;
      V.xs[o.u + i] = h;
      if (V.xsl) V.xsl[o.u + i] = e - (h - s);
    } else {
      const TF d = V.xs[o.u + i];
      if (P.first) V.out[o.x + i] = (double)d;
      else V.xs[o.x + i] = d;
      for (int l = 0; l < o.nl; ++l) V.u[P.list[o.l0 + l] + i] = d;
    }
    return;
  }
  if (la_is_row(kind)) {
    constexpr int F = LaGeom<TF>::VW, S = F == 4 ? 16 : 8;
    if (mode == LA_FEW) la_row_run<TF, F>(a, kind, o, loc, P, V);
    else if (mode == LA_MID) la_row_run<TF, 8>(a, kind, o, loc, P, V);
    else la_row_run<TF, S>(a, kind, o, loc, P, V);
    return;
  }
  switch (LaGeom<TF>::shape(la_rows(kind, o), mode)) {
    case 8: la_col_run<TF, 8, false>(a, kind, o, loc, P, V); break;
    case 4: la_col_run<TF, 4, false>(a, kind, o, loc, P, V); break;
    case 2: la_col_run<TF, 2, false>(a, kind, o, loc, P, V); break;
    case -4: la_col_run<TF, 4, true>(a, kind, o, loc, P, V); break;
    case -2: la_col_run<TF, 2, true>(a, kind, o, loc, P, V); break;
    default: la_col_run<TF, 1, true>(a, kind, o, loc, P, V);
  }
}

// Dynamic shared memory for nph phases: the phases, and per warp and phase the
// item and the operation it starts with.
template <typename TF>
inline size_t la_smem(int nph) {
  return (size_t)std::max(nph, 1) * (sizeof(LevelPhase<TF>) + (size_t)LA_NW * (sizeof(LevelOp<TF>) + sizeof(LevelItem)));
}

// Phases [0, nph) of `phases`, a bounded grid barrier between them (bar, err,
// spin_limit, bias as in k_apply; cooperative launch).
template <typename TF>
__global__ void __launch_bounds__(LA_NT, 3)
    k_apply_levels(const LevelPhase<TF>* __restrict__ phases, int nph, LevelVecs<TF> V, unsigned* bar, int* err,
                   unsigned spin_limit, unsigned bias) {
  constexpr int OW = (int)(sizeof(LevelOp<TF>) / 8);  // lane l < OW carries word l of a descriptor
  extern __shared__ __align__(16) unsigned char dyn[];
  LevelPhase<TF>* ptab = reinterpret_cast<LevelPhase<TF>*>(dyn);
  LevelOp<TF>* op0 = reinterpret_cast<LevelOp<TF>*>(ptab + nph);             // [warp][phase]
  LevelItem* it0 = reinterpret_cast<LevelItem*>(op0 + (size_t)LA_NW * nph);  // [warp][phase]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // four consecutive items (neighbouring rows of one block) go to one CTA
  const int gw = ((warp >> 2) * (int)gridDim.x + (int)blockIdx.x) * 4 + (warp & 3), GW = LA_NW * (int)gridDim.x;
  for (int p = threadIdx.x; p < nph; p += LA_NT) ptab[p] = phases[p];
  __syncthreads();
  op0 += (size_t)warp * nph;
  it0 += (size_t)warp * nph;
  for (int p = lane; p < nph; p += 32) {
    LevelItem it{-1, 0};
    if (gw < ptab[p].nitems) {
      it = ptab[p].items[gw];
      op0[p] = ptab[p].ops[it.op];
    }
    it0[p] = it;
  }
  __syncwarp();
  for (int p = 0; p < nph; ++p) {
    const LevelPhase<TF>& P = ptab[p];
    const int kind = P.kind, nitems = P.nitems;
    const int mode = P.mode;
    LevelOp<TF>& o = op0[p];  // the warp's current operation
    int i = gw, loc = it0[p].loc;
    bool waited = p == 0;
    LevelItem nx{0, 0};  // the next item
    if (i + GW < nitems) nx = P.items[i + GW];
    for (;;) {
      LaVec<TF> a[8];
      unsigned long long w = 0;  // the next item's operation
      const int nloc = nx.loc;
      const bool more = i + GW < nitems;
      if (i < nitems) {
        la_fetch<TF>(a, kind, mode, o, loc);
        if (more) {
          if (lane < OW) w = __ldg(reinterpret_cast<const unsigned long long*>(P.ops + nx.op) + lane);
          if (i + 2 * GW < nitems) nx = P.items[i + 2 * GW];
        }
      }
      if (!waited) {
        if (!grid_wait(bar, (unsigned)p * gridDim.x + bias, err, spin_limit)) return;
        waited = true;
      }
      if (i >= nitems) break;
      la_run<TF>(a, kind, o, loc, P, V);
      __syncwarp();
      if (!more) break;
      if (lane < OW) reinterpret_cast<unsigned long long*>(&o)[lane] = w;
      __syncwarp();
      i += GW;
      loc = nloc;
    }
    __syncwarp();
    if (p + 1 < nph) grid_arrive(bar);
  }
}

}  // namespace spand
