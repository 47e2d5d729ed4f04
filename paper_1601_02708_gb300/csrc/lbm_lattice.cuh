// lbm_lattice.cuh -- D2Q9 lattice constants and the node-level pieces of the
// step: equilibrium, maximum-entropy boundary solves.  Device code only.
#pragma once
#include <cstdint>

namespace lbm {

// D2Q9: 0 rest, 1 E, 2 N, 3 W, 4 S, 5 NE, 6 NW, 7 SW, 8 SE (Sec. 4.1, the
// standard DnQm lattice with c_s^2 = 1/3).  constexpr functions so that the
// fully unrolled loops fold every lookup into an immediate.
__host__ __device__ constexpr int cx_of(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : (i == 3 || i == 6 || i == 7) ? -1 : 0;
}
__host__ __device__ constexpr int cy_of(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : (i == 4 || i == 7 || i == 8) ? -1 : 0;
}
__host__ __device__ constexpr int opp_of(int i) {
  return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4) + 1 : ((i - 3) % 4) + 5);
}
__host__ __device__ constexpr double w_of(int i) {
  return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
}

// Link word of a node (one uint32 per node).  Byte k of the low three bytes
// has bit i-1 set for direction i = 1..8 when the upstream neighbour x - e_i
//   byte 0: is solid while this step streams (pull -> halfway bounce-back),
//   byte 1: is solid after this step's dissolution flips (reaction, W_s),
//   byte 2: lies outside the lattice across a non-periodic side (unknown);
// bit 24 marks the node itself solid while streaming, bit 25 marks a solid
// node that turns fluid before this step collides (dissolution), bit 26 a
// solid node on the dissolution surface list.  The words
// change only when a node dissolves, so a step decodes its neighbourhood with
// bit tests on one word.
constexpr uint32_t kOwnSolid = 1u << 24;
constexpr uint32_t kOwnPending = 1u << 25;
constexpr uint32_t kListed = 1u << 26;  // solid node on the dissolution surface list
constexpr int kUpSolidShift = 0;
constexpr int kUpPostShift = 8;
constexpr int kUpOutShift = 16;
__host__ __device__ constexpr uint32_t up_bit(int shift, int i) { return 1u << (shift + i - 1); }
// A fluid node without a solid neighbour before or after this step's flips
// has a link word that is zero in these bits.
constexpr uint32_t kClearMask =
    kOwnSolid | kOwnPending | (0xFFu << kUpSolidShift) | (0xFFu << kUpPostShift);

// Index checks of the debug-bounds build (compiled with LBM_DEBUG_BOUNDS, in
// place of a memory checker): an index outside [0, limit) records its check
// site in *flag (the first one wins, the host reports it) and is replaced by
// 0, so the access stays inside the array.  The normal build compiles the
// check away.
#ifdef LBM_DEBUG_BOUNDS
__device__ __forceinline__ long long dbg_idx(long long i, long long limit, int* flag, int site) {
  if (i >= 0 && i < limit) return i;
  if (flag) atomicCAS(flag, 0, site);
  return 0;
}
#else
__device__ __forceinline__ long long dbg_idx(long long i, long long, int*, int) { return i; }
#endif
// Sites (values of the status word >= kSiteBase name the failed check).
enum {
  kSiteBase = 100,
  kSitePull = 101,     // global population read of the step
  kSiteNode = 102,     // per-node global field of the step (word, velocity, rate, u)
  kSiteStore = 103,    // global store of a node value or ghost image
  kSiteSmemPop = 111,  // shared-memory population read (tile pipeline)
  kSiteSmemNode = 112, // shared-memory per-node field (tile pipeline)
  kSiteShare = 121,    // reaction share read by the dissolution
  kSiteList = 122,     // surface-list or flip-list entry
  kSiteAdjGather = 131,  // adjoint state read by the reverse step
  kSiteAdjNode = 132,    // per-node field of the reverse step
};

// Padded layout of every node field: interior node (x, y) lives at column
// x + kXO and row y + kYO of a [rows][pitch] array, pitch a multiple of 32
// with pitch >= nx + 16, rows >= ny + 2.  Column kXO - 1, column nx + kXO,
// row 0 and row ny + 1 are ghost cells: across a periodic side the population
// and reaction fields hold there the image of the wrapped node (written
// through by the node itself).  Eight columns on the left put interior
// x = 0 on a 32-byte sector boundary (8 consecutive FP32 nodes per sector)
// and keep every tile's halo box 16-byte aligned for TMA; the minimum sizes
// (160 columns, 10 rows) let one halo box fit the array.
constexpr int kXO = 8;
constexpr int kYO = 1;

__host__ __device__ constexpr int padded_pitch(int nx) {
  return (nx + 16 + 31) / 32 * 32 < 160 ? 160 : (nx + 16 + 31) / 32 * 32;
}
__host__ __device__ constexpr int padded_rows(int ny) { return ny + 2 < 10 ? 10 : ny + 2; }

// Calls fn(gx, gy) for every ghost image of interior node (x, y) (padded
// coordinates), i.e. its copies across periodic sides within one cell of the
// lattice.
template <class Fn>
__device__ __forceinline__ void for_each_ghost(int x, int y, int nx, int ny, int per_x,
                                               int per_y, Fn&& fn) {
  const int xs[2] = {x, per_x ? (x == 0 ? nx : (x == nx - 1 ? -1 : x)) : x};
  const int ys[2] = {y, per_y ? (y == 0 ? ny : (y == ny - 1 ? -1 : y)) : y};
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      if (a == 0 && b == 0) continue;
      const int gx = xs[a], gy = ys[b];
      if ((a == 1 && gx == x) || (b == 1 && gy == y)) continue;
      fn(gx + kXO, gy + kYO);
    }
}

// Side kinds (lbm_edge_kind); kExchange: a side a slab shares with its
// neighbour in a split lattice (its ghost row is filled by the halo exchange).
enum { kPeriodic = 0, kDirichlet = 1, kNeumann = 2, kExchange = 3 };
enum { kReactNone = 0, kReactSurface = 1, kReactBulk = 2 };


// Index of edge node (x, y) of side s in the edge layout [W|E|S|N].
__device__ __forceinline__ int edge_slot(int s, int x, int y, int nx, int ny) {
  return s == 0 ? y : s == 1 ? ny + y : s == 2 ? 2 * ny + x : 2 * ny + nx + x;
}

// Maximum-entropy Dirichlet, Sec. 4.1.1 (a): the unknowns minimising
// H = sum f log(f/w) under sum f = up are proportional to w.  Computed in
// FP64.  Returns true if the data admit no non-negative solution.
template <typename Real>
__device__ __forceinline__ bool maxent_dirichlet_general(Real (&f)[9], unsigned unknown, double up) {
  double wu = 0.0, known = 0.0;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    if (unknown & (1u << i)) wu += w_of(i);
    else known += (double)f[i];
  }
  const double rest = up - known;
  const double scale = rest / wu;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    if (unknown & (1u << i)) f[i] = (Real)(w_of(i) * scale);
  return rest < 0.0;
}

// Maximum-entropy Neumann, Sec. 4.1.1 (b), for an outward normal (sx, sy)
// with sx, sy in {-1, 0, 1} (a side, or the corner of two Neumann sides).
// Unknowns with e.n = 0 (corner tangents) take halfway bounce-back of the
// node's own post-collision population fbb[opp(i)].  On a side every M^-
// unknown has e.n = -1 and the root gives f proportional to w; at a corner
// (n = (sx, sy)/sqrt 2) the unknowns have e.n = -1/sqrt 2 or -sqrt 2 and the
// root condition is a quadratic in t = exp(gamma / sqrt 2), solved in closed
// form.  Returns kNeuRoot when the root set the unknowns, else the unknowns
// are 0 (the gamma -> -inf limit) and the return is kNeuInfeasible if the
// data admit no root (R > 0) or kNeuZero if R = 0.
enum { kNeuRoot = 0, kNeuInfeasible = 1, kNeuZero = 2 };
template <typename Real>
__device__ __forceinline__ int maxent_neumann_general(Real (&f)[9], unsigned unknown, int sx, int sy,
                              double q, const Real (&fbb)[9]) {
  const bool corner = (sx != 0) && (sy != 0);
  const double inv_len = corner ? 0.70710678118654752440 : 1.0;
  double R = q;
  double w1 = 0.0, w2 = 0.0;  // weights of M^- with |e.n| = 1/sqrt2 (or 1), sqrt2
  unsigned m1 = 0, m2 = 0;
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const int d = cx_of(i) * sx + cy_of(i) * sy;
    if (unknown & (1u << i)) {
      if (d == 0) {
        f[i] = fbb[opp_of(i)];
      } else if (d == -1) {
        m1 |= 1u << i;
        w1 += w_of(i);
      } else {  // d == -2 (corner diagonal)
        m2 |= 1u << i;
        w2 += w_of(i);
      }
    } else {
      R -= (double)d * inv_len * (double)f[i];
    }
  }
  const double S = -R;
  if (!(S > 0.0)) {
#pragma unroll
    for (int i = 1; i < 9; ++i)
      if ((m1 | m2) & (1u << i)) f[i] = (Real)0;
    return S < 0.0 ? kNeuInfeasible : kNeuZero;
  }
  if (!corner) {
    const double scale = S / w1;
#pragma unroll
    for (int i = 1; i < 9; ++i)
      if (m1 & (1u << i)) f[i] = (Real)(w_of(i) * scale);
    return kNeuRoot;
  }
  // (w1 / (sqrt2 e)) t + (sqrt2 w2 / e) t^2 = S
  const double inv_e = 0.36787944117144233;  // exp(-1)
  const double A = w1 * 0.70710678118654752440 * inv_e;
  const double B = w2 * 1.41421356237309504880 * inv_e;
  const double t = 2.0 * S / (A + sqrt(A * A + 4.0 * B * S));
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    if (m1 & (1u << i)) f[i] = (Real)(w_of(i) * t * inv_e);
    if (m2 & (1u << i)) f[i] = (Real)(w_of(i) * t * t * inv_e);
  }
  return kNeuRoot;
}

// The edge solves as the steps run them.  On a side, and at a corner that holds
// Dirichlet data, the unknowns are rest w_i / W_U with W_U = 6/36 (one axis and
// two diagonal directions) or 11/36 (a corner), so a product with 1/6 or 1/11
// stands for the division and the sum of the weights.  What bounds the solve
// is the latency of its chain (an FP64 operation returns after about 200 cycles
// on this part and the general form has some thirty in a row), and with it the
// step of a small lattice, whose boundary nodes are one round of one warp.
// FP32 lattice: the sums and the product run in double-float (sums exact to
// 2^-48 of the largest term) on the FP32 pipe.  What this does not hold goes to
// the FP64 form: values outside 1e-24 .. 1e30 (the low parts leave FP32's range)
// and differences a thousand times smaller than their terms.
// FP64 lattice: the same in FP64, the sum as a tree, seven operations in a row.
// The general form keeps other unknown sets and Neumann corners.
// Ten substeps of a 256 x 64 channel with restore and trace: 145 -> 139 us; one
// gradient over 500 steps at 512 x 512, whose reverse steps transpose the same
// solves: 10.2 -> 8.3 ms; a coarse step of the plain hybrid in FP64: 724 -> 700.
// A substep at 512 x 512: general form alone 6.1 us, FP64 form 5.85, double-float
// 5.6, and 6.15 with a boundary node or two beyond its range (6.9 when those took
// the general form).
constexpr float kEdgeLow = 1e-24f, kEdgeHigh = 1e30f, kEdgeCancel = 1e-3f;

struct EdgeSum {  // hi + lo, not normalised
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float a) {
    const float t = __fadd_rn(hi, a), b = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, b)), __fsub_rn(a, b)));
    hi = t;
  }
  __device__ __forceinline__ void norm() {
    const float t = __fadd_rn(hi, lo);
    lo = __fsub_rn(lo, __fsub_rn(t, hi));
    hi = t;
  }
};
__device__ __forceinline__ EdgeSum edge_split(double v) {
  EdgeSum r;
  r.hi = (float)v;
  r.lo = (float)(v - (double)r.hi);
  return r;
}
// (hi + lo) / c as a pair (normalised), c 6 or 11: the quotient of the
// high part, then that of the remainder
__device__ __forceinline__ EdgeSum edge_over(const EdgeSum& a, int c) {
  const float inv = c == 6 ? 1.f / 6 : 1.f / 11, fc = (float)c;
  EdgeSum r;
  r.hi = __fmul_rn(a.hi, inv);
  r.lo = __fmul_rn(__fadd_rn(__fmaf_rn(-fc, r.hi, a.hi), a.lo), inv);
  r.norm();
  return r;
}
// 36 times the weight of a set of directions
__device__ __forceinline__ int set_weight36(unsigned m) {
  return 4 * __popc(m & 0x1Eu) + __popc(m & 0x1E0u);
}

// The FP64 form, the sums as trees: weight 36 W_U = c is 6 or 11; on a side, whose
// unknowns all have e.n = -1.
template <typename Real>
__device__ __forceinline__ bool dirichlet_tree(Real (&f)[9], unsigned unknown, double up, int c) {
  double k[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) k[i] = unknown & (1u << i) ? 0.0 : (double)f[i];
  const double known = (((k[0] + k[1]) + (k[2] + k[3])) + ((k[4] + k[5]) + (k[6] + k[7]))) + k[8];
  const double rest = up - known;
  const double g = rest * (c == 6 ? 1.0 / 6 : 1.0 / 11), g4 = 4.0 * g;
#pragma unroll
  for (int i = 1; i < 9; ++i)
    if (unknown & (1u << i)) f[i] = (Real)(i < 5 ? g4 : g);
  return rest < 0.0;
}
template <typename Real>
__device__ __forceinline__ int neumann_tree(Real (&f)[9], unsigned unknown, int sx, int sy, double q) {
  double k[9];
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const int d = cx_of(i) * sx + cy_of(i) * sy;
    k[i] = unknown & (1u << i) ? 0.0 : d > 0 ? (double)f[i] : d < 0 ? -(double)f[i] : 0.0;
  }
  const double out = ((k[1] + k[2]) + (k[3] + k[4])) + ((k[5] + k[6]) + (k[7] + k[8]));
  const double S = out - q;
  const bool root = S > 0.0;
  const double g = S * (1.0 / 6), g4 = 4.0 * g;
#pragma unroll
  for (int i = 1; i < 9; ++i)
    if (unknown & (1u << i)) f[i] = root ? (Real)(i < 5 ? g4 : g) : (Real)0;
  return root ? kNeuRoot : S < 0.0 ? kNeuInfeasible : kNeuZero;
}

__device__ __forceinline__ bool maxent_dirichlet(float (&f)[9], unsigned unknown, double up) {
  EdgeSum rest = edge_split(up), known;
  float most = fabsf(rest.hi);
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const float v = unknown & (1u << i) ? 0.f : f[i];
    most = fmaxf(most, fabsf(v));
    known.add(v);
  }
  rest.lo = __fsub_rn(rest.lo, known.lo);
  rest.add(-known.hi);
  rest.norm();
  const float size = fabsf(rest.hi);
  const int c = set_weight36(unknown);
  if ((c == 6 || c == 11) && size > kEdgeLow && size > kEdgeCancel * most && most < kEdgeHigh) {
    const EdgeSum g = edge_over(rest, c);
#pragma unroll
    for (int i = 1; i < 9; ++i)
      if (unknown & (1u << i)) f[i] = i < 5 ? 4.f * g.hi : g.hi;
    return rest.hi < 0.f;
  }
  if (most == 0.f && size == 0.f && up == 0.0) {  // no data and nothing there (nor NaN)
#pragma unroll
    for (int i = 1; i < 9; ++i)
      if (unknown & (1u << i)) f[i] = 0.f;
    return false;
  }
  return c == 6 || c == 11 ? dirichlet_tree(f, unknown, up, c) : maxent_dirichlet_general(f, unknown, up);
}

__device__ __forceinline__ bool maxent_dirichlet(double (&f)[9], unsigned unknown, double up) {
  const int c = set_weight36(unknown);
  return c == 6 || c == 11 ? dirichlet_tree(f, unknown, up, c) : maxent_dirichlet_general(f, unknown, up);
}

__device__ __forceinline__ int maxent_neumann(float (&f)[9], unsigned unknown, int sx, int sy,
                                              double q, const float (&fbb)[9]) {
  if ((sx == 0 || sy == 0) && set_weight36(unknown) == 6) {
    // every unknown has e.n = -1
    EdgeSum S = edge_split(q), out;
    S.hi = -S.hi;
    S.lo = -S.lo;
    float most = fabsf(S.hi);
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      const float d = (float)(cx_of(i) * sx + cy_of(i) * sy);
      const float v = unknown & (1u << i) ? 0.f : d * f[i];
      most = fmaxf(most, fabsf(v));
      out.add(v);
    }
    S.lo = __fadd_rn(S.lo, out.lo);
    S.add(out.hi);
    S.norm();
    const float size = fabsf(S.hi);
    if (size > kEdgeLow && size > kEdgeCancel * most && most < kEdgeHigh) {
      const bool root = S.hi > 0.f;
      const EdgeSum g = edge_over(S, 6);
#pragma unroll
      for (int i = 1; i < 9; ++i)
        if (unknown & (1u << i)) f[i] = root ? (i < 5 ? 4.f * g.hi : g.hi) : 0.f;
      return root ? kNeuRoot : kNeuInfeasible;
    }
    if (most == 0.f && size == 0.f && q == 0.0) {
#pragma unroll
      for (int i = 1; i < 9; ++i)
        if (unknown & (1u << i)) f[i] = 0.f;
      return kNeuZero;
    }
    return neumann_tree(f, unknown, sx, sy, q);
  }
  return maxent_neumann_general(f, unknown, sx, sy, q, fbb);
}

__device__ __forceinline__ int maxent_neumann(double (&f)[9], unsigned unknown, int sx, int sy,
                                              double q, const double (&fbb)[9]) {
  if ((sx != 0 && sy != 0) || set_weight36(unknown) != 6)
    return maxent_neumann_general(f, unknown, sx, sy, q, fbb);
  return neumann_tree(f, unknown, sx, sy, q);
}

// Boundary kind of an edge node (x, y) whose unknown set is not empty:
// Dirichlet wins at corners (*dside >= 0, the first Dirichlet side), else
// Neumann (*nside, the first Neumann side, with the outward normal (sx, sy)
// summed over the node's Neumann sides).
__device__ __forceinline__ void edge_kind(const int (&edge)[4], int x, int y, int nx, int ny,
                                          int* dside, int* nside, int* sx, int* sy) {
  auto bc = [&](int s) { return edge[s] == kDirichlet || edge[s] == kNeumann; };
  const bool on[4] = {x == 0 && bc(0), x == nx - 1 && bc(1), y == 0 && bc(2),
                      y == ny - 1 && bc(3)};
  *dside = -1;
  *nside = -1;
  *sx = 0;
  *sy = 0;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (!on[s]) continue;
    if (edge[s] == kDirichlet && *dside < 0) *dside = s;
    if (edge[s] == kNeumann) {
      if (*nside < 0) *nside = s;
      *sx += (s == 0) ? -1 : (s == 1) ? 1 : 0;
      *sy += (s == 2) ? -1 : (s == 3) ? 1 : 0;
    }
  }
}

// Pore wall of the maximum-entropy kind: Sec. 4.1.1 (b) with zero flux, the
// option beside halfway bounce-back.  `solid` has bit i set where the source
// x - e_i of pull i is solid; on entry f holds the halfway bounce-back value
// in those directions.  The outward normal is the lattice-weighted direction
// to the solid neighbours, n = -sum_{i in solid} w_i e_i, normalised (where it
// cancels, as in a one-node channel, bounce-back stays throughout; which
// unknowns are tangent to it is decided on 36 n, an integer vector).  Unknowns
// with e_i.n >= 0 keep bounce-back; the others become
// w_i exp(-1 - gamma e_i.n) with gamma making sum_i f_i e_i.n zero.  With
// a_i = e_i.n < 0 the flux of those unknowns is -L(gamma),
// L(gamma) = sum |a_i| w_i exp(-1 + gamma |a_i|), so the root solves
// log L(gamma) = log(-R), R = -sum_{others} a_j f_j; log L is convex and
// increasing with slope between the smallest and largest |a_i|, so Newton's
// method converges from any start (in one step when every |a_i| is equal, as
// on a flat wall).
// S is the precision of the solve (the Lagrange multiplier, the normal, the
// fluxes and the exponentials); the lattice's populations f are read and
// written in their own precision Real.  Returns kWallSet, kWallNoRoot if
// R > 0 (no root: those unknowns are set to zero, the gamma -> -infinity
// limit) or kWallNoConv if Newton's method stopped short of its tolerance
// (the last iterate is used).
enum { kWallSet = 0, kWallNoRoot = 1, kWallNoConv = 2 };
template <typename S, typename Real>
__device__ int maxent_wall_general(Real (&f)[9], unsigned solid) {
  // the normal scaled by 36 (the weights are 4/36 and 1/36): integers, so
  // which unknowns are tangent to it, and whether it cancels, is exact
  int mx = 0, my = 0;
#pragma unroll
  for (int i = 1; i < 9; ++i)
    if (solid & (1u << i)) {
      const int w36 = (cx_of(i) != 0 && cy_of(i) != 0) ? 1 : 4;
      mx -= w36 * cx_of(i);
      my -= w36 * cy_of(i);
    }
  if (mx == 0 && my == 0) return kWallSet;
  // FP32 populations in an FP64 solve: integer multiples of them, summed before
  // the normal is scaled, so that a flux that cancels keeps its sign
  constexpr bool kExact = sizeof(S) == 8 && sizeof(Real) == 4;
  const S inv = (S)1 / sqrt((S)(mx * mx + my * my));
  const S nx = (S)mx * inv, ny = (S)my * inv;
  S a[9], R = (S)0, s1 = (S)0, s2 = (S)0;
  unsigned neg = 0u;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    a[i] = (S)cx_of(i) * nx + (S)cy_of(i) * ny;
    if (((solid >> i) & 1u) && cx_of(i) * mx + cy_of(i) * my < 0) {
      neg |= 1u << i;
      s1 -= (S)w_of(i) * a[i];
      s2 += (S)w_of(i) * a[i] * a[i];
    } else if (kExact) {
      R -= (S)(cx_of(i) * mx + cy_of(i) * my) * (S)f[i];
    } else {
      R -= a[i] * (S)f[i];
    }
  }
  if (kExact) R *= inv;
  if (!neg) return kWallSet;
  if (!(R < (S)0)) {
#pragma unroll
    for (int i = 0; i < 9; ++i)
      if (neg & (1u << i)) f[i] = (Real)0;
    return R > (S)0 ? kWallNoRoot : kWallSet;
  }
  if (sizeof(S) == 4 && -R < (S)1e-30) {
    // far below FP32's normal range the exponentials would underflow: the
    // flux-conserving split w_i (-R) / sum w |a| meets the constraint exactly
    // and differs from the maximum-entropy values by less than 1e-30
#pragma unroll
    for (int i = 0; i < 9; ++i)
      if (neg & (1u << i)) f[i] = (Real)((S)w_of(i) * (-R / s1));
    return kWallSet;
  }
  // tolerance on the relative Newton step: a few units of the solve's
  // rounding (FP64 2.2e-16, FP32 1.2e-7)
  constexpr int kIters = sizeof(S) == 8 ? 60 : 24;
  const S tol = sizeof(S) == 8 ? (S)1e-15 : (S)5e-7;
  // An FP64 solve for FP32 populations stops at the first step below 2e-6
  // in g.  phi(g) = log L(g) is convex, with phi' a weighted mean of the
  // unknowns' |a_i| and phi'' their weighted variance (<= 1/2); |a_i| lies
  // in [1 / sqrt(72), sqrt(2)] (an integer c_i . m over |m| <= sqrt(72)).
  // By convexity the error before a Newton step is at most 12 times the
  // step (at most the step itself from below the root), and after it at
  // most |phi''| / (2 phi') < 2.2 times the square of the error before: a
  // step under 2e-6 leaves g within 1.3e-9 and f within 1.8e-9 relative of
  // the root, 30 times below the FP32 rounding the populations then take.
  constexpr bool kLoose = sizeof(S) == 8 && sizeof(Real) == 4;
  const S logR = log(-R);
  // start: the root if every |a_i| were their weighted mean s2 / s1 (in
  // FP32 where FP32 iterations take it from there)
  S g = (S)0;
  bool started = false;
  if constexpr (sizeof(S) == 8) {
    // FP32 iterations (64 times the FP64 rate on this part) bring g to FP32
    // rounding of the root; the FP64 iterations below then need two or three
    // steps to the FP64 tolerance instead of a full solve.  Outside FP32's
    // range, or without FP32 convergence, the FP64 solve starts as above.
    if (-R > 1e-30 && -R < 1e30) {
      float af[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) af[i] = (float)a[i];
      const float logRf = logf((float)-R);
      float gf = (logRf - logf((float)s1) + 1.f) * ((float)s1 / (float)s2);
      bool okf = false;
      for (int it = 0; it < 24; ++it) {
        float L = 0.f, dL = 0.f;
#pragma unroll
        for (int i = 0; i < 9; ++i)
          if (neg & (1u << i)) {
            const float e = (float)w_of(i) * expf(gf * -af[i] - 1.f);
            L -= af[i] * e;
            dL += af[i] * af[i] * e;
          }
        if (!(dL > 0.f) || !(L > 0.f)) break;
        const float step = (logf(L) - logRf) * (L / dL);
        gf -= step;
        if (fabsf(step) <= 5e-7f * (1.f + fabsf(gf))) {
          okf = true;
          break;
        }
      }
      // (for FP32 populations any finite FP32 iterate is a start: Newton's
      // method converges from any start, and the loop below stops on its
      // own step)
      if ((okf || kLoose) && isfinite(gf)) {
        g = (S)gf;
        started = true;
      }
    }
  }
  if (!started) g = (logR - log(s1) + (S)1) * (s1 / s2);
  bool conv = false;
  S last = (S)0;
  for (int it = 0; it < kIters; ++it) {
    S L = (S)0, dL = (S)0;
#pragma unroll
    for (int i = 0; i < 9; ++i)
      if (neg & (1u << i)) {
        const S e = (S)w_of(i) * exp(g * -a[i] - (S)1);
        L -= a[i] * e;
        dL += a[i] * a[i] * e;
      }
    if (!(dL > (S)0)) break;
    const S step = (log(L) - logR) * (L / dL);
    g -= step;
    last = step;
    if (kLoose ? fabs(step) <= (S)2e-6 : fabs(step) <= tol * ((S)1 + fabs(g))) {
      conv = true;
      break;
    }
  }
  // an iteration that ended oscillating at its rounding level has converged
  if (!conv && fabs(last) <= (S)16 * tol * ((S)1 + fabs(g))) conv = true;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    if (neg & (1u << i)) f[i] = (Real)((S)w_of(i) * exp(g * -a[i] - (S)1));
  return conv ? kWallSet : kWallNoConv;
}

// Double-float arithmetic: an unevaluated pair hi + lo carrying about 48
// significant bits on the FP32 pipe (Dekker's products by a fused
// multiply-add, Knuth's two-sum).  The operations are named one by one: a
// product that the compiler merged into a neighbouring sum would have its
// rounding error, which the low part holds already, counted twice.
struct Df {
  float hi, lo;
};
__device__ __forceinline__ Df df_norm(float p, float e) {  // |e| <= |p|
  const float s = __fadd_rn(p, e);
  return Df{s, __fsub_rn(e, __fsub_rn(s, p))};
}
__device__ __forceinline__ Df df_mul(Df a, Df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  return df_norm(p, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.hi, -p))));
}
__device__ __forceinline__ Df df_mul(Df a, float b) {
  const float p = __fmul_rn(a.hi, b);
  return df_norm(p, __fmaf_rn(a.lo, b, __fmaf_rn(a.hi, b, -p)));
}
__device__ __forceinline__ Df df_add(Df a, Df b) {
  const float s = __fadd_rn(a.hi, b.hi), bb = __fsub_rn(s, a.hi);
  return df_norm(s, __fadd_rn(__fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb)),
                              __fadd_rn(a.lo, b.lo)));
}
__host__ __device__ constexpr Df df_const(double v) { return Df{(float)v, (float)(v - (double)(float)v)}; }

// The pore wall's equation as a polynomial.  With the normal scaled by 36 to
// the integer vector m = (mx, my), every unknown's e_i.n is -d_i / |m| with an
// integer d_i > 0, so with t = exp(gamma / |m|) the unknowns are
// (w_i / e) t^d_i and zero flux asks for
//     p(t) = sum 36 w_i d_i t^d_i = 36 e T,   T = sum_{others} (e_j.m) f_j,
// whose coefficients are integers.  d_i takes four values only: A = |mx| and
// B = |my| on the axes, A + B and |A - B| on the diagonals (each with at most
// one unknown, or two diagonals at A when B = 0), all formed from t^min(A, B)
// and t^|A - B|: no exponential and no logarithm but in the FP32 start.
struct WallPoly {
  int A, B;            // |mx|, |my| (at most 6)
  float ka, kb, ks, kd;  // coefficients of t^A, t^B, t^(A+B), t^|A-B|
};

// Start of the root in FP32: Newton's method on the convex log p as a function
// of x = log t (it converges from any start; one step when every exponent is
// equal, as on a flat wall).  Returns t, or 0 if it did not converge.
__device__ __forceinline__ float wall_start(const WallPoly& w, float C) {
  const float a = (float)w.A, b = (float)w.B, s = a + b, d = fabsf(a - b);
  const int mn = min(w.A, w.B), df = abs(w.A - w.B);
  const float logC = logf(C);
  const float k0 = (w.ka + w.kb) + (w.ks + w.kd);
  float x = (logC - logf(k0)) * (k0 / (w.ka * a + w.kb * b + w.ks * s + w.kd * d));
  for (int it = 0; it < 24; ++it) {
    const float t = expf(x), t2 = t * t, t4 = t2 * t2;
    const float q = ((mn & 1) ? t : 1.f) * ((mn & 2) ? t2 : 1.f) * ((mn & 4) ? t4 : 1.f);
    const float r = ((df & 1) ? t : 1.f) * ((df & 2) ? t2 : 1.f) * ((df & 4) ? t4 : 1.f);
    const float big = q * r;  // t^max(A, B)
    // (a term without an unknown may overflow: it must not turn 0 into NaN)
    const float pa = w.ka > 0.f ? w.ka * (w.A >= w.B ? big : q) : 0.f;
    const float pb = w.kb > 0.f ? w.kb * (w.A >= w.B ? q : big) : 0.f;
    const float ps = w.ks > 0.f ? w.ks * (big * q) : 0.f;
    const float pd = w.kd > 0.f ? w.kd * r : 0.f;
    const float p = (pa + pb) + (ps + pd);
    const float dp = (pa * a + pb * b) + (ps * s + pd * d);
    if (!(dp > 0.f) || !isfinite(dp)) return 0.f;
    const float step = (logf(p) - logC) * (p / dp);
    x -= step;
    if (fabsf(step) <= 5e-7f * (1.f + fabsf(x))) return expf(x);
  }
  return 0.f;
}

// Values (w_i / e) t^d_i of the unknowns by exponent, for axis directions along
// x and y and for diagonals with d = A + B and d = |A - B|.
template <typename Real>
struct WallValues {
  Real a, b, s, d;
};

// FP32 populations: one evaluation of p in double-float at the FP32 start, one
// Newton step from its residual.  The relative step delta of t is at most 4e-6
// (else the evaluation is repeated at the stepped start), which leaves t within
// (d - 1) / 2 delta^2 < 1e-10 and the unknowns within 1.1e-9 relative of the
// root before their FP32 rounding.  Returns false if the start did not
// converge.
__device__ __forceinline__ bool wall_root(const WallPoly& w, Df T, WallValues<float>& v) {
  constexpr Df k36e = df_const(36.0 * 2.71828182845904523536);
  constexpr Df kAxis = df_const(1.0 / 9.0 * 0.36787944117144232160);
  constexpr Df kDiag = df_const(1.0 / 36.0 * 0.36787944117144232160);
  const Df C = df_mul(T, k36e);
  float t = wall_start(w, C.hi);
  if (!(t > 0.f)) return false;
  const int mn = min(w.A, w.B), df = abs(w.A - w.B);
  const float a = (float)w.A, b = (float)w.B, s = a + b, d = (float)df;
  const Df one{1.f, 0.f};
  for (int it = 0; it < 4; ++it) {
    const Df t1{t, 0.f};
    const Df t2 = df_mul(t1, t1), t4 = df_mul(t2, t2);
    const Df q = df_mul(df_mul((mn & 2) ? t2 : one, (mn & 1) ? t : 1.f), (mn & 4) ? t4 : one);
    const Df r = df_mul(df_mul((df & 2) ? t2 : one, (df & 1) ? t : 1.f), (df & 4) ? t4 : one);
    const Df big = df_mul(q, r), all = df_mul(big, q);
    const Df pa = w.A >= w.B ? big : q, pb = w.A >= w.B ? q : big;
    const Df p = df_add(df_add(df_mul(pa, w.ka), df_mul(pb, w.kb)),
                        df_add(df_mul(all, w.ks), df_mul(r, w.kd)));
    const float dp = (w.ka * a * pa.hi + w.kb * b * pb.hi) + (w.ks * s * all.hi + w.kd * d * r.hi);
    const float delta =
        __fadd_rn(__fsub_rn(C.hi, p.hi), __fsub_rn(C.lo, p.lo)) / dp;
    if (!(fabsf(delta) <= 4e-6f)) {
      t *= 1.f + delta;
      if (!(t > 0.f) || !isfinite(t)) return false;
      continue;
    }
    auto value = [&](Df pw, float e, Df k) {  // k pw (1 + delta)^e to second order
      const float f = __fmul_rn(pw.hi, k.hi);
      const float lo = __fmaf_rn(pw.hi, k.lo, __fmaf_rn(pw.lo, k.hi, __fmaf_rn(pw.hi, k.hi, -f)));
      const float c = e * delta;
      return __fadd_rn(f, __fmaf_rn(f, fmaf(0.5f * (c - delta), c, c), lo));
    };
    v.a = value(pa, a, kAxis);
    v.b = value(pb, b, kAxis);
    v.s = value(all, s, kDiag);
    v.d = value(r, d, kDiag);
    return true;
  }
  return false;
}

// FP64 populations: Newton's method on p in FP64 from the FP32 start; a step
// under 1e-8 leaves the quadratic remainder below FP64 rounding.
__device__ __forceinline__ bool wall_root(const WallPoly& w, double T, WallValues<double>& v) {
  constexpr double kE = 2.71828182845904523536, kInvE = 0.36787944117144232160;
  const double C = 36.0 * kE * T;
  const float start = wall_start(w, (float)C);
  if (!(start > 0.f)) return false;
  double t = (double)start;
  const int mn = min(w.A, w.B), df = abs(w.A - w.B);
  const double ka = w.ka, kb = w.kb, ks = w.ks, kd = w.kd;
  const double da = ka * w.A, db = kb * w.B, ds = ks * (w.A + w.B), dd = kd * df;
  bool near = false;
  for (int it = 0; it < 8; ++it) {
    const double t2 = t * t, t4 = t2 * t2;
    double q = (mn & 1) ? t : 1.0, r = (df & 1) ? t : 1.0;
    if (mn & 2) q *= t2;
    if (mn & 4) q *= t4;
    if (df & 2) r *= t2;
    if (df & 4) r *= t4;
    const double big = q * r, all = big * q;
    const double pa = w.A >= w.B ? big : q, pb = w.A >= w.B ? q : big;
    if (near) {
      v.a = w_of(1) * kInvE * pa;
      v.b = w_of(1) * kInvE * pb;
      v.s = w_of(5) * kInvE * all;
      v.d = w_of(5) * kInvE * r;
      return true;
    }
    const double p = (ka * pa + kb * pb) + (ks * all + kd * r);
    const double dp = (da * pa + db * pb) + (ds * all + dd * r);
    const double delta = (C - p) / dp;
    t += t * delta;
    if (!(t > 0.0)) return false;
    near = fabs(delta) <= 1e-8;
  }
  return false;
}

// The wall solve of a step.  The FP64 solve takes the polynomial form: with
// its exponentials in FP64 (1/64 of the FP32 rate on this part, and every warp
// with one wall node pays for 32) the solve took nearly all of the step's time,
// 521 us a step at 1200 x 900 with FP32 populations; with one double-float
// evaluation on the FP32 pipe the step takes 42 (bounce-back walls: 12.5).  The
// general form, in logarithms, takes over where T is outside 1e-24 .. 1e24 for
// FP32 populations (there the low parts of the FP32 pairs or the powers of t
// leave FP32's range), outside 1e-34 .. 1e34 for FP64 ones (the range of the FP32
// start), where a flux of FP32 populations cancels, or where the start did not
// converge; it works on a copy of f, so that the usual path keeps f in
// registers.  A lattice that starts empty has many such walls ahead of its
// front: there a step takes 56 us instead of 184.
template <typename S, typename Real>
__device__ __noinline__ int maxent_wall_rare(Real* f, unsigned solid) {
  Real g[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) g[i] = f[i];
  const int r = maxent_wall_general<S>(g, solid);
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = g[i];
  return r;
}

template <typename S, typename Real>
__device__ __forceinline__ int maxent_wall(Real (&f)[9], unsigned solid) {
  if constexpr (sizeof(S) == 4) {
    return maxent_wall_general<S>(f, solid);
  } else {
    int mx = 0, my = 0;
#pragma unroll
    for (int i = 1; i < 9; ++i)
      if (solid & (1u << i)) {
        const int w36 = i >= 5 ? 1 : 4;
        mx -= w36 * cx_of(i);
        my -= w36 * cy_of(i);
      }
    if (mx == 0 && my == 0) return kWallSet;
    WallPoly w{abs(mx), abs(my), 0.f, 0.f, 0.f, 0.f};
    unsigned neg = 0u;
    // T = sum_{others} (e_j.m) f_j: integer multiples of the populations,
    // summed in FP64, or in double-float for FP32 populations
    double T = 0.0;
    float Th = 0.f, Tl = 0.f, most = 0.f;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      const int d = -(cx_of(i) * mx + cy_of(i) * my);
      if (((solid >> i) & 1u) && d > 0) {
        neg |= 1u << i;
        if (i == 1 || i == 3) w.ka += (float)(4 * d);
        else if (i == 2 || i == 4) w.kb += (float)(4 * d);
        else if (d == w.A + w.B) w.ks += (float)d;
        else w.kd += (float)d;
      } else if constexpr (sizeof(Real) == 8) {
        T -= (double)d * f[i];
      } else {
        const float p = __fmul_rn((float)-d, f[i]), e = __fmaf_rn((float)-d, f[i], -p);
        const float s = __fadd_rn(Th, p), bb = __fsub_rn(s, Th);
        Tl = __fadd_rn(Tl, __fadd_rn(__fadd_rn(__fsub_rn(Th, __fsub_rn(s, bb)), __fsub_rn(p, bb)), e));
        Th = s;
        most = fmaxf(most, fabsf(p));
      }
    }
    if (!neg) return kWallSet;
    const Df Td = df_norm(Th, Tl);
    const Real size = sizeof(Real) == 8 ? (Real)T : (Real)Td.hi;
    // the pair holds the sum to 2^-48 of its largest term: where less than a
    // thousandth of that is left (or a product overflows) the rare form sums it
    const Real least = sizeof(Real) == 8 ? (Real)0 : (Real)(kEdgeCancel * most);
    if (!(size >= -least) || (size == (Real)0 && least == (Real)0)) {
#pragma unroll
      for (int i = 1; i < 9; ++i)
        if (neg & (1u << i)) f[i] = (Real)0;
      return size < (Real)0 ? kWallNoRoot : kWallSet;
    }
    WallValues<Real> v;
    constexpr double kLow = sizeof(Real) == 8 ? 1e-34 : 1e-24;
    bool ok = size > (Real)kLow && size < (Real)(1.0 / kLow) && size > least;
    if (ok) {
      if constexpr (sizeof(Real) == 8) ok = wall_root(w, T, v);
      else ok = wall_root(w, Td, v);
    }
    if (!ok) {
      Real g[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) g[i] = f[i];
      const int r = maxent_wall_rare<S, Real>(g, solid);
#pragma unroll
      for (int i = 0; i < 9; ++i) f[i] = g[i];
      return r;
    }
#pragma unroll
    for (int i = 1; i < 9; ++i)
      if (neg & (1u << i)) {
        const int d = -(cx_of(i) * mx + cy_of(i) * my);
        f[i] = i == 1 || i == 3 ? v.a : i == 2 || i == 4 ? v.b : d == w.A + w.B ? v.s : v.d;
      }
    return kWallSet;
  }
}

}  // namespace lbm
