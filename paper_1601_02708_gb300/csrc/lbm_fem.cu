// lbm_fem.cu -- the continuum solver of the hybrid method: Q1 finite
// elements for the advection-diffusion equation on a structured rectangular
// mesh, stepped on the GPU (lbm_fem_*, declared in include/lbm_ade.h).
//
// Sec. 3: Galerkin weak form (Sec. 3.1.1) and SUPG (Sec. 3.1.2, Eq. "SUPG",
// "SUPG_tau"); Sec. 6.1.1: semi-discrete M d' + K d = 0 advanced by the
// generalized trapezoidal rule (Eq. "FEM_discrete"),
//     (M + theta dt K) d^{n+1} = (M - (1 - theta) dt K) d^n,
// Dirichlet nodes taking their prescribed values at t^{n+1}; every other
// boundary (the mesh edge and the edge of switched-off elements) is
// zero-flux.
//
// The element matrices of a bilinear element with uniform D and v are
// tensor products of the 1-D linear-element matrices
//     m(h) = h/6 [[2,1],[1,2]], k(h) = 1/h [[1,-1],[-1,1]],
//     c = 1/2 [[-1,1],[-1,1]]  (int phi_a phi_b'),
// assembled once on the host into 9-diagonal (one per neighbour offset)
// arrays of A = M + theta dt K and B = M - (1 - theta) dt K.  The rows of
// Dirichlet and inactive nodes are the identity in A and zero in B.  Each step
// solves A x = B d^n (+ prescribed values) by Jacobi-preconditioned
// BiCGSTAB in FP64 inside one cooperative launch, the host reading the outcome
// once per step: by tiles held in shared memory where the mesh fits (about
// 160,000 nodes, k_bicgstab_tile), else over the nodes in global memory with
// grid-wide barriers between the phases (k_bicgstab).  Sums are the same in
// every block and in every run.  A
// solve starts from the last converged solution (the previous Schwarz
// iterate inside Algorithm 1), else from d^n.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <vector>

#include "lbm_ade.h"
#include "lbm_ctx.h"

namespace {

#define FCK(call)                                                                \
  do {                                                                           \
    cudaError_t e_ = (call);                                                     \
    if (e_ != cudaSuccess)                                                       \
      return ctx_fail(e_ == cudaErrorMemoryAllocation ? LBM_ERR_NOMEM : LBM_ERR_CUDA, \
                      "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_),    \
                      __FILE__, __LINE__);                                       \
  } while (0)

constexpr int kThreads = 256;

// Outcome of one solve, written by the solver for the host.
struct Scal {
  double bnorm2, rnorm2;  // squared norms of the free rows' rhs and final residual
  int done;               // converged
  int breakdown;          // BiCGSTAB broke down before converging
};

struct Vec {
  double *x, *r, *rhat, *p, *phat, *v, *s, *shat, *t;
};

// Row (i, j) of A x for the 9-diagonal matrix: A[k][row] multiplies the
// neighbour at offset di = k % 3 - 1, dj = k / 3 - 1.
__device__ __forceinline__ double spmv_row(const double* __restrict__ A, const double* x,
                                           int i, int j, int nxn, int nyn, long long n) {
  const long long row = (long long)j * nxn + i;
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int di = k % 3 - 1, dj = k / 3 - 1;
    const int ii = i + di, jj = j + dj;
    if (ii < 0 || ii >= nxn || jj < 0 || jj >= nyn) continue;
    // x may have been written by other blocks of this launch (behind a grid
    // barrier): read it through L2, not the non-coherent L1
    acc += A[k * n + row] * __ldcg(x + (long long)jj * nxn + ii);
  }
  return acc;
}

// Row (i, j) of A y where y_m = g(m) * invd[m] is formed on the fly from
// vectors complete behind the last grid barrier (read through L2).
template <class G>
__device__ __forceinline__ double spmv_row_of(const double* __restrict__ A,
                                              const double* __restrict__ invd, G g, int i, int j,
                                              int nxn, int nyn, long long n) {
  const long long row = (long long)j * nxn + i;
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int di = k % 3 - 1, dj = k / 3 - 1;
    const int ii = i + di, jj = j + dj;
    if (ii < 0 || ii >= nxn || jj < 0 || jj >= nyn) continue;
    const long long m = (long long)jj * nxn + ii;
    acc += A[k * n + row] * (g(m) * invd[m]);
  }
  return acc;
}
// The search direction's update r + beta (p - omega v), one expression for
// the owner's stored value and for the neighbours' on-the-fly values.
__device__ __forceinline__ double next_dir(double r, double p, double v, double beta,
                                           double omega) {
  return r + beta * (p - omega * v);
}

// ---- the linear solve as one cooperative launch -----------------------------
// Every block runs the same BiCGSTAB iteration over a grid-stride share of the
// nodes; the three points per iteration where a dot product must be summed
// (the vectors the sparse products read are complete there too) are
// grid-wide barriers.  Partial dots are written per block and folded by every block in
// the same fixed order, so all blocks take the same decisions.  Each barrier
// wait is bounded: on expiry the status word is set and the blocks return.

constexpr long long kBarrierSpin = 1ll << 24;

struct Solve {
  const double* A;       // [9][n]
  const double* invd;    // [n] 1 / diagonal of A (the Jacobi preconditioner)
  const double* B;       // [9][n]
  double* d;             // state: d^n in, d^{n+1} out
  const int* fixed_id;   // -1 free, -2 inactive, >= 0 index into fixed_val
  const double* fixed_val;
  double* b;
  Vec w;
  double* part;          // [4][gridDim.x] partial dots
  unsigned* bar;         // [2] barrier count and generation
  int* status;           // 0, or 1 after an expired barrier wait
  Scal* sc;              // results: iterations, norms, breakdown
  int* iters;
  int nxn, nyn;
  long long n;
  double tol;
  int max_iter;
  int warm;  // start from w.x (the last converged solution) instead of d^n
};

// Grid-wide barrier (all blocks are resident: cooperative launch).  Returns
// false if the wait expired.
__device__ __forceinline__ bool grid_sync(unsigned* bar, int* status) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = bar + 1;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(bar, 1u) == gridDim.x - 1) {
      bar[0] = 0u;
      __threadfence();
      atomicAdd(bar + 1, 1u);
      ok = 1;
    } else {
      long long i = 0;
      while (*gen == g && ++i < kBarrierSpin) {
      }
      ok = *gen != g;
      if (!ok) atomicExch(status, 1);
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// Block partials of two dot products into part0/part1 [blockIdx.x].
__device__ __forceinline__ void block_dot2(double v0, double v1, double* part0, double* part1) {
  __shared__ double s0[kThreads / 32], s1[kThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v0 += __shfl_down_sync(0xffffffffu, v0, o);
    v1 += __shfl_down_sync(0xffffffffu, v1, o);
  }
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (lane == 0) {
    s0[wp] = v0;
    s1[wp] = v1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, c = 0.0;
    for (int k = 0; k < kThreads / 32; ++k) {
      a += s0[k];
      c += s1[k];
    }
    part0[blockIdx.x] = a;
    if (part1) part1[blockIdx.x] = c;
  }
}

// Sums of the gridDim.x partials of two dot products, the same in every
// block: thread t adds partials t and t + kThreads, each warp folds its
// threads with a fixed shuffle tree, and every thread adds the warp sums in
// warp order.  Each thread issues its loads together, so a fold costs one
// trip to L2 rather than one per partial.  gridDim.x <= kFoldCap (the host
// clamps the grid).
constexpr int kFoldCap = 2 * kThreads;
__device__ __forceinline__ void grid_fold2(const double* pa, const double* pb, double& ra,
                                           double& rb) {
  __shared__ double wa[kThreads / 32], wb[kThreads / 32];
  const int t = threadIdx.x, nb = (int)gridDim.x;
  // written by other blocks before the last grid barrier: read through L2
  const double a0 = t < nb ? __ldcg(pa + t) : 0.0;
  const double a1 = t + kThreads < nb ? __ldcg(pa + t + kThreads) : 0.0;
  const double b0 = pb && t < nb ? __ldcg(pb + t) : 0.0;
  const double b1 = pb && t + kThreads < nb ? __ldcg(pb + t + kThreads) : 0.0;
  double a = a0 + a1, b = b0 + b1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  if ((t & 31) == 0) {
    wa[t >> 5] = a;
    wb[t >> 5] = b;
  }
  __syncthreads();
  a = 0.0;
  b = 0.0;
#pragma unroll
  for (int k = 0; k < kThreads / 32; ++k) {
    a += wa[k];
    b += wb[k];
  }
  ra = a;
  rb = b;
  __syncthreads();  // the warp sums may be overwritten by the next fold
}
__device__ __forceinline__ double grid_fold(const double* part) {
  double a, b;
  grid_fold2(part, nullptr, a, b);
  return a;
}

__global__ void __launch_bounds__(kThreads) k_bicgstab(const Solve S) {
  const long long n = S.n;
  const int nxn = S.nxn, nyn = S.nyn;
  const long long stride = (long long)gridDim.x * kThreads;
  const long long p0 = blockIdx.x * (long long)kThreads + threadIdx.x;
  double* P0 = S.part;
  double* P1 = S.part + gridDim.x;
  double* P2 = S.part + 2 * gridDim.x;
  double* P3 = S.part + 3 * gridDim.x;
  const Vec w = S.w;
  const double* A = S.A;

  // right-hand side (prescribed rows: their values), initial guess
  double bb = 0.0;
  for (long long p = p0; p < n; p += stride) {
    const int i = (int)(p % nxn), j = (int)(p / nxn);
    const int f = S.fixed_id[p];
    double bv, xv;
    if (f >= 0) {
      bv = S.fixed_val[f];
      xv = bv;
    } else if (f == -2) {  // inactive
      bv = 0.0;
      xv = 0.0;
    } else {
      bv = spmv_row(S.B, S.d, i, j, nxn, nyn, n);
      xv = S.warm ? w.x[p] : S.d[p];
    }
    S.b[p] = bv;
    w.x[p] = xv;
    // the residual is measured against the free rows' right-hand side (the
    // prescribed rows are met exactly from the start and stay so)
    if (f == -1) bb += bv * bv;
  }
  block_dot2(bb, 0.0, P0, nullptr);
  if (!grid_sync(S.bar, S.status)) return;

  // r = b - A x, rhat = r, p = r
  double rr = 0.0;
  for (long long p = p0; p < n; p += stride) {
    const int i = (int)(p % nxn), j = (int)(p / nxn);
    const double r = S.b[p] - spmv_row(A, w.x, i, j, nxn, nyn, n);
    w.r[p] = r;
    w.rhat[p] = r;
    w.p[p] = r;
    w.v[p] = 0.0;  // the first direction update r + 0 (p - 0 v) reads it
    rr += r * r;
  }
  block_dot2(rr, 0.0, P1, nullptr);
  if (!grid_sync(S.bar, S.status)) return;
  double bnorm2, rnorm2;
  grid_fold2(P0, P1, bnorm2, rnorm2);
  double rho = rnorm2, alpha = 0.0, omega = 0.0, beta = 0.0;
  const double tol2 = S.tol * S.tol * bnorm2;
  bool done = rnorm2 <= tol2, breakdown = false;
  int it = 0;
  // Three grid barriers an iteration: each sparse product forms its input
  // vector on the fly from vectors that are complete behind the last barrier
  // (the new search direction p = r + beta (p - omega v) with the
  // preconditioner, then s = r - alpha v with it), so neither needs a
  // barrier of its own.  p and v alternate between two buffers, because the
  // products read the previous ones while the owners write the new ones.
  double* pc = w.p;     // search direction of the last iteration
  double* pn = w.phat;  // this iteration's
  double* vc = w.v;     // A (p invd) of the last iteration
  double* vn = w.shat;  // this iteration's
  while (!done && it < S.max_iter) {
    double d0 = 0.0;
    for (long long p = p0; p < n; p += stride) {
      const int i = (int)(p % nxn), j = (int)(p / nxn);
      pn[p] = next_dir(w.r[p], pc[p], vc[p], beta, omega);
      const double v = spmv_row_of(
          A, S.invd,
          [&](long long m) {
            return next_dir(__ldcg(w.r + m), __ldcg(pc + m), __ldcg(vc + m), beta, omega);
          },
          i, j, nxn, nyn, n);
      vn[p] = v;
      d0 += w.rhat[p] * v;
    }
    block_dot2(d0, 0.0, P0, nullptr);
    if (!grid_sync(S.bar, S.status)) return;
    const double rv = grid_fold(P0);
    if (rv == 0.0 || !isfinite(rv)) {
      breakdown = true;
      break;
    }
    alpha = rho / rv;
    double ts = 0.0, tt = 0.0;
    for (long long p = p0; p < n; p += stride) {
      const int i = (int)(p % nxn), j = (int)(p / nxn);
      const double sv = w.r[p] - alpha * vn[p];
      w.s[p] = sv;
      const double t = spmv_row_of(
          A, S.invd, [&](long long m) { return __ldcg(w.r + m) - alpha * __ldcg(vn + m); }, i, j,
          nxn, nyn, n);
      w.t[p] = t;
      ts += t * sv;
      tt += t * t;
    }
    block_dot2(ts, tt, P0, P1);
    if (!grid_sync(S.bar, S.status)) return;
    double tsum, tsv;
    grid_fold2(P1, P0, tsum, tsv);
    omega = tsum > 0.0 ? tsv / tsum : 0.0;
    double rh = 0.0;
    rr = 0.0;
    for (long long p = p0; p < n; p += stride) {
      const double sv = w.s[p];
      w.x[p] += alpha * (pn[p] * S.invd[p]) + omega * (sv * S.invd[p]);
      const double r = sv - omega * w.t[p];
      w.r[p] = r;
      rh += w.rhat[p] * r;
      rr += r * r;
    }
    block_dot2(rh, rr, P2, P3);
    if (!grid_sync(S.bar, S.status)) return;
    double rho_new;
    grid_fold2(P2, P3, rho_new, rnorm2);
    ++it;
    if (rnorm2 <= tol2) {
      done = true;
      break;
    }
    if (rho_new == 0.0 || omega == 0.0 || !isfinite(rho_new)) {
      breakdown = true;
      break;
    }
    beta = (rho_new / rho) * (alpha / omega);
    rho = rho_new;
    double* tp = pc;
    pc = pn;
    pn = tp;
    double* tv = vc;
    vc = vn;
    vn = tv;
  }
  // every block copies its own share of x: no barrier needed
  for (long long p = p0; p < n; p += stride) S.d[p] = w.x[p];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    S.sc->bnorm2 = bnorm2;
    S.sc->rnorm2 = rnorm2;
    S.sc->done = done ? 1 : 0;
    S.sc->breakdown = breakdown ? 1 : 0;
    *S.iters = it;
  }
}

// ---- the linear solve with its vectors in shared memory ---------------------
// The same preconditioned BiCGSTAB for systems whose nodes fit the SMs' shared
// memory, one block and one tile of tw x th nodes per SM.  What bounds it is
// the FP64 pipe (1/64 of the FP32 rate on this part: a warp instruction holds
// the SM's for 16 cycles) and the latency of the sums over the grid, so:
//  - a block keeps r, p, v, p invd, s invd, t and the operator's rows of its
//    tile in shared memory, and r, p, v, t of the one-node ring around it too,
//    updating the ring's entries itself (1.26 times the tile's work at 22 x 13
//    nodes) instead of forming nine neighbours' values for every node;
//  - only the nodes on a tile's border go through global memory, v after the
//    first product and t after the second;
//  - two sums over the grid an iteration instead of three: with t.s, t.t,
//    rhat.s, rhat.t and s.s from the second one, rhat.r = rhat.s - omega rhat.t
//    and r.r = s.s - 2 omega t.s + omega^2 t.t.  Where that difference cancels
//    ten digits the two products are summed directly;
//  - every value that crosses blocks carries its own tag (put_tagged): no
//    barrier, counter or memory fence, one trip through L2 for a sum;
//  - scalars are formed by one thread.
// A step of a 400 x 100 mesh with 13 to 17 iterations took 640 us with the
// cooperative solve above (which forms p and s of nine neighbours per node and
// crosses three atomic barriers an iteration) and takes 220 us; one of 40 x 10
// elements in a single block, bound by that SM's FP64 pipe, took 15 us an
// iteration, now 9.  An iteration's time is the FP64 pipe's latency (about 200
// cycles an operation) along its chains: 2 us of products, 2 us of scalars, and
// about 5 us for the two exchanges.
constexpr int kTileVals = 5;        // values an exchange carries at most
constexpr int kTileSlot = 8;        // 16-byte words from block to block: one 128-byte line
constexpr int kTileMaxBlocks = 256;  // at most eight per polling lane
// 12 warps: one node a thread of the 286-node tiles of a 400 x 100 mesh and of
// their rings (with 8 the few nodes left over cost a second pass).  A step of
// 23 iterations with 8, 12 and 16 warps, us: 451 nodes 227, 229, 256; 20,301
// 277, 279, 326; 40,501 339, 314, 354; 60,501 363, 390, 408; 100,651 433, 421,
// 485; 135,751 469, 468, 546.
constexpr int kTileThreads = 384;
constexpr unsigned long long kTileWaitNs = 2000000000ull;  // 2 s

struct Outcome {  // of one solve, in page-locked host memory
  Scal sc;
  int iters, status;
};

struct TileSolve {
  const double* A;
  const double* invd;
  const double* B;
  double* d;         // state: d^n in, d^{n+1} out
  double* xw;        // the last converged solution
  const int* fixed_id;
  const double* fixed_val;
  // [n] v and t on the tiles' borders, tagged (tpub: r before the first
  // iteration).  A block writes v again only past the exchange that follows
  // its neighbours' reads of it (the second product's; for t the next first
  // product's), so a reader never misses its tag.
  ulonglong2* vpub;
  ulonglong2* tpub;
  ulonglong2* slots;  // [2][blocks][kTileSlot] exchanged values
  Outcome* out;
  int nxn, nyn, tw, th, ntx;
  unsigned epoch;    // tag of the solve's first exchange
  double tol;
  int max_iter, warm;
};

// Shared memory of a block, in doubles.
__host__ __device__ constexpr size_t tile_doubles(int tw, int th) {
  const size_t ring = (size_t)(tw + 2) * (th + 2), own = (size_t)tw * th;
  return 7 * ring + 11 * own + kTileVals * kTileThreads + ring + own;
}

// Exponent field of a double: 0 for zeros and numbers below the normal range,
// 0x7ff for infinities and NaN.
__device__ __forceinline__ int exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

__device__ __forceinline__ unsigned long long tile_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// A double in memory that other blocks read while it is written: two 64-bit
// words, each half of it beside the tag of the exchange it belongs to.  A
// reader knows the value by its words alone, so no flag, counter or fence
// stands between the blocks.
__device__ __forceinline__ void put_tagged(ulonglong2* at, double v, unsigned tag) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned long long t = (unsigned long long)tag << 32;
  asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(at), "l"(t | (b & 0xFFFFFFFFull)),
               "l"(t | (b >> 32))
               : "memory");
}
// The values with this tag at n places (at most N), all loads of a round in
// flight together; bounded, false when the wait expired.
template <int N, class At>
__device__ __forceinline__ bool get_tagged(At at, int n, unsigned tag, double (&v)[N]) {
  unsigned long long t0 = 0;
  for (int spins = 1;; ++spins) {
    unsigned long long lo[N], hi[N];
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i < n)
        asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];"
                     : "=l"(lo[i]), "=l"(hi[i])
                     : "l"(at(i))
                     : "memory");
    bool all = true;
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i < n) {
        all = all && (unsigned)(lo[i] >> 32) == tag && (unsigned)(hi[i] >> 32) == tag;
        v[i] = __longlong_as_double((long long)((lo[i] & 0xFFFFFFFFull) | (hi[i] << 32)));
      } else {
        v[i] = 0.0;
      }
    if (all) return true;
    if ((spins & 255) == 0) {
      const unsigned long long now = tile_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > kTileWaitNs) return false;
    }
  }
}

// Sum of a warp's 32 x N doubles (the first n of each lane), the same in every
// lane.  An FP64 addition returns after about 200 cycles here, so a shuffle
// tree of them is slow; integers are not: every value is rounded once to
// 2^-53 of the largest one's power of two, and the integers are summed exactly
// in any order (three limbs, one reduction instruction each).  The rounding is
// no more than that of adding the values one by one in FP64.
template <int N>
__device__ __forceinline__ double warp_sum(const double (&a)[N], int n) {
  static_assert(32 * N <= 512, "54-bit integers, 9 bits of headroom, a sign");
  constexpr unsigned kFull = 0xffffffffu;
  unsigned top = 0;
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (i < n) top = max(top, (unsigned)exponent(a[i]));
  top = __reduce_max_sync(kFull, top);
  if (top == 0u) top = 1u;  // zeros and numbers below the normal range, in units of 2^-1074
  if (top == 0x7ffu) return __longlong_as_double(0x7ff8000000000000ll);
  long long s = 0;
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (i < n) {
      const long long b = __double_as_longlong(a[i]);
      const int e = (int)((b >> 52) & 0x7ff), sh = (int)top - (e > 0 ? e : 1);
      long long m = ((b & 0xFFFFFFFFFFFFFll) | (e > 0 ? 0x10000000000000ll : 0ll)) << 1;
      m = sh > 54 ? 0 : (m + ((1ll << sh) >> 1)) >> sh;
      s += b < 0 ? -m : m;
    }
  const unsigned lo = __reduce_add_sync(kFull, (unsigned)s & 0x3FFFFFFu);
  const unsigned mid = __reduce_add_sync(kFull, (unsigned)(s >> 26) & 0x3FFFFFFu);
  const int hi = __reduce_add_sync(kFull, (int)(s >> 52));
  const long long S = ((long long)hi << 52) + ((long long)mid << 26) + (long long)lo;
  // value = S 2^(top - 1023 - 53)
  if (top <= 64u) return ldexp((double)S, (int)top - 1076);
  return (double)S * __longlong_as_double((long long)(top - 53u) << 52);
}

// Sums of V values over the threads of every block, left in sums[V] (the same
// in every block): warp k sums the block's value k, the first warp writes the
// block's values to its slot, and warp k reads and sums every block's value k;
// meanwhile the other warps fetch the ring's border values, pub[rnode] to
// u[rpos].  A slot is a 128-byte line of its own, written by one instruction:
// a line that is written several times while it is polled is fetched anew
// after every write, and values arrived 2.4 to 4.6 us after the last block had
// written (words of eight blocks in a line, or five writes to one line) instead
// of 0.9.  Slots alternate between two sets: a block can write a set again only
// after every block has read it, since the exchange between them needs them
// all.  The caller synchronises before it reads sums or the ring; *dead is set
// when a wait expired.
template <int V>
__device__ __forceinline__ void tile_exchange(const double (&v)[V], int active, ulonglong2* slots,
                                              unsigned tag, double* red, double* sums, int* dead,
                                              const ulonglong2* pub, const int* rnode,
                                              const int* rpos, int nr, double* u) {
  constexpr int kW = kTileThreads / 32, kB = kTileMaxBlocks / 32;
  static_assert(V < kW, "a warp per value, and some for the ring");
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, nb = (int)gridDim.x;
  ulonglong2* set = slots + (size_t)(tag & 1u) * nb * kTileSlot;
#pragma unroll
  for (int k = 0; k < V; ++k) red[k * kTileThreads + t] = v[k];
  __syncthreads();
  if (w < V) {
    double a[kW];
#pragma unroll
    for (int i = 0; i < kW; ++i) a[i] = red[w * kTileThreads + 32 * i + lane];
    const double s = warp_sum(a, active);
    if constexpr (V == 1) {
      if (lane == 0) put_tagged(set + (size_t)blockIdx.x * kTileSlot, s, tag);
    } else {
      if (lane == 0) sums[w] = s;
      asm volatile("bar.sync 1, %0;" ::"n"(32 * V) : "memory");
      if (w == 0 && lane < V) put_tagged(set + (size_t)blockIdx.x * kTileSlot + lane, sums[lane], tag);
      if (w == 0) __syncwarp();
      asm volatile("bar.sync 1, %0;" ::"n"(32 * V) : "memory");  // sums is rewritten below
    }
    double g[kB];
    if (!get_tagged([&](int i) { return set + (size_t)(lane + 32 * i) * kTileSlot + w; },
                    (nb - lane + 31) / 32, tag, g))
      *dead = 1;
    __syncwarp();
    const double total = warp_sum(g, (nb + 31) / 32);
    if (lane == 0) sums[w] = total;
  } else {
    for (int e = t - 32 * V; e < nr; e += kTileThreads - 32 * V) {
      double val[1];
      if (!get_tagged([&](int) { return pub + rnode[e]; }, 1, tag, val)) *dead = 1;
      u[rpos[e]] = val[0];
    }
  }
}

__global__ void __launch_bounds__(kTileThreads) k_bicgstab_tile(const TileSolve S) {
  extern __shared__ double sm[];
  __shared__ double sums[kTileVals];
  __shared__ double bc[3];  // alpha, omega, beta
  // 0 go on, 1 converged, 2 broke down, 3 iteration limit, 4 sum again, 5 a wait expired
  __shared__ int stop;
  __shared__ int nring, dead;
  const int nxn = S.nxn, nyn = S.nyn, ld = S.tw + 2, ring = ld * (S.th + 2), cap = S.tw * S.th;
  const int x0 = (int)(blockIdx.x % S.ntx) * S.tw, y0 = (int)(blockIdx.x / S.ntx) * S.th;
  const int ow = min(S.tw, nxn - x0), oh = min(S.th, nyn - y0), own = ow * oh;
  const long long n = (long long)nxn * nyn;
  const int tid = threadIdx.x;
  const bool lead = tid == 0;
  double* r = sm;            // ring arrays: [th + 2][ld]
  double* p = r + ring;
  double* v = p + ring;
  double* t = v + ring;
  double* y = t + ring;      // p invd (x before the first iteration)
  double* z = y + ring;      // s invd
  double* iv = z + ring;
  double* A = iv + ring;     // [9][cap] the operator's rows of the tile
  double* x = A + 9 * cap;
  double* rhat = x + cap;
  double* red = rhat + cap;  // [kTileVals][kTileThreads]
  int* rpos = (int*)(red + kTileVals * kTileThreads);  // ring list: position, node
  int* rnode = rpos + ring;
  int* opos = rnode + ring;  // position of each own node, border flag in bit 30
  int* onode = opos + cap;
  constexpr int kBorder = 1 << 30;
  unsigned tag = S.epoch;

  if (lead) nring = dead = 0;
  __syncthreads();
  auto start = [&](long long g) {  // the solve's starting value at a node
    const int f = S.fixed_id[g];
    return f >= 0 ? S.fixed_val[f] : f == -2 ? 0.0 : S.warm ? S.xw[g] : S.d[g];
  };
  for (int c = tid; c < ring; c += kTileThreads) {
    const int cj = c / ld, ci = c - cj * ld, gi = x0 + ci - 1, gj = y0 + cj - 1;
    const bool in = ci <= ow + 1 && cj <= oh + 1 && gi >= 0 && gi < nxn && gj >= 0 && gj < nyn;
    const bool mine = in && ci >= 1 && ci <= ow && cj >= 1 && cj <= oh;
    const long long g = (long long)gj * nxn + gi;
    r[c] = p[c] = v[c] = t[c] = z[c] = 0.0;
    y[c] = in ? start(g) : 0.0;
    iv[c] = in ? S.invd[g] : 0.0;
    if (mine) {
      const int q = (cj - 1) * ow + (ci - 1);
      const bool edge = ci == 1 || ci == ow || cj == 1 || cj == oh;
      opos[q] = c | (edge ? kBorder : 0);
      onode[q] = (int)g;
    } else if (in) {
      const int e = atomicAdd(&nring, 1);
      rpos[e] = c;
      rnode[e] = (int)g;
    }
  }
  for (int e = tid; e < 9 * own; e += kTileThreads) {
    const int k = e / own, q = e - k * own, qj = q / ow, qi = q - qj * ow;
    A[k * cap + q] = S.A[k * n + (long long)(y0 + qj) * nxn + x0 + qi];
  }
  __syncthreads();
  // row q of A u for a ring array u (entries off the mesh are zero)
  auto row = [&](const double* u, int q, int c) {
    double acc[3] = {0.0, 0.0, 0.0};  // three chains: an FP64 operation is slow to return
#pragma unroll
    for (int k = 0; k < 9; ++k) acc[k / 3] += A[k * cap + q] * u[c + (k / 3 - 1) * ld + (k % 3 - 1)];
    return (acc[0] + acc[1]) + acc[2];
  };
  // right-hand side and first residual; the norm is that of the free rows
  double bb = 0.0, rr = 0.0;
  for (int q = tid; q < own; q += kTileThreads) {
    const int c = opos[q] & ~kBorder, g = onode[q], f = S.fixed_id[g];
    double bv;
    if (f >= 0) bv = S.fixed_val[f];
    else if (f == -2) bv = 0.0;
    else {
      bv = spmv_row(S.B, S.d, x0 + (c % ld) - 1, y0 + (c / ld) - 1, nxn, nyn, n);
      bb += bv * bv;
    }
    const double rq = bv - row(y, q, c);
    x[q] = y[c];
    rhat[q] = rq;
    r[c] = p[c] = rq;
    if (opos[q] & kBorder) put_tagged(S.tpub + g, rq, tag);
    rr += rq * rq;
  }
  const int nr = nring;
  const int active = min(kTileThreads, own + 31) / 32;  // warps that hold own nodes
  {
    const double val[2] = {bb, rr};
    tile_exchange<2>(val, active, S.slots, tag, red, sums, &dead, S.tpub, rnode, rpos, nr, r);
  }
  __syncthreads();
  // thread 0's state: norms, rho and the iteration count
  double bnorm2 = 0.0, rnorm2 = 0.0, tol2 = 0.0, rho = 0.0, rv = 0.0;
  int it = 0;
  if (lead) {
    bnorm2 = sums[0];
    rnorm2 = rho = sums[1];
    tol2 = S.tol * S.tol * bnorm2;
    bc[0] = bc[1] = bc[2] = 0.0;
    stop = dead ? 5 : rnorm2 <= tol2 ? 1 : S.max_iter <= 0 ? 3 : 0;
  }
  __syncthreads();
  while (!stop) {
    ++tag;
    // p = r + beta (p - omega v), on the ring too; y = p invd
    const double beta = bc[2], omega_old = bc[1];
    for (int c = tid; c < ring; c += kTileThreads) {
      const double pc = next_dir(r[c], p[c], v[c], beta, omega_old);
      p[c] = pc;
      y[c] = pc * iv[c];
    }
    __syncthreads();
    double dot[1] = {0.0};
    for (int q = tid; q < own; q += kTileThreads) {
      const int c = opos[q] & ~kBorder;
      const double vq = row(y, q, c);
      v[c] = vq;
      if (opos[q] & kBorder) put_tagged(S.vpub + onode[q], vq, tag);
      dot[0] += rhat[q] * vq;
    }
    tile_exchange<1>(dot, active, S.slots, tag, red, sums, &dead, S.vpub, rnode, rpos, nr, v);
    if (lead) {  // the thread that folded the sum
      rv = sums[0];
      if (rv == 0.0 || !isfinite(rv)) stop = 2;
      else bc[0] = rho / rv;
    }
    __syncthreads();
    if (stop) break;
    // s = r - alpha v (in place), z = s invd
    const double alpha = bc[0];
    for (int c = tid; c < ring; c += kTileThreads) {
      const double sc = r[c] - alpha * v[c];
      r[c] = sc;
      z[c] = sc * iv[c];
    }
    __syncthreads();
    ++tag;
    double d5[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int q = tid; q < own; q += kTileThreads) {
      const int c = opos[q] & ~kBorder;
      const double tq = row(z, q, c), sq = r[c], hq = rhat[q];
      t[c] = tq;
      if (opos[q] & kBorder) put_tagged(S.tpub + onode[q], tq, tag);
      x[q] += alpha * y[c];
      d5[0] += tq * sq;
      d5[1] += tq * tq;
      d5[2] += hq * sq;
      d5[3] += hq * tq;
      d5[4] += sq * sq;
    }
    tile_exchange<5>(d5, active, S.slots, tag, red, sums, &dead, S.tpub, rnode, rpos, nr, t);
    __syncthreads();
    // omega = t.s / t.t and beta = (rho_new / rho) (alpha / omega), where
    // alpha / rho = 1 / (rhat.v): the two divisions run side by side, in lanes
    // 0 and 1 of the first warp
    double rho_new = 0.0, omega_l = 0.0, per_rho = 0.0;
    bool far = false;
    auto verdict = [&]() {  // thread 0, after rho_new and rnorm2
      ++it;
      if (dead) stop = 5;
      else if (rnorm2 <= tol2) stop = 1;
      else if (rho_new == 0.0 || omega_l == 0.0 || !isfinite(rho_new)) stop = 2;
      else if (it >= S.max_iter) stop = 3;
      else {
        stop = 0;
        bc[2] = rho_new * per_rho;
        if (far) bc[2] = rho_new / rv * per_rho;
      }
      rho = rho_new;
    };
    if (tid < 32) {
      const double rv0 = __shfl_sync(0xffffffffu, rv, 0);
      // the product t.s rhat.v is of the data's fourth power, and out of range
      // before their squares are: then beta = (rho_new / rhat.v) (t.t / t.s)
      far = (unsigned)(exponent(sums[0]) + exponent(rv0) - 1023 - 64) > 1900u;
      const double q = tid == 1 ? sums[1] / (far ? sums[0] : sums[0] * rv0) : sums[0] / sums[1];
      per_rho = __shfl_sync(0xffffffffu, q, 1);
      omega_l = sums[1] > 0.0 ? q : 0.0;
      if (lead) {
        bc[1] = omega_l;
        rho_new = sums[2] - omega_l * sums[3];
        rnorm2 = sums[4] - omega_l * (2.0 * sums[0] - omega_l * sums[1]);
        if ((!(rnorm2 > 1e-10 * sums[4]) && sums[4] > 0.0) ||
            exponent(sums[2]) - exponent(rho_new) > 33)  // (2^-33 = 1.2e-10)
          stop = 4;
        else verdict();
      }
    }
    __syncthreads();
    const double omega = bc[1];
    for (int q = tid; q < own; q += kTileThreads) x[q] += omega * z[opos[q] & ~kBorder];
    for (int c = tid; c < ring; c += kTileThreads) r[c] -= omega * t[c];
    if (stop == 4) {  // (the same in every block: all hold the same sums)
      __syncthreads();
      double d2[2] = {0.0, 0.0};
      for (int q = tid; q < own; q += kTileThreads) {
        const double rq = r[opos[q] & ~kBorder];
        d2[0] += rhat[q] * rq;
        d2[1] += rq * rq;
      }
      ++tag;
      tile_exchange<2>(d2, active, S.slots, tag, red, sums, &dead, nullptr, rnode, rpos, 0, t);
      __syncthreads();
      if (lead) {
        rho_new = sums[0];
        rnorm2 = sums[1];
        verdict();
      }
      __syncthreads();
    }
  }
  if (dead) {  // a wait expired (stop is 2 or 5 in this block)
    if (lead) *(volatile int*)&S.out->status = 1;
    return;
  }
  // the solution, and the warm start of the next solve
  for (int q = tid; q < own; q += kTileThreads) {
    S.d[onode[q]] = x[q];
    S.xw[onode[q]] = x[q];
  }
  if (lead && blockIdx.x == 0) {
    S.out->sc.bnorm2 = bnorm2;
    S.out->sc.rnorm2 = rnorm2;
    S.out->sc.done = stop == 1 ? 1 : 0;
    S.out->sc.breakdown = stop == 2 ? 1 : 0;
    S.out->iters = it;
  }
}

// FE interpolation (bilinear on the containing element) of d at points
__global__ void k_interp(const double* __restrict__ d, int nex, int ney, double x0, double y0,
                         double hx, double hy, const double* __restrict__ xy, int npts,
                         double* __restrict__ out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= npts) return;
  const double px = (xy[2 * k] - x0) / hx, py = (xy[2 * k + 1] - y0) / hy;
  int i = (int)floor(px), j = (int)floor(py);
  i = i < 0 ? 0 : (i > nex - 1 ? nex - 1 : i);
  j = j < 0 ? 0 : (j > ney - 1 ? ney - 1 : j);
  const double gx = px - i, gy = py - j;
  const int nxn = nex + 1;
  const double* r0 = d + (long long)j * nxn + i;
  const double* r1 = r0 + nxn;
  out[k] = r0[0] * (1 - gx) * (1 - gy) + r0[1] * gx * (1 - gy) + r1[1] * gx * gy +
           r1[0] * (1 - gx) * gy;
}

}  // namespace

struct lbm_fem {
  lbm_fem_params p;
  int nxn = 0, nyn = 0;
  long long n = 0;
  int n_dir = 0;
  cudaStream_t stream = nullptr;
  int device = 0;
  double* A = nullptr;  // [9][n]
  double* B = nullptr;  // [9][n]
  double* d = nullptr;  // state
  double* b = nullptr;  // right-hand side
  double* invd = nullptr;  // 1 / diagonal of A
  Vec w{};
  double* vecs = nullptr;   // storage of w
  int* fixed_id = nullptr;  // per node: index into the prescribed values, -1 free, -2 inactive
  double* fixed_val = nullptr;
  double* part = nullptr;   // [4][grid] partial dots
  Scal* sc = nullptr;
  int* iters = nullptr;
  unsigned* bar = nullptr;  // grid barrier [2]
  int* status = nullptr;
  int grid = 0;             // blocks of the cooperative solve (all resident)
  double* scratch = nullptr;  // staging of host points / results of lbm_fem_interpolate
  Outcome* pinned = nullptr;  // page-locked outcome of a solve
  // solve by tiles (k_bicgstab_tile): tile size, 0 where the mesh does not fit
  int tw = 0, th = 0, tiles = 0;
  size_t tile_smem = 0;
  ulonglong2* tagged = nullptr;  // exchange slots [2][tiles][kTileSlot], then v and t [2][n]
  size_t tagged_b = 0;
  unsigned epoch = 1;           // tag of the next solve's first exchange
  size_t scratch_n = 0;
  int last_iters = 0;
  double last_resid = 0.0;
  // w.x holds the last converged solution: the next solve starts from it.
  // Within a Schwarz step (Algorithm 1) every iteration after the first
  // solves the same system with nearby Dirichlet data, so the previous
  // iterate is a far better start than d^n; in plain time stepping it is
  // d^n itself.  The answer is the same to the solve's tolerance.
  bool warm = false;
};

namespace {

// Tile of k_bicgstab_tile for the mesh: the one whose block does the least
// FP64 work per iteration, in warp instructions (6 a ring entry and 26 an own
// node, and about 80 + 6 (blocks / 32 + 5) for the sums), among those whose
// blocks are at most one per SM and fit its shared memory, which is the better
// solve wherever it fits: a step of 23 iterations takes 229 us instead of 266
// with 451 nodes, 262 instead of 703 with 5,151, 279 instead of 687 with 20,301,
// 390 instead of 1008 with 60,501, 468 instead of 1217 with 135,751.  Larger meshes keep
// the cooperative solve over all nodes (tiles = 0).
constexpr size_t kTileSmem = 200 * 1024;
void pick_tile(lbm_fem* f, int sms) {
  const int most = sms < kTileMaxBlocks ? sms : kTileMaxBlocks;
  const int cap = (int)(kTileSmem / sizeof(double) / 18);  // no tile holds more nodes
  long long best = -1;
  f->tiles = 0;
  if (f->n > (long long)most * cap) return;
  for (int tw = 1; tw <= f->nxn && tw <= cap; ++tw)
    for (int th = 1; th <= f->nyn && tw * th <= cap; ++th) {
      const long long nb = (long long)((f->nxn + tw - 1) / tw) * ((f->nyn + th - 1) / th);
      if (nb > most) continue;
      const size_t smem = tile_doubles(tw, th) * sizeof(double);
      if (smem > kTileSmem) continue;
      const long long ring = ((tw + 2) * (th + 2) + 31) / 32, own = (tw * th + 31) / 32;
      const long long cost = 6 * ring + 26 * own + 6 * ((nb + 31) / 32);
      if (best < 0 || cost < best) {
        best = cost;
        f->tw = tw;
        f->th = th;
        f->tiles = (int)nb;
        f->tile_smem = smem;
      }
    }
}

void fem_free(lbm_fem* f) {
  void* ptrs[] = {f->A, f->B, f->d, f->b, f->vecs, f->fixed_id, f->fixed_val, f->part,
                  f->sc, f->iters, f->scratch, f->bar, f->status, f->invd, f->tagged};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (f->pinned) cudaFreeHost(f->pinned);
  delete f;
}

// Element matrices (Galerkin + SUPG) of one hx x hy element in the local
// node order (0,0), (1,0), (1,1), (0,1).
void element(const lbm_fem_params& p, double tau, double Me[4][4], double Ke[4][4]) {
  const double mx[2][2] = {{p.hx / 3, p.hx / 6}, {p.hx / 6, p.hx / 3}};
  const double my[2][2] = {{p.hy / 3, p.hy / 6}, {p.hy / 6, p.hy / 3}};
  const double kx[2][2] = {{1 / p.hx, -1 / p.hx}, {-1 / p.hx, 1 / p.hx}};
  const double ky[2][2] = {{1 / p.hy, -1 / p.hy}, {-1 / p.hy, 1 / p.hy}};
  const double c[2][2] = {{-0.5, 0.5}, {-0.5, 0.5}};  // int phi_a phi_b'
  const int loc[4][2] = {{0, 0}, {1, 0}, {1, 1}, {0, 1}};
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 4; ++b) {
      const int ia = loc[a][0], ja = loc[a][1], ib = loc[b][0], jb = loc[b][1];
      const double mass = mx[ia][ib] * my[ja][jb];
      const double adv = p.vx * c[ia][ib] * my[ja][jb] + p.vy * mx[ia][ib] * c[ja][jb];
      const double dif = p.D * (kx[ia][ib] * my[ja][jb] + mx[ia][ib] * ky[ja][jb]);
      // SUPG: the test function gains tau v.grad N_a
      const double adv_t = p.vx * c[ib][ia] * my[ja][jb] + p.vy * mx[ia][ib] * c[jb][ja];
      const double vv = p.vx * p.vx * kx[ia][ib] * my[ja][jb] +
                        p.vy * p.vy * mx[ia][ib] * ky[ja][jb] +
                        p.vx * p.vy * (c[ib][ia] * c[ja][jb] + c[ia][ib] * c[jb][ja]);
      Me[a][b] = mass + tau * adv_t;
      Ke[a][b] = adv + dif + tau * vv;
    }
}

// tau_e = h / (2|v|) (coth Pe - 1/Pe), Pe = |v| h / (2D), h the element
// length along the flow, min(hx / |v^_x|, hy / |v^_y|).
double supg_tau(const lbm_fem_params& p) {
  const double speed = std::hypot(p.vx, p.vy);
  if (!p.supg || speed == 0.0) return 0.0;
  const double ux = std::fabs(p.vx) / speed, uy = std::fabs(p.vy) / speed;
  double h = INFINITY;
  if (ux > 0) h = std::fmin(h, p.hx / ux);
  if (uy > 0) h = std::fmin(h, p.hy / uy);
  if (!(p.D > 0.0)) return h / (2.0 * speed);
  const double pe = speed * h / (2.0 * p.D);
  const double xi = pe > 30.0 ? 1.0 - 1.0 / pe : (std::cosh(pe) / std::sinh(pe) - 1.0 / pe);
  return h / (2.0 * speed) * xi;
}

lbm_status fem_setup(lbm_fem* f, const uint8_t* elem_active, const int* dir_nodes,
                     const double* d0) {
  const lbm_fem_params& p = f->p;
  const int nxn = f->nxn;
  const long long n = f->n;
  std::vector<double> A(9 * n, 0.0), B(9 * n, 0.0);
  std::vector<char> touched(n, 0);
  double Me[4][4], Ke[4][4];
  element(p, supg_tau(p), Me, Ke);
  const int loc[4][2] = {{0, 0}, {1, 0}, {1, 1}, {0, 1}};
  const double ca = p.theta * p.dt, cb = -(1.0 - p.theta) * p.dt;
  for (int j = 0; j < p.ney; ++j)
    for (int i = 0; i < p.nex; ++i) {
      if (elem_active && !elem_active[(long long)j * p.nex + i]) continue;
      for (int a = 0; a < 4; ++a) {
        const int ra = (j + loc[a][1]) * nxn + (i + loc[a][0]);
        touched[ra] = 1;
        for (int b = 0; b < 4; ++b) {
          const int di = loc[b][0] - loc[a][0], dj = loc[b][1] - loc[a][1];
          const int k = (dj + 1) * 3 + (di + 1);
          A[k * n + ra] += Me[a][b] + ca * Ke[a][b];
          B[k * n + ra] += Me[a][b] + cb * Ke[a][b];
        }
      }
    }
  std::vector<int> fid(n, -1);
  for (long long q = 0; q < n; ++q)
    if (!touched[q]) fid[q] = -2;
  for (int k = 0; k < f->n_dir; ++k) {
    const int q = dir_nodes[k];
    if (q < 0 || q >= n) return ctx_fail(LBM_ERR_ARG, "lbm_fem_init: Dirichlet node %d out of range", q);
    if (fid[q] >= 0) return ctx_fail(LBM_ERR_ARG, "lbm_fem_init: Dirichlet node %d repeated", q);
    fid[q] = k;
  }
  for (long long q = 0; q < n; ++q)
    if (fid[q] != -1) {  // identity row in A, zero row in B
      for (int k = 0; k < 9; ++k) {
        A[k * n + q] = k == 4 ? 1.0 : 0.0;
        B[k * n + q] = 0.0;
      }
    }
  std::vector<double> invd(n);
  for (long long q = 0; q < n; ++q) invd[q] = 1.0 / A[4 * n + q];
  FCK(cudaMemcpyAsync(f->A, A.data(), 9 * n * sizeof(double), cudaMemcpyHostToDevice, f->stream));
  FCK(cudaMemcpyAsync(f->invd, invd.data(), n * sizeof(double), cudaMemcpyHostToDevice,
                      f->stream));
  FCK(cudaMemcpyAsync(f->B, B.data(), 9 * n * sizeof(double), cudaMemcpyHostToDevice, f->stream));
  FCK(cudaMemcpyAsync(f->fixed_id, fid.data(), n * sizeof(int), cudaMemcpyHostToDevice, f->stream));
  std::vector<double> d(n, 0.0);
  if (d0) {
    const bool dev = ctx_on_device(d0);
    if (dev) FCK(cudaMemcpy(d.data(), d0, n * sizeof(double), cudaMemcpyDeviceToHost));
    else std::memcpy(d.data(), d0, n * sizeof(double));
  }
  for (long long q = 0; q < n; ++q)
    if (fid[q] == -2) d[q] = 0.0;
  FCK(cudaMemcpyAsync(f->d, d.data(), n * sizeof(double), cudaMemcpyHostToDevice, f->stream));
  FCK(cudaStreamSynchronize(f->stream));
  return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_fem_init(lbm_fem** out, const lbm_fem_params* p, const uint8_t* elem_active,
                        int n_dir, const int* dir_nodes, const double* d0, void* stream) {
  if (!out || !p) return ctx_fail(LBM_ERR_ARG, "lbm_fem_init: null argument");
  *out = nullptr;
  if (p->nex < 1 || p->ney < 1 || !(p->hx > 0) || !(p->hy > 0) || !(p->dt > 0) ||
      !(p->theta >= 0.0 && p->theta <= 1.0) || !(p->D >= 0.0) || n_dir < 0 ||
      (n_dir > 0 && !dir_nodes))
    return ctx_fail(LBM_ERR_ARG, "lbm_fem_init: bad parameters");
  if ((long long)(p->nex + 1) * (p->ney + 1) > (1ll << 30))
    return ctx_fail(LBM_ERR_ARG, "lbm_fem_init: mesh too large");
  lbm_fem* f = new lbm_fem();
  f->p = *p;
  if (!(f->p.tol > 0)) f->p.tol = 1e-12;
  if (f->p.max_iter <= 0) f->p.max_iter = 1000;
  f->nxn = p->nex + 1;
  f->nyn = p->ney + 1;
  f->n = (long long)f->nxn * f->nyn;
  f->n_dir = n_dir;
  f->stream = (cudaStream_t)stream;
  const long long n = f->n;
  cudaError_t e = cudaSuccess;
  auto al = [&](void** ptr, size_t bytes) {
    if (e == cudaSuccess) e = cudaMalloc(ptr, bytes);
  };
  al((void**)&f->A, 9 * n * sizeof(double));
  al((void**)&f->B, 9 * n * sizeof(double));
  al((void**)&f->d, n * sizeof(double));
  al((void**)&f->b, n * sizeof(double));
  al((void**)&f->invd, n * sizeof(double));
  al((void**)&f->vecs, 9 * n * sizeof(double));
  al((void**)&f->fixed_id, n * sizeof(int));
  al((void**)&f->fixed_val, (n_dir > 0 ? n_dir : 1) * sizeof(double));
  {
    int dev = 0, sms = 0, coop = 0, per_sm = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    f->device = dev;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bicgstab, kThreads, 0);
    if (e == cudaSuccess && (!coop || per_sm < 1)) {
      fem_free(f);
      return ctx_fail(LBM_ERR_CUDA, "lbm_fem_init: the device has no cooperative launch");
    }
    const long long need = (n + kThreads - 1) / kThreads;
    long long cap = (long long)sms * (per_sm < 2 ? per_sm : 2);
    if (cap > kFoldCap) cap = kFoldCap;  // partials one fold can take
    f->grid = (int)(need < cap ? need : cap);
    if (e == cudaSuccess) pick_tile(f, sms);
    if (e == cudaSuccess && f->tiles > 0)
      e = cudaFuncSetAttribute(k_bicgstab_tile, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kTileSmem);
  }
  al((void**)&f->part, 4 * (size_t)(f->grid > 0 ? f->grid : 1) * sizeof(double));
  if (e == cudaSuccess) e = cudaMallocHost((void**)&f->pinned, sizeof(Outcome));
  if (f->tiles > 0) {
    f->tagged_b = 2 * ((size_t)f->tiles * kTileSlot + (size_t)n) * sizeof(ulonglong2);
    al((void**)&f->tagged, f->tagged_b);
    if (e == cudaSuccess) e = cudaMemsetAsync(f->tagged, 0, f->tagged_b, f->stream);
  }
  al((void**)&f->sc, sizeof(Scal));
  al((void**)&f->iters, sizeof(int));
  al((void**)&f->bar, 2 * sizeof(unsigned));
  al((void**)&f->status, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(f->bar, 0, 2 * sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(f->status, 0, sizeof(int));
  if (e != cudaSuccess) {
    fem_free(f);
    return ctx_fail(LBM_ERR_NOMEM, "lbm_fem_init: %s", cudaGetErrorString(e));
  }
  double* v = f->vecs;
  f->w = Vec{v, v + n, v + 2 * n, v + 3 * n, v + 4 * n, v + 5 * n, v + 6 * n, v + 7 * n, v + 8 * n};
  const lbm_status st = fem_setup(f, elem_active, dir_nodes, d0);
  if (st != LBM_OK) {
    fem_free(f);
    return st;
  }
  *out = f;
  return LBM_OK;
}

lbm_status lbm_fem_step(lbm_fem* f, const double* dir_values) {
  if (!f) return ctx_fail(LBM_ERR_ARG, "lbm_fem_step: null solver");
  if (f->n_dir > 0 && !dir_values) return ctx_fail(LBM_ERR_ARG, "lbm_fem_step: null values");
  cudaStream_t s = f->stream;
  const double* fixed = f->fixed_val;
  if (f->n_dir > 0) {
    if (ctx_in_reach(dir_values, f->device)) fixed = dir_values;  // read in place: this call waits
    else FCK(cudaMemcpyAsync(f->fixed_val, dir_values, f->n_dir * sizeof(double),
                             cudaMemcpyDefault, s));
  }
  Outcome& h = *f->pinned;
  h = Outcome{};
  if (f->tiles > 0) {
    // a solve makes at most 3 exchanges an iteration and one before the first
    const unsigned long long span = 3ull * (unsigned)f->p.max_iter + 8;
    if (f->epoch + span > 0xFFFFFFFFull) {  // tags about to repeat: start over
      FCK(cudaMemsetAsync(f->tagged, 0, f->tagged_b, s));
      f->epoch = 1;
    }
    ulonglong2* pub = f->tagged + 2 * (size_t)f->tiles * kTileSlot;
    TileSolve T{f->A, f->invd, f->B, f->d, f->w.x, f->fixed_id, fixed, pub, pub + f->n, f->tagged,
                f->pinned, f->nxn, f->nyn, f->tw, f->th, (f->nxn + f->tw - 1) / f->tw, f->epoch,
                f->p.tol, f->p.max_iter, f->warm ? 1 : 0};
    f->epoch += (unsigned)(span < 0x7FFFFFFFull ? span : 0x7FFFFFFFull);
    void* args[] = {&T};
    FCK(cudaLaunchCooperativeKernel((const void*)k_bicgstab_tile, dim3(f->tiles), dim3(kTileThreads),
                                    args, f->tile_smem, s));
    FCK(cudaGetLastError());
    FCK(cudaStreamSynchronize(s));
  } else {
    Solve S;
    S.A = f->A;
    S.invd = f->invd;
    S.B = f->B;
    S.d = f->d;
    S.fixed_id = f->fixed_id;
    S.fixed_val = fixed;
    S.b = f->b;
    S.w = f->w;
    S.part = f->part;
    S.bar = f->bar;
    S.status = f->status;
    S.sc = f->sc;
    S.iters = f->iters;
    S.nxn = f->nxn;
    S.nyn = f->nyn;
    S.n = f->n;
    S.tol = f->p.tol;
    S.max_iter = f->p.max_iter;
    S.warm = f->warm ? 1 : 0;
    void* args[] = {&S};
    FCK(cudaLaunchCooperativeKernel((const void*)k_bicgstab, dim3(f->grid), dim3(kThreads), args,
                                    0, s));
    FCK(cudaGetLastError());
    FCK(cudaMemcpyAsync(&h.sc, f->sc, sizeof(Scal), cudaMemcpyDeviceToHost, s));
    FCK(cudaMemcpyAsync(&h.iters, f->iters, sizeof(int), cudaMemcpyDeviceToHost, s));
    FCK(cudaMemcpyAsync(&h.status, f->status, sizeof(int), cudaMemcpyDeviceToHost, s));
    FCK(cudaStreamSynchronize(s));
  }
  f->last_iters = h.iters;
  f->last_resid = h.sc.bnorm2 > 0 ? std::sqrt(h.sc.rnorm2 / h.sc.bnorm2) : std::sqrt(h.sc.rnorm2);
  f->warm = !h.status && h.sc.done;
  if (h.status) {
    cudaMemsetAsync(f->status, 0, sizeof(int), s);
    cudaMemsetAsync(f->bar, 0, 2 * sizeof(unsigned), s);
    return ctx_fail(LBM_ERR_TIMEOUT, "lbm_fem_step: a grid barrier wait of the solve expired");
  }
  if (h.sc.breakdown && !h.sc.done)
    return ctx_fail(LBM_ERR_STATE, "lbm_fem_step: BiCGSTAB broke down (relative residual %.3e)",
                    f->last_resid);
  if (!h.sc.done)
    return ctx_fail(LBM_ERR_STATE, "lbm_fem_step: no convergence in %d iterations (residual %.3e)",
                    f->p.max_iter, f->last_resid);
  return LBM_OK;
}

lbm_status lbm_fem_interpolate(lbm_fem* f, int npts, const double* xy, double* out) {
  if (!f || npts < 0 || (npts > 0 && (!xy || !out)))
    return ctx_fail(LBM_ERR_ARG, "lbm_fem_interpolate: bad arguments");
  if (npts == 0) return LBM_OK;
  cudaStream_t s = f->stream;
  const bool xy_dev = ctx_on_device(xy), out_dev = ctx_on_device(out);
  const double* dxy = xy;
  double* dout = out;
  double* tmp = nullptr;
  if (!xy_dev || !out_dev) {
    if (f->scratch_n < 3 * (size_t)npts) {
      FCK(cudaStreamSynchronize(s));
      if (f->scratch) cudaFree(f->scratch);
      f->scratch = nullptr;
      f->scratch_n = 0;
      FCK(cudaMalloc((void**)&f->scratch, 3 * (size_t)npts * sizeof(double)));
      f->scratch_n = 3 * (size_t)npts;
    }
    tmp = f->scratch;
    if (!xy_dev) {
      FCK(cudaMemcpyAsync(tmp, xy, 2 * (size_t)npts * sizeof(double), cudaMemcpyHostToDevice, s));
      dxy = tmp;
    }
    if (!out_dev) dout = tmp + 2 * (size_t)npts;
  }
  const lbm_fem_params& p = f->p;
  k_interp<<<(npts + 127) / 128, 128, 0, s>>>(f->d, p.nex, p.ney, p.x0, p.y0, p.hx, p.hy, dxy,
                                               npts, dout);
  FCK(cudaGetLastError());
  if (!out_dev) FCK(cudaMemcpyAsync(out, dout, (size_t)npts * sizeof(double), cudaMemcpyDeviceToHost, s));
  if (tmp) FCK(cudaStreamSynchronize(s));
  return LBM_OK;
}

lbm_status lbm_fem_get(lbm_fem* f, double* d) {
  if (!f || !d) return ctx_fail(LBM_ERR_ARG, "lbm_fem_get: null argument");
  FCK(cudaMemcpyAsync(d, f->d, f->n * sizeof(double), cudaMemcpyDefault, f->stream));
  if (!ctx_on_device(d)) FCK(cudaStreamSynchronize(f->stream));
  return LBM_OK;
}

lbm_status lbm_fem_set(lbm_fem* f, const double* d) {
  if (!f || !d) return ctx_fail(LBM_ERR_ARG, "lbm_fem_set: null argument");
  FCK(cudaMemcpyAsync(f->d, d, f->n * sizeof(double), cudaMemcpyDefault, f->stream));
  if (!ctx_on_device(d)) FCK(cudaStreamSynchronize(f->stream));
  return LBM_OK;
}

lbm_status lbm_fem_solver_info(lbm_fem* f, int* iters, double* rel_resid) {
  if (!f) return ctx_fail(LBM_ERR_ARG, "lbm_fem_solver_info: null solver");
  if (iters) *iters = f->last_iters;
  if (rel_resid) *rel_resid = f->last_resid;
  return LBM_OK;
}

void lbm_fem_destroy(lbm_fem* f) {
  if (!f) return;
  cudaStreamSynchronize(f->stream);
  fem_free(f);
}

}  // extern "C"
