// rbf.cu -- interface interpolation of stage two in three dimensions (Sec.
// 2.1, Fig. 2.2; pdd_interface_interp): per plane, a radial basis function
// interpolant with the cubic kernel |r|^3 and a linear polynomial term through
// the plane's nodes and n_bnd points per edge of the plane's perimeter, where
// the boundary data g are known.  The saddle-point system
//   [Phi P; P^T 0] [w; c] = [v; 0],  Phi_ij = |x_i - x_j|^3,  P_i = (1, s_i, t_i)
// is solved in FP64 by Gaussian elimination with partial pivoting, then
// evaluated at the query points.
//
// What bounds it: the FP64 pipe (1/64 rate: 2 lanes per clock and SM).  On the
// 9 planes of the 4096-node workload (M about 590) the elimination needs
// 6.0e8 multiply-adds (1.0 ms on all 152 SMs) and the evaluation at 9 x 129^2
// points 8.7e7 kernel values (1.4 ms at ten FP64 instructions each).
//
// Elimination.  Right-looking in panels of NB columns over the list of rows
// that have not been a pivot yet (rows are not moved).  Two launches per panel:
//   1. rbf_step_kernel<..., kNext>: the columns of the next panel are updated
//      by the current one, and the pivot rows' entries of all columns formed;
//   2. rbf_step_kernel<..., kRest>: one block per plane factors the next panel
//      (pivot search, multipliers) while the other blocks update all the
//      columns behind it by the current panel.
// So the serial pivot chain of a panel runs beside the update, which spreads
// over the whole GPU.  Every matrix element sees the same multiply-adds in
// the same order as in the plain row-by-row elimination (one FMA per step in
// step order, l = a / pivot), whatever the panel width.  A factored row stays where
// it is in A, with the list of the pivot rows beside (perm); only its entries in the
// panel after its own go aside: the blocks of launch 1 that update that panel all
// form them for themselves, so none may overwrite them in A.
//
// Measured on the 9 planes (device time): 11.75 ms by one 8-block cluster per
// plane with a cluster barrier per step (20 us a step); 2.2 ms in panels (step
// launches 109 us at the first panel, where the update bounds them, to 23 us at
// the last ones, where the 16 pivot steps do) and 0.25 ms of back
// substitution.  Evaluation 2.28 -> 1.56 ms (its FP64 floor is 1.4 ms).
#include <cmath>
#include <cstring>
#include <vector>

#include "ctx.hpp"
#include "models.cuh"

namespace pdd {

constexpr int64_t kRbfMaxSystem = 6144;  // unknowns per plane (weights + 3)
constexpr int kRbfThreads = 512;
constexpr int kRbfTileR = 32, kRbfTileC = 32;  // rows and columns of an update tile
constexpr size_t kRbfOwnSm = 116 * 1024;  // more than half of an SM's shared memory
constexpr size_t kRbfBackBytes = sizeof(double) + sizeof(int32_t);  // shared memory of a row in the back substitution
constexpr size_t kRbfPanelBytes = 200 * 1024;  // panel in shared memory (rows x NB doubles)

struct RbfPlane {
  int64_t node0, m;      // this plane's nodes: [node0, node0 + m) of the call's list
  int64_t sys0;          // offset of its system A (M rows of M + 1: the matrix, then the right-hand side)
  int64_t row0;          // offset of its rows in the per-row arrays (M of them)
  int64_t pts0;          // offset of its 2-D points (M - 3 of them) and values
  int64_t q0, q;         // its query points
  int32_t axis, M;       // plane normal axis; system size
  double pos;
};

// Scratch of the elimination (device pointers, all planes).
struct RbfWork {
  const RbfPlane *planes;
  int32_t n_planes;
  double *A;             // systems, row-major, M x (M + 1) each
  double *side;          // pivot rows' entries in the panel after their own [row0 + step][NB]
  int32_t *perm;         // pivot rows in step order [row0 + step]
  double *x;             // solutions [row0 + k]
  double *L[2];          // multipliers of the active rows, by panel parity: [row0 + pos][NB]
  int32_t *act[2];       // active rows (not yet a pivot) after a panel, by parity: [row0 + pos]
  double *L11[2];        // per plane: multipliers of the panel's pivot rows [NB][NB]
  int32_t *piv[2];       // per plane: the panel's pivot rows [NB]
  int *singular;
};

// sqrt of r2 >= 0 in FP64 by Heron's iteration from a binary32 seed: the
// hardware reciprocal square root y of r2 cut to a float gives s0 = r2 y and
// h = y / 2 (20 bits kept, in the high words), and two corrections
// s <- s + (r2 - s^2) h (the residual exact by FMA) reach the last bit: the
// relative error goes 2^-20 -> 2^-39 -> below 2^-58 before the final rounding
// (0.504 units in the last place at most over 2^21 numbers of any exponent).  Four FP64 instructions, where the library's square root takes several times
// that on this 1/64-rate pipe.  Outside [2^-100, 2^100) (a query on a point,
// far-away points) the library function.
__device__ __forceinline__ double sqrt_r2(double r2) {
  const int hi = __double2hiint(r2);
  if (static_cast<unsigned>(hi - (923 << 20)) >= (200u << 20)) return sqrt(r2);
  // the high word's 11-bit exponent rebiased to 8 bits, 20 mantissa bits kept
  const float f = __int_as_float((hi - (896 << 20)) << 3);
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const double s0 = __hiloint2double((__float_as_int(f * y) >> 3) + (896 << 20), 0);
  const double h = __hiloint2double((__float_as_int(0.5f * y) >> 3) + (896 << 20), 0);
  const double s1 = fma(fma(-s0, s0, r2), h, s0);
  return fma(fma(-s1, s1, r2), h, s1);
}

// The plane's two in-plane coordinates of a 3-D point.
__device__ __forceinline__ void plane_coords(int axis, const double *x, double &s, double &t) {
  s = x[axis == 0 ? 1 : 0];
  t = x[axis == 2 ? 1 : 2];
}

// Interpolation points of every plane: its nodes, then n_bnd points per edge
// of its perimeter (corners once) with the boundary data g.
template <class Model>
__global__ void rbf_points_kernel(const RbfPlane *planes, int32_t n_planes, const double *nodes,
                                  const double *vals, int32_t n_bnd, ModelConst mc, double *pts,
                                  double *pv) {
  const int p = blockIdx.y;
  if (p >= n_planes) return;
  const RbfPlane P = planes[p];
  const int64_t npt = P.M - 3;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < npt;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    double s, t, v;
    if (i < P.m) {
      plane_coords(P.axis, nodes + 3 * (P.node0 + i), s, t);
      v = vals[P.node0 + i];
    } else {
      // perimeter of the unit square in (s, t): edge e, point k of n_bnd
      const int64_t b = i - P.m;
      const int e = static_cast<int>(b / n_bnd);
      const double u = static_cast<double>(b % n_bnd) / n_bnd;
      s = e == 0 ? u : (e == 1 ? 1.0 : (e == 2 ? 1.0 - u : 0.0));
      t = e == 0 ? 0.0 : (e == 1 ? u : (e == 2 ? 1.0 : 1.0 - u));
      double x[3];
      x[P.axis] = P.pos;
      x[P.axis == 0 ? 1 : 0] = s;
      x[P.axis == 2 ? 1 : 2] = t;
      v = Model::template g<double>(mc, x);
    }
    pts[2 * (P.pts0 + i)] = s;
    pts[2 * (P.pts0 + i) + 1] = t;
    pv[P.pts0 + i] = v;
  }
}

// The systems (matrix and right-hand side in one row), the first list of
// active rows: all of them.
__global__ void rbf_assemble_kernel(RbfWork W, const double *pts, const double *pv) {
  const RbfPlane P = W.planes[blockIdx.y];
  const int M = P.M, ld = M + 1, npt = M - 3;
  double *A = W.A + P.sys0;
  const double *xy = pts + 2 * P.pts0;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
       e < static_cast<int64_t>(M) * ld; e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int i = static_cast<int>(static_cast<uint32_t>(e) / static_cast<uint32_t>(ld));
    const int j = static_cast<int>(e) - i * ld;
    double a;
    if (j == M) {
      a = i < npt ? pv[P.pts0 + i] : 0.0;
      W.act[1][P.row0 + i] = i;
    } else if (i < npt && j < npt) {
      const double ds = xy[2 * i] - xy[2 * j], dt = xy[2 * i + 1] - xy[2 * j + 1];
      const double r2 = ds * ds + dt * dt;
      a = r2 * sqrt_r2(r2);
    } else if (i < npt) {
      a = j == npt ? 1.0 : xy[2 * i + (j - npt - 1)];
    } else if (j < npt) {
      a = i == npt ? 1.0 : xy[2 * j + (i - npt - 1)];
    } else {
      a = 0.0;
    }
    A[e] = a;
  }
}

// 1 / b to 20 bits for 2^-500 < |b| < 2^500: the hardware reciprocal of the
// mantissa (20 bits of it, from the high word), the exponent negated in
// integers.  No FP64 instruction.
__device__ __forceinline__ double rcp_seed(double b) {
  const int hi = __double2hiint(b);
  const float m = __int_as_float(((hi & 0xfffff) << 3) | 0x3f800000);  // in [1, 2)
  const int y = __float_as_int(rcp_approx(m)) >> 3;                    // exponent 126 or 127
  const int e = (hi >> 20) & 0x7ff;
  return __hiloint2double((y + ((1023 - 127 + 1023 - e) << 20)) | (hi & 0x80000000), 0);
}
// a / b from r = rcp_seed(b): the quotient corrected twice by its exact
// remainder (FMA), 20 -> 40 -> 53 bits: 0.505 units in the last place at most.
// Five FP64 instructions and no serial reciprocal, where a division takes several
// times that.  (The interpolant's error against extended precision is no larger
// than with divisions and library roots throughout: 0.92 of it in the geometric
// mean over 14 planes of some 590 unknowns, 0.5 to 1.5 from one to the next.)
__device__ __forceinline__ double seeded_div(double a, double b, double r) {
  double q = a * r;
  q = fma(fma(-q, b, a), r, q);
  return fma(fma(-q, b, a), r, q);
}
// v / d from the rounded reciprocal r = 1 / d: corrected once.
__device__ __forceinline__ double back_quotient(double v, double d, double r) {
  return fma(fma(-v * r, d, v), r, v * r);
}
__device__ __forceinline__ bool seed_range(double b) {
  return fabs(b) > 0x1p-500 && fabs(b) < 0x1p500;
}

// Shared memory of an update tile: pivot rows and multipliers.
__host__ __device__ constexpr int rbf_tile_doubles(int NB) {
  return NB * kRbfTileC + kRbfTileR * (NB + 1);
}

// Named barriers of a step block: kRbfThreads workers and the pivot warp.
__device__ __forceinline__ void bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
enum { kBarCand = 1, kBarPivot = 2, kBarWork = 3 };

// Factor panel `panel` of a plane (columns [k0, k0 + nb)): one block.  The
// active rows' panel entries sit in shared memory, column by column; worker t
// owns the list positions t, t + 512, ...  Each step takes the unused row of
// largest |entry| (lowest row index on ties), forms the multipliers of the
// other unused rows and updates their remaining panel entries.  The chain from
// one pivot to the next is what bounds the panel (an FP64 instruction occupies
// its scheduler's pipe for 64 clocks), so a step first does only what the next
// pivot needs, the multipliers and the next column, and publishes the next
// column's candidates; while the extra warp picks the pivot (integers only: an
// FP64 reciprocal there would queue behind the workers' updates), the workers
// update the columns behind.  On return the list
// of rows still active, their multipliers, the pivot rows and their own
// multipliers are stored for the update, and A has the panel's columns of the
// pivot rows.
template <int NB>
__device__ void rbf_factor_panel(const RbfWork &W, const RbfPlane &P, int panel, double *smem) {
  const int k0 = panel * NB;
  const int M = P.M, ld = M + 1;
  if (k0 >= M) return;
  const int nb = min(NB, M - k0);
  const int R = M - k0;  // active rows before this panel
  const int par = panel & 1;
  const int32_t *act = W.act[par ^ 1] + P.row0;
  double *A = W.A + P.sys0;
  double *S = smem;  // S[c * R + pos]
  constexpr int nw = kRbfThreads / 32, kAll = kRbfThreads + 32;
  __shared__ uint32_t c_hi[2][nw], c_lo[2][nw];
  __shared__ int32_t c_pos[2][nw];
  __shared__ int32_t s_piv[NB];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp == nw) {
    // the pivot warp: step kk's pivot from the workers' candidates
    for (int kk = 0; kk < nb; ++kk) {
      const int sl = kk & 1;
      bar_sync(kBarCand, kAll);
      const uint32_t hi = lane < nw ? c_hi[sl][lane] : 0u;
      const uint32_t mh = __reduce_max_sync(kFull, hi);
      unsigned who = __ballot_sync(kFull, hi == mh && lane < nw);
      if (__popc(who) > 1) {  // equal high words: the low words, then the position, decide
        const uint32_t lo = (who >> lane) & 1u ? c_lo[sl][lane] : 0u;
        const uint32_t ml = __reduce_max_sync(kFull, lo);
        const bool top = ((who >> lane) & 1u) && lo == ml;
        const int32_t pos = top ? c_pos[sl][lane] : 0x7fffffff;
        const int32_t mp = __reduce_min_sync(kFull, pos);
        who = __ballot_sync(kFull, top && pos == mp);
      }
      const int src = __ffs(who) - 1;
      // (some row is unused, so some key is not 0; the largest is 1 or 2 when all
      // their entries are NaN or zero: flagged, the solution is not used)
      if (lane == 0) {
        if (mh == 0u && c_lo[sl][src] <= 2u) *W.singular = 1;
        s_piv[kk] = c_pos[sl][src];
      }
      __syncwarp();
      bar_sync(kBarPivot, kAll);
    }
    return;
  }
  for (int e = tid; e < R * NB; e += kRbfThreads) {
    const int pos = e / NB, c = e % NB;
    if (c < nb) S[c * R + pos] = A[static_cast<int64_t>(act[pos]) * ld + k0 + c];
  }
  bar_sync(kBarWork, kRbfThreads);
  uint32_t used = 0;  // bit i: own position tid + 512 i has been a pivot
  // candidate of this thread: bits of |entry| plus two (1 for NaN, 0: no unused
  // row, so that the panel's pivots are distinct rows whatever the entries are)
  // and its position (the list keeps rows in increasing order, so the lowest
  // position is the lowest row)
  unsigned long long key = 0;
  int32_t kpos = 0x7fffffff;
  auto consider = [&](double v, int pos) {
    // (integers only: the FP64 pipe is what bounds the panel)
    const unsigned long long m =
        static_cast<unsigned long long>(__double_as_longlong(v)) & 0x7fffffffffffffffull;
    const unsigned long long b = m <= 0x7ff0000000000000ull ? m + 2 : 1ull;
    if (b > key) {
      key = b;
      kpos = pos;
    }
  };
  // warp candidate of step kk: largest key, then lowest position
  auto publish = [&](int kk) {
    const uint32_t hi = static_cast<uint32_t>(key >> 32), lo = static_cast<uint32_t>(key);
    const uint32_t mh = __reduce_max_sync(kFull, hi);
    unsigned who = __ballot_sync(kFull, hi == mh);
    if (__popc(who) > 1) {  // equal high words: the low words, then the position, decide
      const uint32_t ml = __reduce_max_sync(kFull, hi == mh ? lo : 0u);
      const bool top = hi == mh && lo == ml;
      const int32_t mp = __reduce_min_sync(kFull, top ? kpos : 0x7fffffff);
      who = __ballot_sync(kFull, top && kpos == mp);
    }
    if (lane == __ffs(who) - 1) {
      c_hi[kk & 1][warp] = mh;
      c_lo[kk & 1][warp] = lo;
      c_pos[kk & 1][warp] = kpos;
    }
    __threadfence_block();
    __syncwarp();
    bar_arrive(kBarCand, kAll);
  };
  for (int pos = tid; pos < R; pos += kRbfThreads) consider(S[pos], pos);
  publish(0);
  for (int kk = 0; kk < nb; ++kk) {
    bar_sync(kBarPivot, kAll);
    const int pr = s_piv[kk];
    const double akk = S[kk * R + pr];
    if (pr % kRbfThreads == tid) used |= 1u << (pr / kRbfThreads);
    const int ea = (__double2hiint(akk) >> 20) & 0x7ff;
    const bool seeded = ea > 523 && ea < 1523;  // |akk| in [2^-499, 2^500)
    const double r = rcp_seed(akk);
    const int c1 = kk + 1;
    const double p1 = c1 < nb ? S[c1 * R + pr] : 0.0;
    key = 0;
    kpos = 0x7fffffff;
    // (the pivot row's entries are read by every thread and written by none)
    for (int i = 0, pos = tid; pos < R; ++i, pos += kRbfThreads) {
      if ((used >> i) & 1u) continue;
      const double a = S[kk * R + pos];
      const double l = seeded ? seeded_div(a, akk, r) : a / akk;
      S[kk * R + pos] = l;
      if (c1 < nb) {
        const double v = fma(-l, p1, S[c1 * R + pos]);
        S[c1 * R + pos] = v;
        consider(v, pos);
      }
    }
    if (c1 < nb) publish(c1);
    for (int i = 0, pos = tid; pos < R; ++i, pos += kRbfThreads) {
      if ((used >> i) & 1u) continue;
      const double l = S[kk * R + pos];
#pragma unroll 4
      for (int c = kk + 2; c < nb; ++c)
        S[c * R + pos] = fma(-l, S[c * R + pr], S[c * R + pos]);
    }
  }
  bar_sync(kBarWork, kRbfThreads);
  // the panel's columns of the pivot rows in A, the list, their multipliers
  double *L11 = W.L11[par] + (blockIdx.x * NB) * NB;
  for (int e = tid; e < nb * nb; e += kRbfThreads) {
    const int i = e / nb, c = e % nb;
    const double v = S[c * R + s_piv[i]];
    if (c >= i) A[static_cast<int64_t>(act[s_piv[i]]) * ld + k0 + c] = v;
    else L11[i * NB + c] = v;
  }
  if (tid < nb) W.perm[P.row0 + k0 + tid] = W.piv[par][blockIdx.x * NB + tid] = act[s_piv[tid]];
  // rows still active keep their order: the new position is the old one less
  // the pivots before it
  int32_t *act2 = W.act[par] + P.row0;
  double *L = W.L[par] + P.row0 * NB;
  for (int i = 0, pos = tid; pos < R; ++i, pos += kRbfThreads) {
    if ((used >> i) & 1u) continue;
    int np = pos;
    for (int c = 0; c < nb; ++c) np -= s_piv[c] < pos ? 1 : 0;
    act2[np] = act[pos];
    for (int c = 0; c < nb; ++c) L[static_cast<int64_t>(np) * NB + c] = S[c * R + pos];
  }
}

// The pivot rows' entries of panel `panel` in the TC columns from column c0
// (below c1): a unit lower triangular solve, a warp per pivot row and a lane
// per column, so that the triangle spreads over the four schedulers' FP64
// pipes.  The result is left in Us [NB][TC] and stored: kSide, the columns of the
// panel after it, aside (by the block that is to, `store`); else in place.
template <int NB, int TC, bool kSide>
__device__ void rbf_pivot_rows(const RbfWork &W, const RbfPlane &P, int plane, int panel, int c0,
                               int c1, double *Us, double *L11, bool store) {
  const int k0 = panel * NB, ld = P.M + 1;
  const int nb = min(NB, P.M - k0);
  const int par = panel & 1, tid = threadIdx.x;
  const int i = tid >> 5, c = tid & 31;
  const bool on = i < nb && c < TC && c0 + c < c1;
  double ui = 0.0;
  double *const at = W.A + P.sys0 + static_cast<int64_t>(on ? W.piv[par][plane * NB + i] : 0) * ld + c0 + c;
  if (on) ui = *at;
  for (int e = tid; e < NB * NB; e += kRbfThreads) {
    const int row = e / NB, k = e % NB;
    L11[e] = k < row && row < nb ? W.L11[par][plane * NB * NB + e] : 0.0;
  }
  bar_sync(kBarWork, kRbfThreads);
#pragma unroll
  for (int k = 0; k < NB; ++k) {
    if (i == k && c < TC) Us[k * TC + c] = ui;
    bar_sync(kBarWork, kRbfThreads);
    if (i > k && on) ui = fma(-L11[i * NB + k], Us[k * TC + c], ui);
  }
  if (on && store) {
    if constexpr (kSide) W.side[(P.row0 + k0 + i) * NB + c] = ui;
    else *at = ui;
  }
}

// Update by panel `panel` (already factored, the pivot rows' entries Us
// [NB][TC]) of a tile of TC columns from column c0 (below c1) and TR active
// rows from position r0: one FMA per element and pivot, in pivot order.
// Threads tid of kRbfThreads; Ls: [TR][NB + 1] of shared memory.  mid() runs once
// the tile's own loads are under way, sync() before Us and Ls are read.
template <int NB, int TC, int TR, class Mid, class Sync>
__device__ void rbf_update_tile(const RbfWork &W, const RbfPlane &P, int panel, int r0, int c0,
                                int c1, const double *Us, double *Ls, int tid, Mid mid, Sync sync) {
  const int k0 = panel * NB, ld = P.M + 1;
  const int nb = min(NB, P.M - k0);
  const int R = P.M - k0 - nb;
  const int par = panel & 1;
  double *A = W.A + P.sys0;
  const int rows = min(TR, R - r0);
  const double *L = W.L[par] + (P.row0 + r0) * NB;
  const int32_t *act = W.act[par] + P.row0 + r0;
  const int tx = tid % TC, ty = tid / TC, j = c0 + tx;
  constexpr int kStep = kRbfThreads / TC;   // rows between a thread's own
  constexpr int kOwn = (TR + kStep - 1) / kStep;
  double a[kOwn];
  double *pa[kOwn];
#pragma unroll
  for (int q = 0; q < kOwn; ++q) {
    const int row = ty + q * kStep;
    pa[q] = row < rows && j < c1 ? A + static_cast<int64_t>(act[row]) * ld + j : nullptr;
    a[q] = pa[q] ? *pa[q] : 0.0;
  }
  mid();
  for (int e = tid; e < rows * NB; e += kRbfThreads)
    Ls[(e / NB) * (NB + 1) + e % NB] = e % NB < nb ? L[e] : 0.0;
  sync();
  double u[NB];
#pragma unroll
  for (int k = 0; k < NB; ++k) u[k] = Us[k * TC + tx];
#pragma unroll
  for (int q = 0; q < kOwn; ++q) {
    if (!pa[q]) continue;
    const double *l = Ls + (ty + q * kStep) * (NB + 1);
    double v = a[q];
#pragma unroll
    for (int k = 0; k < NB; ++k)
      if (k < nb) v = fma(-l[k], u[k], v);
    *pa[q] = v;
  }
}

// kFirst: panel 0 of every plane is factored (blockIdx.x = plane).
// kNext, blockIdx.y = plane: blocks [0, row_tiles) update the columns of panel
// + 1 by `panel` (the first stores the pivot rows' part); the others form the pivot
// rows' entries of 32 columns behind them.
// kRest: blocks [0, n_planes) factor panel + 1; the others update the columns
// behind it by `panel`, two tiles per block (tile index = (plane, row tile,
// column tile), column tiles fastest).  Launched with more than half of an
// SM's shared memory per block, so that a panel has its SM's FP64 pipe to
// itself.
enum { kFirst = 0, kNext = 1, kRest = 2 };
template <int NB, int kRole>
__global__ void __launch_bounds__(kRole == kNext ? kRbfThreads : kRole == kRest ? 2 * kRbfThreads
                                                                 : kRbfThreads + 32)
rbf_step_kernel(const __grid_constant__ RbfWork W, int panel, int row_tiles, int col_tiles) {
  extern __shared__ __align__(16) double rbf_smem[];
  constexpr int TC = kRbfTileC;
  static_assert(NB * 32 <= kRbfThreads, "a warp per pivot row");
  if constexpr (kRole == kFirst) {
    rbf_factor_panel<NB>(W, W.planes[blockIdx.x], 0, rbf_smem);
  } else if constexpr (kRole == kNext) {
    const RbfPlane P = W.planes[blockIdx.y];
    const int k0 = panel * NB;
    if (k0 >= P.M) return;
    const int R = P.M - k0 - min(NB, P.M - k0);
    double *L11 = rbf_smem, *Us = L11 + NB * NB, *Ls = Us + NB * TC;
    if (static_cast<int>(blockIdx.x) < row_tiles) {
      const int r0 = blockIdx.x * kRbfTileR, c0 = k0 + NB, c1 = min(k0 + 2 * NB, P.M);
      if (R <= 0 || r0 >= R) return;  // no next panel, or no such rows
      rbf_pivot_rows<NB, NB, true>(W, P, blockIdx.y, panel, c0, c1, Us, L11, blockIdx.x == 0);
      rbf_update_tile<NB, NB, kRbfTileR>(W, P, panel, r0, c0, c1, Us, Ls, threadIdx.x, [] {},
                                         [] { bar_sync(kBarWork, kRbfThreads); });
    } else {
      const int c0 = min(k0 + 2 * NB, P.M) + (blockIdx.x - row_tiles) * TC;
      if (c0 > P.M) return;
      rbf_pivot_rows<NB, TC, false>(W, P, blockIdx.y, panel, c0, P.M + 1, Us, L11, true);
    }
  } else {
    if (static_cast<int>(blockIdx.x) < W.n_planes) {
      if (threadIdx.x < kRbfThreads + 32)
        rbf_factor_panel<NB>(W, W.planes[blockIdx.x], panel + 1, rbf_smem);
      return;
    }
    // two independent tiles per block
    const int half = threadIdx.x / kRbfThreads, tid = threadIdx.x % kRbfThreads;
    int t = (blockIdx.x - W.n_planes) * 2 + half;
    const int ct = t % col_tiles;
    t /= col_tiles;
    const int rt = t % row_tiles, p = t / row_tiles;
    if (p >= W.n_planes) return;
    const RbfPlane P = W.planes[p];
    const int k0 = panel * NB, ld = P.M + 1;
    const int r0 = rt * kRbfTileR, c0 = min(k0 + 2 * NB, P.M) + ct * TC;
    if (k0 + NB >= P.M || r0 >= P.M - k0 - NB || c0 > P.M) return;
    double *Us = rbf_smem + half * rbf_tile_doubles(NB), *Ls = Us + NB * TC;
    // the pivot rows' entries, one per thread, loaded beside the tile's rows
    static_assert(NB * TC <= kRbfThreads, "one entry per thread");
    const int uj = c0 + tid % TC;
    const bool has_u = tid < NB * TC && uj <= P.M;
    const int32_t upiv = has_u ? W.piv[panel & 1][p * NB + tid / TC] : 0;
    double u = 0.0;
    const int bar = kBarWork + half;
    rbf_update_tile<NB, TC, kRbfTileR>(W, P, panel, r0, c0, P.M + 1, Us, Ls, tid,
                                       [&] {
                                         if (has_u) u = W.A[P.sys0 + static_cast<int64_t>(upiv) * ld + uj];
                                       },
                                       [&] {
                                         if (tid < NB * TC) Us[tid] = u;
                                         bar_sync(bar, kRbfThreads);
                                       });
  }
}

// Back substitution, one block per plane, from the last rows up in blocks of
// 32: one warp solves the 32 x 32 triangle (a lane per row; the 32 reciprocals
// formed together, the quotient corrected once by its exact remainder), then
// every row above
// subtracts the block's 32 columns, one thread per row.
template <int NB>
__global__ void __launch_bounds__(kRbfThreads) rbf_backsub_kernel(const __grid_constant__ RbfWork W) {
  extern __shared__ __align__(16) double rbf_smem[];
  const RbfPlane P = W.planes[blockIdx.x];
  const int M = P.M, ld = M + 1;
  const double *A = W.A + P.sys0, *side = W.side + P.row0 * NB;
  // step k's row of the triangular factor, column j >= k
  auto u_at = [&](int k, const double *row, int j) {
    const int s = j - (k / NB + 1) * NB;
    const double *at = s >= 0 && s < NB ? side + static_cast<int64_t>(k) * NB + s : row + j;
    return *at;
  };
  double *y = rbf_smem;        // M
  int32_t *perm = reinterpret_cast<int32_t *>(y + M);
  __shared__ double T[32][33];
  const int tid = threadIdx.x, lane = tid & 31;
  for (int k = tid; k < M; k += kRbfThreads) {
    const int32_t row = W.perm[P.row0 + k];
    perm[k] = row;
    y[k] = A[static_cast<int64_t>(row) * ld + M];
  }
  for (int b1 = M; b1 > 0;) {
    const int b0 = max(0, b1 - 32), nb = b1 - b0;
    __syncthreads();
    for (int e = tid; e < nb * nb; e += kRbfThreads) {
      const int i = e / nb, c = e % nb;
      if (c >= i) T[i][c] = u_at(b0 + i, A + static_cast<int64_t>(perm[b0 + i]) * ld, b0 + c);
    }
    __syncthreads();
    if (tid < 32) {
      const double d = lane < nb ? T[lane][lane] : 1.0;
      const double r = 1.0 / d;
      const bool seeded = seed_range(d);
      double v = lane < nb ? y[b0 + lane] : 0.0;
      for (int i = nb - 1; i >= 0; --i) {
        const double q = seeded ? back_quotient(v, d, r) : v / d;
        const double xi = __shfl_sync(kFull, q, i);
        if (lane == i) v = xi;
        else if (lane < i) v = fma(-T[lane][i], xi, v);
      }
      if (lane < nb) y[b0 + lane] = v;
    }
    __syncthreads();
    for (int k = tid; k < b0; k += kRbfThreads) {
      const double *row = A + static_cast<int64_t>(perm[k]) * ld;
      double v = y[k];
#pragma unroll 8
      for (int c = 0; c < nb; ++c) v = fma(-u_at(k, row, b0 + c), y[b0 + c], v);
      y[k] = v;
    }
    b1 = b0;
  }
  __syncthreads();
  for (int k = tid; k < M; k += kRbfThreads) W.x[P.row0 + k] = y[k];
}

// The interpolant at the query points, kRbfQ of them per thread, points and
// weights staged through shared memory.  Ten FP64 instructions per (query,
// point) pair (the squared distance 4, its square root 4, two products): the
// FP64 pipe is the bound.
constexpr int kRbfQ = 2;
constexpr int kRbfEvalBlock = 128, kRbfEvalPts = 256;
__global__ void __launch_bounds__(kRbfEvalBlock)
rbf_eval_kernel(const __grid_constant__ RbfWork W, const double *__restrict__ pts,
                const double *__restrict__ query, double *__restrict__ out) {
  __shared__ double2 sxy[kRbfEvalPts];
  __shared__ double sw[kRbfEvalPts];
  const RbfPlane P = W.planes[blockIdx.y];
  const int npt = P.M - 3;
  const double *w = W.x + P.row0;
  const double2 *xy = reinterpret_cast<const double2 *>(pts) + P.pts0;
  for (int64_t base = static_cast<int64_t>(blockIdx.x) * (kRbfEvalBlock * kRbfQ); base < P.q;
       base += static_cast<int64_t>(gridDim.x) * (kRbfEvalBlock * kRbfQ)) {
    double s[kRbfQ], t[kRbfQ], acc[kRbfQ];
#pragma unroll
    for (int u = 0; u < kRbfQ; ++u) {
      const int64_t j = min(base + u * kRbfEvalBlock + threadIdx.x, P.q - 1);
      plane_coords(P.axis, query + 3 * (P.q0 + j), s[u], t[u]);
      acc[u] = w[npt] + w[npt + 1] * s[u] + w[npt + 2] * t[u];
    }
    for (int i0 = 0; i0 < npt; i0 += kRbfEvalPts) {
      const int n = min(kRbfEvalPts, npt - i0);
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += kRbfEvalBlock) {
        sxy[i] = xy[i0 + i];
        sw[i] = w[i0 + i];
      }
      __syncthreads();
#pragma unroll 2
      for (int i = 0; i < n; ++i) {
        const double2 p = sxy[i];
        const double wi = sw[i];
#pragma unroll
        for (int u = 0; u < kRbfQ; ++u) {
          const double ds = s[u] - p.x, dt = t[u] - p.y;
          const double r2 = ds * ds + dt * dt;
          acc[u] = fma(wi, r2 * sqrt_r2(r2), acc[u]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kRbfQ; ++u) {
      const int64_t j = base + u * kRbfEvalBlock + threadIdx.x;
      if (j < P.q) out[P.q0 + j] = acc[u];
    }
  }
}

// The launches of the elimination and the back substitution for panel width NB.
template <int NB>
static pdd_status rbf_launch(pdd_ctx *ctx, const RbfWork &W, int Mmax) {
  const size_t panel_smem = static_cast<size_t>(Mmax) * NB * sizeof(double);
  const size_t next_smem = (NB * NB + rbf_tile_doubles(NB)) * sizeof(double);
  auto *first = rbf_step_kernel<NB, kFirst>;
  auto *next = rbf_step_kernel<NB, kNext>;
  auto *rest = rbf_step_kernel<NB, kRest>;
  // (the limits belong to the kernels on the device, not to this call: constants,
  // so that a small system lowers nothing under another thread's elimination)
  PDD_CUDA_TRY(ctx, cudaFuncSetAttribute(first, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kRbfPanelBytes)));
  PDD_CUDA_TRY(ctx, cudaFuncSetAttribute(rest, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(std::max(kRbfPanelBytes, kRbfOwnSm))));
  const int panels = (Mmax + NB - 1) / NB;
  const unsigned np = static_cast<unsigned>(W.n_planes);
  first<<<np, kRbfThreads + 32, panel_smem, ctx->stream>>>(W, 0, 0, 0);
  for (int p = 0; p < panels; ++p) {
    // active rows of the largest plane after this panel, and the columns behind
    // the next one, the right-hand side included (smaller planes have fewer)
    const int left = std::max(0, Mmax - (p + 1) * NB);
    const int rt = (left + kRbfTileR - 1) / kRbfTileR;
    const int ct = (std::max(0, left - NB) + kRbfTileC) / kRbfTileC;
    next<<<dim3(static_cast<unsigned>(rt + ct), np), kRbfThreads, next_smem, ctx->stream>>>(W, p, rt, ct);
    if (left > 0) {
      // the block's shared memory: the next panel of the largest plane
      const size_t sm = std::max(kRbfOwnSm, static_cast<size_t>(left) * NB * sizeof(double));
      rest<<<np + (np * static_cast<unsigned>(rt * ct) + 1) / 2, 2 * kRbfThreads, sm, ctx->stream>>>(W, p, rt, ct);
    }
    PDD_CUDA_TRY(ctx, cudaGetLastError());
  }
  PDD_CUDA_TRY(ctx, cudaFuncSetAttribute(rbf_backsub_kernel<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kRbfMaxSystem * kRbfBackBytes)));
  rbf_backsub_kernel<NB><<<np, kRbfThreads, static_cast<size_t>(Mmax) * kRbfBackBytes, ctx->stream>>>(W);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  return PDD_OK;
}

pdd_status interface_interp_impl(pdd_ctx *ctx, int32_t n_planes, const int32_t *h_axis,
                                 const double *h_pos, const int64_t *h_node_count,
                                 const double *d_nodes, const double *d_vals, int32_t n_bnd,
                                 const int64_t *h_query_count, const double *d_query,
                                 double *d_out, const int64_t *h_node_off) {
  if (ctx->prob.dim != 3 || ctx->prob.kind != PDD_PROB_ELLIPTIC_MANUFACTURED)
    return fail(ctx, PDD_EINVAL, "interface interpolation on planes covers the 3-D family");
  if (n_planes < 1 || n_planes > 64) return fail(ctx, PDD_EINVAL, "n_planes must be in [1, 64]");
  if (!h_axis || !h_pos || !h_node_count || !h_query_count)
    return fail(ctx, PDD_EINVAL, "null host array");
  if (n_bnd < 1 || n_bnd > 1024) return fail(ctx, PDD_EINVAL, "n_bnd must be in [1, 1024]");
  std::vector<RbfPlane> pl(static_cast<size_t>(n_planes));
  int64_t node0 = 0, sys0 = 0, row0 = 0, pts0 = 0, q0 = 0;
  int32_t Mmax = 0;
  for (int p = 0; p < n_planes; ++p) {
    if (h_axis[p] < 0 || h_axis[p] > 2) return fail(ctx, PDD_EINVAL, "axis must be 0, 1 or 2");
    if (!(h_pos[p] > 0.0 && h_pos[p] < 1.0)) return fail(ctx, PDD_EINVAL, "plane outside (0, 1)");
    if (h_node_count[p] < 0 || h_query_count[p] < 0) return fail(ctx, PDD_EINVAL, "negative count");
    const int64_t M = h_node_count[p] + 4LL * n_bnd + 3;
    if (M > kRbfMaxSystem) return fail(ctx, PDD_EINVAL, "plane %d: system of %lld unknowns above %lld",
                                       p, static_cast<long long>(M), static_cast<long long>(kRbfMaxSystem));
    RbfPlane &P = pl[p];
    P.node0 = h_node_off ? h_node_off[p] : node0;
    P.m = h_node_count[p];
    P.sys0 = sys0;
    P.row0 = row0;
    P.pts0 = pts0;
    P.q0 = q0;
    P.q = h_query_count[p];
    P.axis = h_axis[p];
    P.M = static_cast<int32_t>(M);
    P.pos = h_pos[p];
    node0 += P.m;
    sys0 += M * (M + 1);
    row0 += M;
    pts0 += M - 3;
    q0 += P.q;
    Mmax = std::max(Mmax, P.M);
  }
  if ((node0 > 0 && (!d_nodes || !d_vals)) || (q0 > 0 && (!d_query || !d_out)))
    return fail(ctx, PDD_EINVAL, "null buffer");
  if (q0 == 0) return PDD_OK;
  PDD_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  // the widest panel whose rows fit in one block's shared memory (16 columns
  // up to 1600 unknowns, 8 up to 3200, 4 up to the largest system)
  const int NB = static_cast<size_t>(Mmax) * 16 * sizeof(double) <= kRbfPanelBytes ? 16
               : static_cast<size_t>(Mmax) * 8 * sizeof(double) <= kRbfPanelBytes ? 8 : 4;
  static_assert(kRbfMaxSystem * 4 * sizeof(double) <= kRbfPanelBytes, "panel of the largest system");
  const size_t NP = static_cast<size_t>(n_planes);
  size_t o = 256;  // the singular flag
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align_up(o + bytes, 256);
    return at;
  };
  const size_t off_pl = take(pl.size() * sizeof(RbfPlane));
  const size_t off_pts = take(static_cast<size_t>(pts0) * 2 * sizeof(double));
  const size_t off_pv = take(static_cast<size_t>(pts0) * sizeof(double));
  const size_t off_A = take(static_cast<size_t>(sys0) * sizeof(double));
  const size_t off_side = take(static_cast<size_t>(row0) * NB * sizeof(double));
  const size_t off_perm = take(static_cast<size_t>(row0) * sizeof(int32_t));
  const size_t off_x = take(static_cast<size_t>(row0) * sizeof(double));
  size_t off_L[2], off_act[2], off_L11[2], off_piv[2];
  for (int h = 0; h < 2; ++h) {
    off_L[h] = take(static_cast<size_t>(row0) * NB * sizeof(double));
    off_act[h] = take(static_cast<size_t>(row0) * sizeof(int32_t));
    off_L11[h] = take(NP * NB * NB * sizeof(double));
    off_piv[h] = take(NP * NB * sizeof(int32_t));
  }
  pdd_status st = ensure_scratch(ctx, o);
  if (st != PDD_OK) return st;
  char *base = static_cast<char *>(ctx->scratch);
  auto *d_pl = reinterpret_cast<RbfPlane *>(base + off_pl);
  double *pts = reinterpret_cast<double *>(base + off_pts);
  double *pv = reinterpret_cast<double *>(base + off_pv);
  RbfWork W;
  W.planes = d_pl;
  W.n_planes = n_planes;
  W.A = reinterpret_cast<double *>(base + off_A);
  W.side = reinterpret_cast<double *>(base + off_side);
  W.perm = reinterpret_cast<int32_t *>(base + off_perm);
  W.x = reinterpret_cast<double *>(base + off_x);
  for (int h = 0; h < 2; ++h) {
    W.L[h] = reinterpret_cast<double *>(base + off_L[h]);
    W.act[h] = reinterpret_cast<int32_t *>(base + off_act[h]);
    W.L11[h] = reinterpret_cast<double *>(base + off_L11[h]);
    W.piv[h] = reinterpret_cast<int32_t *>(base + off_piv[h]);
  }
  W.singular = reinterpret_cast<int *>(base);
  PDD_CUDA_TRY(ctx, cudaMemsetAsync(base, 0, 256, ctx->stream));
  PDD_CUDA_TRY(ctx, cudaMemcpyAsync(d_pl, pl.data(), pl.size() * sizeof(RbfPlane),
                                    cudaMemcpyHostToDevice, ctx->stream));
  const dim3 g1(static_cast<unsigned>(std::min<int64_t>((Mmax + 255) / 256, 64)),
                static_cast<unsigned>(n_planes));
  rbf_points_kernel<EllipticManufactured><<<g1, 256, 0, ctx->stream>>>(
      d_pl, n_planes, d_nodes, d_vals, n_bnd, ctx->mc, pts, pv);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  const dim3 g2(static_cast<unsigned>(std::min<int64_t>((int64_t(Mmax) * Mmax + 255) / 256, 4096)),
                static_cast<unsigned>(n_planes));
  rbf_assemble_kernel<<<g2, 256, 0, ctx->stream>>>(W, pts, pv);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  st = NB == 16 ? rbf_launch<16>(ctx, W, Mmax)
     : NB == 8 ? rbf_launch<8>(ctx, W, Mmax)
               : rbf_launch<4>(ctx, W, Mmax);
  if (st != PDD_OK) return st;
  int64_t qmax = 0;
  for (const auto &P : pl) qmax = std::max(qmax, P.q);
  constexpr int64_t kPer = kRbfEvalBlock * kRbfQ;
  const dim3 g3(static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>((qmax + kPer - 1) / kPer, 65535))),
                static_cast<unsigned>(n_planes));
  rbf_eval_kernel<<<g3, kRbfEvalBlock, 0, ctx->stream>>>(W, pts, d_query, d_out);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  int hs = 0;
  PDD_CUDA_TRY(ctx, cudaMemcpyAsync(&hs, W.singular, sizeof hs, cudaMemcpyDeviceToHost, ctx->stream));
  PDD_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
  if (hs) return fail(ctx, PDD_EINVAL, "singular interpolation system (coincident nodes?)");
  return PDD_OK;
}

}  // namespace pdd
