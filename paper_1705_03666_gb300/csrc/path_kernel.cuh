// path_kernel.cuh -- the interface-node path kernel (stage one of PDD).
//
// One persistent launch advances every (node, path) of a wave of the global,
// node-major path index space g = node * n_paths + p.  Each lane owns one
// path at a time and takes the next one from its warp's stash of set-up paths
// (refilled 32 indices at a time from an atomic cursor), so no lane waits for
// a long path of another node and the only idle time is at the very end of
// the wave.  Scores are added at once to exact per-node integer sums
// (nodefix.cuh), so the per-node mean and standard error do not depend on
// which lane ran which path and no per-path score is stored.
//
// Per step (Eq. 2.8, Dirichlet/elliptic reduction of Sec. 2.2, left-point rule):
//   X' = X + b(X) dt + sigma sqrt(dt) xi,  Y' = Y e^{c(X) dt},  Z' = Z + f(X) Y dt,
// then the exit test: hard exit when X' leaves the closed domain (exit point =
// first crossing of the segment), else, with the bridge test, exit when
// U < P = 1 - prod_j (1 - exp(-2 d_j d'_j / (sigma^2 dt))) over faces with
// 2 d_j d'_j < 18 sigma^2 dt (exit point = X' projected on the face with the
// largest term).  P is accumulated without cancellation (bridge_exit) and
// near-ties of the FP32 path are decided in FP64.  Score = g(X_tau) Y' + Z'
// (Eq. 2.7).
//
// What bounds it: instruction issue (no contraction, next to no bytes), and
// with it the lanes that an instruction finds idle.  So the four steps of a
// unit run without a branch: a lane only notes whether any of them could have
// been an exit (fast_unit: one bound per step on the distance to the
// boundary, conservative against every test above).  A unit so noted is not
// taken: its start is parked, the lane takes another path, and the warp runs
// 32 parked units together, with the exact tests, all lanes busy
// (recheck_units).  Paths that exited there are scored at once; false alarms
// (about one per path) go back to the stash.
#pragma once

#include <cmath>

#include "common.cuh"
#include "models.cuh"
#include "nodefix.cuh"
#include "normal_tables.cuh"

namespace pdd {

// Threads per block of the forward path kernel, both precisions.  In binary32 ptxas
// gives 128-thread blocks 72 registers and the SM holds seven (28 warps); 256-thread
// blocks are held to 64 registers for four (32 warps): 840 against 836 ms on the 3-D
// solve when that was measured.
constexpr int kForwardBlock = 128;

struct PathArgs {
  const double *nodes;          // [n_nodes][D]
  uint64_t n_paths;             // paths per node
  uint64_t path_offset;         // first path index
  uint32_t node_offset;         // stream index of node 0 (node j draws node_offset + j)
  uint64_t begin, end;          // global index range of this launch (a wave)
  unsigned long long *cursor;   // queue cursor for this wave (starts at 0)
  unsigned long long *counters; // [0] path steps, [1] capped, [2] bad nodes
  NodeFix *fix;                 // forward mode: per-node exact sums [n_nodes]
  void *score;                  // gradient mode: GradRec[end - begin]
  double *dump_score;           // forward mode, optional: score per path [end - begin]
  double *dump_exit;            // forward mode, optional: exit point per path [end - begin][D]
  int32_t *steps;               // [end - begin] or null
  RoundKeys rk;
  double inv_s2dt;              // 1 / (sigma^2 dt)
  double dt_d, sdt_d, thr_d;    // FP64 path: dt, sigma sqrt(dt), 9 sigma^2 dt
  double ecdt_d;                // e^{c dt} for constant killing (FP64)
  float dt_f, sdt_f, thr_f;     // FP32 path
  float l2cdt_f;                // c dt log2(e) for constant killing (FP32)
  int32_t max_steps;
  int32_t bridge;
  float edge_c1, edge_c0;       // fast_unit's bound (see path_step_args)
  const double2 *normal_tables; // FP64 paths: NormalTables
  float lr_scale;               // sqrt(dt) / sigma (gradient mode)
  ModelConst mc;
};

// Constant killing: Y_n = e^{c n dt}.  Every path runs through the same
// sequence Y_0, Y_1, ..., so a rounded recurrence Y <- Y e^{c dt} would carry
// the same rounding error into every path (in binary32 it drifts by ~1e-5
// over 500 steps); the FP32 path therefore evaluates Y_n from n directly
// (exp2 of n c dt log2 e, a few ulp, no accumulation).  In FP64 the
// recurrence is accurate to n ulp and is kept.
// log2 of a face count (the union bound's factor), counts 1 .. 6.
constexpr float kLog2Count[7] = {0.0f, 0.0f, 1.0f, 1.5849625007211562f, 2.0f,
                                 2.321928094887362f, 2.584962500721156f};

// Step constants of a launch from dt, sigma, the killing rate and the bridge
// flag (host).  kReach: the most faces that can be within bridge reach of one
// step together.
//
// The bound of fast_unit (edge_bound).  With e a lower bound on the distance of a point to
// every face (Geom::edge; <= 0 outside), every d_j d'_j >= e e', so the step
// cannot cross while log2 U >= log2 kReach - 2 log2(e) e e' / (sigma^2 dt).
// log2 U is bounded below by the bits of U read as a fixed-point number
// (exponent and mantissa: at most 0.086 low), scaled by 2^15 and offset by
// 2^23: one byte permute.  So the test is
//   float(2^23 + bits(U) / 2^8) >= edge_c0 + edge_c1 e e',
// false also for e e' <= 0 (possible exit through the boundary) and for NaN.
// The margin covers the rounding of the exponents (2^-10 is over four times
// all of them), the near-tie window of the exact test and the rounding of e
// (2^-25 absolute, which weighs 2^-25 (e + e') 2.9 / (sigma^2 dt) with e, e'
// within 12 sigma sqrt(dt) where U can matter: below 2e-6 / (sigma sqrt(dt))).
// Without the bridge test the slope is -inf: only e e' <= 0 fails.
__host__ __device__ inline void edge_bound(double s, bool bridge, int kReach, float *c0, float *c1) {
  const double margin = 0x1p-10 + 4e-6 / s;  // s = sigma sqrt(dt)
  *c0 = static_cast<float>(8388608.0 + 32768.0 * (127.0 + log2(static_cast<double>(kReach)) + margin));
  *c1 = bridge ? static_cast<float>(-2.0 * 1.4426950408889634 * 32768.0 / (s * s)) : -INFINITY;
}
inline void path_step_args(PathArgs &a, double sig, double dt, double c_kill, bool bridge,
                           int kReach) {
  a.inv_s2dt = 1.0 / (sig * sig * dt);
  a.dt_d = dt;
  a.sdt_d = sig * std::sqrt(dt);
  a.thr_d = 9.0 * sig * sig * dt;
  a.ecdt_d = std::exp(c_kill * dt);
  a.dt_f = static_cast<float>(a.dt_d);
  a.sdt_f = static_cast<float>(a.sdt_d);
  a.thr_f = static_cast<float>(a.thr_d);
  a.l2cdt_f = static_cast<float>(c_kill * dt * 1.4426950408889634);
  a.bridge = bridge ? 1 : 0;
  edge_bound(a.sdt_d, bridge, kReach, &a.edge_c0, &a.edge_c1);
}

template <typename R> struct StepConst;
template <> struct StepConst<float> {
  float dt, sdt, thr, l2cdt, inv_s2dt;
  float b2;    // -2 log2(e) / (sigma^2 dt): exp(-2 m / (sigma^2 dt)) = 2^(b2 m)
  float boff;  // 0 with the bridge test, -inf without (every bound below is 0)
  float edge_c0, edge_c1;  // fast_unit's bound (edge_bound)
  StepConst() = default;
  __device__ __forceinline__ StepConst(const PathArgs &a)
      : dt(a.dt_f), sdt(a.sdt_f), thr(a.thr_f), l2cdt(a.l2cdt_f),
        inv_s2dt(static_cast<float>(a.inv_s2dt)),
        b2(static_cast<float>(-2.0 * 1.4426950408889634 * a.inv_s2dt)),
        boff(a.bridge ? 0.0f : -INFINITY), edge_c0(a.edge_c0), edge_c1(a.edge_c1) {}
  // half-space crossing probability for a step with d d' = m
  __device__ __forceinline__ float cross_p(float m) const { return ex2_approx(b2 * m); }
  // Bound on every crossing probability of a step whose smallest d d' over
  // D candidate faces is m: 1 - prod_j (1 - p_j) <= D p(m), raised by the
  // factor 2^(2^-12) = 1 + 1.7e-4, which covers the near-tie window (2^-18
  // relative) and the rounding of the exponents (< 1e-5 relative for the
  // probabilities above 2^-26 that a uniform can fall below).  0 without the
  // bridge test.
  template <int D> __device__ __forceinline__ float cross_bound(float m) const {
    constexpr float kOff = kLog2Count[D] + 2.44140625e-4f;
    return ex2_approx(fmaf(b2, m, kOff + boff));
  }
  __device__ __forceinline__ float kill(float, int32_t n_next) const {
    return ex2_approx(static_cast<float>(n_next) * l2cdt);
  }
  // the same for a step count held as a float (exact below 2^24)
  __device__ __forceinline__ float kill_f(float n_next) const { return ex2_approx(n_next * l2cdt); }
  // e^{-a} for a >= 0 (hardware exp2, ~2 ulp; a near-tie decision is redone
  // in FP64 by the caller).
  __device__ __forceinline__ float exp_neg(float a) const {
    return ex2_approx(-1.4426950408889634f * a);
  }
};
template <> struct StepConst<double> {
  double dt, sdt, thr, e, inv_s2dt;
  double boff;  // 0 with the bridge test, -inf without
  float edge_c0, edge_c1;
  __device__ __forceinline__ StepConst(const PathArgs &a)
      : dt(a.dt_d), sdt(a.sdt_d), thr(a.thr_d), e(a.ecdt_d), inv_s2dt(a.inv_s2dt),
        boff(a.bridge ? 0.0 : -INFINITY), edge_c0(a.edge_c0), edge_c1(a.edge_c1) {}
  __device__ __forceinline__ double kill(double y, int32_t) const { return y * e; }
  __device__ __forceinline__ double exp_neg(double a) const { return exp(-a); }
  __device__ __forceinline__ double cross_p(double m) const { return exp(-2.0 * m * inv_s2dt); }
  template <int D> __device__ __forceinline__ double cross_bound(double m) const {
    return static_cast<double>(D) * 1.0000001 * exp(boff - 2.0 * m * inv_s2dt);
  }
};

// FP32 step constants for time step dt, generator (1/2) sigma^2 Lap, a
// constant killing rate c and the bridge test on or off, rounded from the
// same FP64 expressions the host uses for PathArgs.
template <class Geom>
__device__ __forceinline__ StepConst<float> make_step_const(double dt, double sigma, double c,
                                                            bool bridge) {
  StepConst<float> k;
  k.dt = static_cast<float>(dt);
  k.sdt = static_cast<float>(sigma * sqrt(dt));
  k.thr = static_cast<float>(9.0 * sigma * sigma * dt);
  k.l2cdt = static_cast<float>(c * dt * 1.4426950408889634);
  k.inv_s2dt = static_cast<float>(1.0 / (sigma * sigma * dt));
  k.b2 = static_cast<float>(-2.0 * 1.4426950408889634 / (sigma * sigma * dt));
  k.boff = bridge ? 0.0f : -INFINITY;
  const double s = sigma * sqrt(dt);
  edge_bound(s, bridge, Geom::reach(s), &k.edge_c0, &k.edge_c1);
  return k;
}

// FP64 re-decision of a near tie of the 2-D box bridge test from the same
// binary32 products d_j d'_j, kept out of line: it almost never runs, and
// inlined its FP64 code enlarged the 2-D kernels enough to stall them on
// instruction fetch (the gradient pass 156 -> 121 ms once it moved out; the
// 3-D kernel measured faster with its three-face form inline, 850 against
// 857 ms).
static __device__ __noinline__ bool bridge_box2_tie(float U, float inv_s2dt, float p0, float p1) {
  const float pr[2] = {p0, p1};
  double Pd = 0.0;
  const double s = 2.0 * static_cast<double>(inv_s2dt);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const double aa = s * static_cast<double>(pr[c]);
    if (aa < 18.0) {
      const double p = exp(-aa);
      Pd = Pd + p * (1.0 - Pd);
    }
  }
  return static_cast<double>(U) < Pd;
}

// Brownian-bridge exit probability over the faces within reach,
// P = 1 - prod_j (1 - p_j), p_j = exp(-2 d_j d'_j / (sigma^2 dt)), accumulated
// as P <- P + p_j (1 - P) (no cancellation, so accurate for tiny P).  FP32
// path: compensated binary32, and a decision with |U - P| within 2^-18 P is
// re-taken from the same distances in FP64.  Returns the face with the
// largest p_j, or -1 when no face is within reach or U >= P.
template <int NC, typename R>
__device__ __forceinline__ int bridge_exit(const StepConst<R> &k, const R *prod, const int *face,
                                           R U) {
  R P = R(0), pbest = R(-1);
  int jbest = -1;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const R aa = R(2) * prod[c] * k.inv_s2dt;
    if (aa < R(18)) {
      const R p = k.exp_neg(aa);
      P = P + p * (R(1) - P);
      if (p > pbest) { pbest = p; jbest = face[c]; }
    }
  }
  if (jbest < 0) return -1;
  bool take = U < P;
  if constexpr (sizeof(R) == 4) {
    if (fabsf(U - P) <= 3.814697265625e-06f * P) {  // near tie: FP64 from the same products
      if constexpr (NC == 2) {
        take = bridge_box2_tie(U, k.inv_s2dt, prod[0], prod[1]);
      } else {
        double Pd = 0.0;
        const double s = 2.0 * static_cast<double>(k.inv_s2dt);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const double aa = s * static_cast<double>(prod[c]);
          if (aa < 18.0) {
            const double p = exp(-aa);
            Pd = Pd + p * (1.0 - Pd);
          }
        }
        take = static_cast<double>(U) < Pd;
      }
    }
  }
  return take ? jbest : -1;
}

// FP64 re-decision of a near tie of the general-domain bridge test, from the
// same binary32 face distances (kept out of line: it almost never runs, and
// inlined it put FP64 instructions into the step code of every warp that
// reaches the bridge test).  2-D geometries.
template <class Geom>
static __device__ __noinline__ bool bridge_generic_tie(float U, float inv_s2dt, float x0, float x1,
                                                       float xn0, float xn1) {
  const float X[2] = {x0, x1}, Xn[2] = {xn0, xn1};
  double Pd = 0.0;
  const double s = 2.0 * static_cast<double>(inv_s2dt);
#pragma unroll
  for (int j = 0; j < Geom::kFaces; ++j) {
    const double aa = s * static_cast<double>(Geom::face_dist(j, X) * Geom::face_dist(j, Xn));
    if (aa < 18.0) {
      const double p = exp(-aa);
      Pd = Pd + p * (1.0 - Pd);
    }
  }
  return static_cast<double>(U) < Pd;
}

// Bridge over all faces of a general domain (distances from Geom::face_dist):
// P = 1 - prod_j (1 - p_j) accumulated as P + p (1 - P) over the faces with
// 2 d d' / (sigma^2 dt) < 18; FP32 near-ties decided in FP64.  Returns the
// face with the largest p_j if U < P, else -1.
template <class Geom, typename R>
__device__ __forceinline__ int bridge_generic(const StepConst<R> &k, const R *X, const R *Xn, R U) {
  R P = R(0), pbest = R(-1);
  int jbest = -1;
#pragma unroll
  for (int j = 0; j < Geom::kFaces; ++j) {
    const R aa = R(2) * (Geom::face_dist(j, X) * Geom::face_dist(j, Xn)) * k.inv_s2dt;
    if (aa < R(18)) {
      const R p = k.exp_neg(aa);
      P = P + p * (R(1) - P);
      if (p > pbest) { pbest = p; jbest = j; }
    }
  }
  if (jbest < 0) return -1;
  bool take = U < P;
  if constexpr (sizeof(R) == 4) {
    static_assert(Geom::D == 2, "the out-of-line tie test takes 2-D points");
    if (fabsf(U - P) <= 3.814697265625e-06f * P)
      take = bridge_generic_tie<Geom>(U, k.inv_s2dt, X[0], X[1], Xn[0], Xn[1]);
  }
  return take ? jbest : -1;
}

// Number of likelihood-ratio accumulators carried per path (gradient mode).
constexpr int kMaxLR = 16;

// FP64 re-decision of a near tie U ~ exp(-2 m / (sigma^2 dt)) (kept out of
// line: it almost never runs and would otherwise be inlined at every step).
static __device__ __noinline__ bool bridge_tie_fp64(float U, float mn, float inv_s2dt) {
  return static_cast<double>(U) <
         exp(-2.0 * static_cast<double>(mn) * static_cast<double>(inv_s2dt));
}

// Exit codes of em_step.
constexpr int kStepContinue = -2;
constexpr int kStepHardExit = -1;   // >= 0: bridge exit through that face
// A path stopped by the step cap (set by callers): scored at the projection of
// its last point on the nearest face.
constexpr int kStepCapped = -3;

// One Euler-Maruyama step with the exit test.  On kStepContinue, X, Y, Z
// advance; on an exit, X keeps the start of the step, Xn receives its end,
// Y and Z receive their exit values, and the caller resolves the exit point
// (exit_score): the path kernel where it reruns parked units, the gradient kernel
// 32 paths at a time from its exit queue, the plain one through path_unit.  With
// kLR the drift-weight likelihood-ratio sums L are advanced by this step's noise
// (the exiting step included).
template <class Model, class Geom, typename R, bool kLR, class Env>
__device__ __forceinline__ int em_step(const Env &a, const StepConst<R> &k, R *X, R &Y, R &Z,
                                       const R *xi, uint32_t uw, int32_t n, R *Xn, R *L) {
  constexpr int D = Model::D;
  R b[D];
  R f = R(0);
#pragma unroll
  for (int d = 0; d < D; ++d) b[d] = R(0);
  if constexpr (kLR) {
    Model::coeffs_lr(a.mc, X, b, f, xi, L);
  } else if constexpr (Model::kDrift || Model::kSource) {
    Model::coeffs(a.mc, X, b, f);
  }
  // (an axis without drift skips b dt: X + 0 dt is X exactly, so the result
  // is the same)
#pragma unroll
  for (int d = 0; d < D; ++d) {
    if ((Model::kDriftAxes >> d) & 1u)
      Xn[d] = X[d] + b[d] * k.dt + k.sdt * xi[d];
    else
      Xn[d] = X[d] + k.sdt * xi[d];
  }
  R Zn = Z;
  if constexpr (Model::kSource) Zn = Z + f * Y * k.dt;
  R Yn = Y;
  if constexpr (Model::kKill == 1) Yn = k.kill(Y, n + 1);
  Y = Yn;
  Z = Zn;
  if constexpr (!Geom::kFastScreen) {
    // general domains: a lower bound on the smallest d d' (> 0: X' inside)
    // and the union bound over all faces screen the step; below the bound,
    // the exact tests (every face within reach, P = 1 - prod (1 - p_j))
    const R mnb = Geom::screen_lb(X, Xn);
    const R U = unif<R>(uw);
    if (!(mnb > R(0)) || U < k.template cross_bound<Geom::kFaces>(mnb)) {
      if (!Geom::inside_closed(Xn)) return kStepHardExit;
      if (a.bridge) {
        const int jbest = bridge_generic<Geom, R>(k, X, Xn, U);
        if (jbest >= 0) return jbest;
      }
    }
  } else {
    const R mn = Geom::screen_mn(X, Xn);
    // mn > 0 puts X' strictly inside.  U lies above every crossing
    // probability the step can have (and above its near-tie window) at most
    // steps: one bound decides that, and the probability itself is formed
    // only below it.  Both tests share one branch.
    const R U = unif<R>(uw);
    const R bnd = k.template cross_bound<D>(mn);
    if (!(mn > R(0)) || U < bnd) {
      if (!(mn > R(0)) && !Geom::inside_closed(Xn)) return kStepHardExit;
      if (U < bnd) {
        // A step within reach of one face crosses with
        // exp(-2 min d d' / (sigma^2 dt)); a step within reach of two or more
        // faces (an edge or a corner) takes the general combination.
        R prod[D];
        int face[D];
        Geom::screen(X, Xn, prod, face);
        bool cross;
        if (Geom::second_min(prod) < k.thr) {
          cross = bridge_exit<D, R>(k, prod, face, U) >= 0;
        } else {
          const R p = k.cross_p(mn);
          cross = U < p;
          if constexpr (sizeof(R) == 4) {
            if (fabsf(U - p) <= 3.814697265625e-06f * p) cross = bridge_tie_fp64(U, mn, k.inv_s2dt);
          }
        }
        if (cross) {
          int jbest = face[0];
          R pmin = prod[0];
#pragma unroll
          for (int d = 1; d < D; ++d)
            if (prod[d] < pmin) { pmin = prod[d]; jbest = face[d]; }
          return jbest;
        }
      }
    }
  }
#pragma unroll
  for (int d = 0; d < D; ++d) X[d] = Xn[d];
  return kStepContinue;
}

// Exit point of a step that left the domain (first crossing of X -> Xn) or
// crossed a face by the bridge (Xn projected on it), and the path's score
// g(X_tau) Y + Z (Eq. 2.7).
template <class Model, class Geom, typename R>
__device__ __forceinline__ R exit_score(const ModelConst &mc, int code, const R *X, const R *Xn,
                                        R Y, R Z, R *xe) {
  constexpr int D = Model::D;
  if (code == kStepHardExit) {
    Geom::segment_exit(X, Xn, xe);
  } else {
#pragma unroll
    for (int d = 0; d < D; ++d) xe[d] = Xn[d];
    Geom::project(code, xe);
  }
  return Model::g(mc, xe) * Y + Z;
}

// Word whose bytes 3, 2, 1 are the low bytes of c, b, a: the bridge uniform
// of a 3-D step comes from bits the Box-Muller maps (bits 9..31) do not use.
__device__ __forceinline__ uint32_t low_bytes_word(uint32_t a, uint32_t b, uint32_t c) {
  return __byte_perm(__byte_perm(a, b, 0x0400u), c, 0x4210u);
}

// Random numbers of the four-step unit that starts at step n = 4q: normals
// z[D j .. D j + D - 1] and the bridge-uniform word u[j] of step n + j, from
// the twelve words w0..w11 of Philox blocks 3q, 3q+1, 3q+2.  d <= 2: step
// 4q + j takes BM(w[2j], w[2j+1]) (d = 1: the first) and the uniform word
// w[8+j].  d = 3: normals z0..z11 = BM of the word pairs (w0,w1) ..
// (w10,w11), step 4q + j takes z[3j..3j+2] and low_bytes_word(w[3j],
// w[3j+1], w[3j+2]).  Either way 0.75 blocks per step, the least that holds
// the step's normals and a 23-bit uniform.
// bm(a, b, z0, z1) is the Box-Muller map.
template <int D, typename R, class BM>
__device__ __forceinline__ void unit_randoms(int32_t n, const PhiloxPath &pp, const RoundKeys &rk,
                                             R *z, uint32_t *u, BM bm) {
  if constexpr (D == 3) {
    const uint64_t p = static_cast<uint64_t>(kPhiloxM0) * (3u * (static_cast<uint32_t>(n) >> 2));
    const uint4 A = philox10_product(p, pp, rk);
    const uint4 B = philox10_product(p + kPhiloxM0, pp, rk);
    const uint4 C = philox10_product(p + 2ull * kPhiloxM0, pp, rk);
    bm(A.x, A.y, z[0], z[1]);
    bm(A.z, A.w, z[2], z[3]);
    bm(B.x, B.y, z[4], z[5]);
    bm(B.z, B.w, z[6], z[7]);
    bm(C.x, C.y, z[8], z[9]);
    bm(C.z, C.w, z[10], z[11]);
    u[0] = low_bytes_word(A.x, A.y, A.z);
    u[1] = low_bytes_word(A.w, B.x, B.y);
    u[2] = low_bytes_word(B.z, B.w, C.x);
    u[3] = low_bytes_word(C.y, C.z, C.w);
  } else {
    const uint64_t p = static_cast<uint64_t>(kPhiloxM0) * (3u * (static_cast<uint32_t>(n) >> 2));
    const uint4 A = philox10_product(p, pp, rk);
    const uint4 B = philox10_product(p + kPhiloxM0, pp, rk);
    const uint4 C = philox10_product(p + 2ull * kPhiloxM0, pp, rk);
    const uint32_t w[8] = {A.x, A.y, A.z, A.w, B.x, B.y, B.z, B.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      R z1;
      bm(w[2 * j], w[2 * j + 1], z[D * j], z1);
      if constexpr (D == 2) z[D * j + 1] = z1;
    }
    u[0] = C.x;
    u[1] = C.y;
    u[2] = C.z;
    u[3] = C.w;
  }
}
template <int D, typename R>
__device__ __forceinline__ void unit_randoms(int32_t n, const PhiloxPath &pp, const RoundKeys &rk,
                                             R *z, uint32_t *u) {
  unit_randoms<D, R>(n, pp, rk, z, u,
                     [](uint32_t a, uint32_t b, R &z0, R &z1) { box_muller<R>(a, b, z0, z1); });
}
// The forward path kernel's: binary64 normals from the launch's tables.
template <int D, typename R>
__device__ __forceinline__ void path_randoms(const RoundKeys &rk, const double2 *tables, int32_t n,
                                             const PhiloxPath &pp, R *z, uint32_t *u) {
  if constexpr (sizeof(R) == 8) {
    const NormalTables t(tables);
    unit_randoms<D, R>(n, pp, rk, z, u, [&](uint32_t wa, uint32_t wb, R &z0, R &z1) {
      box_muller_tables(t, wa, wb, z0, z1);
    });
  } else {
    unit_randoms<D, R>(n, pp, rk, z, u);
  }
}

// One loop unit of a path: up to four steps, with the random numbers of
// unit_randoms.  They are formed before the unit's first step: they do not
// depend on the path, so their integer work can interleave with the steps'
// floating-point work.  n counts the steps taken; the unit stops at an exit
// (returns its code, X the start and Xn the end of the exiting step) or at
// max_steps (returns kStepContinue).
template <class Model, class Geom, typename R, bool kLR, bool kSplitCap, class Env>
__device__ __forceinline__ int path_unit_code(const Env &a, const StepConst<R> &k,
                                              const PhiloxPath &pp, const RoundKeys &rk,
                                              int32_t max_steps, R *X, R &Y, R &Z, int32_t &n,
                                              R *Xn, R *L) {
  constexpr int D = Model::D;
  int code;
  R z[4 * D];
  uint32_t u[4];
  unit_randoms<D, R>(n, pp, rk, z, u);
  // kSplitCap: a unit that cannot reach the step cap tests only for exits;
  // one that can (rare: a path near max_steps) takes the steps one at a time
  // with the cap test, its random numbers shifted down by static indices.
  // Without it (kernels whose own body is large, where the second copy of
  // the unit cost more than the tests it saves), every step tests both.
  if (!kSplitCap) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      code = em_step<Model, Geom, R, kLR>(a, k, X, Y, Z, z + D * j, u[j], n, Xn, L);
      ++n;
      if (code != kStepContinue || n >= max_steps) break;
    }
  } else if (n <= max_steps - 4) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      code = em_step<Model, Geom, R, kLR>(a, k, X, Y, Z, z + D * j, u[j], n, Xn, L);
      ++n;
      if (code != kStepContinue) break;
    }
  } else {
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      code = em_step<Model, Geom, R, kLR>(a, k, X, Y, Z, z, u[0], n, Xn, L);
      ++n;
      if (code != kStepContinue || n >= max_steps) break;
#pragma unroll
      for (int i = 0; i < 3 * D; ++i) z[i] = z[i + D];
#pragma unroll
      for (int i = 0; i < 3; ++i) u[i] = u[i + 1];
    }
  }
  return code;
}

// path_unit_code followed, at an exit, by the path's score (returns true,
// score in s, exit point in xe).
template <class Model, class Geom, typename R, bool kLR, class Env>
__device__ __forceinline__ bool path_unit(const Env &a, const StepConst<R> &k, const PhiloxPath &pp,
                                          const RoundKeys &rk, int32_t max_steps, R *X, R &Y,
                                          R &Z, int32_t &n, R &s, R *xe, R *L) {
  R Xn[Model::D];
  const int code =
      path_unit_code<Model, Geom, R, kLR, false>(a, k, pp, rk, max_steps, X, Y, Z, n, Xn, L);
  if (code == kStepContinue) return false;
  s = exit_score<Model, Geom, R>(a.mc, code, X, Xn, Y, Z, xe);
  return true;
}

// Node of global path index g (32-bit division when the indices fit).
__device__ __forceinline__ uint64_t path_node(const PathArgs &a, uint64_t g) {
  if (a.end <= 0xffffffffull)
    return static_cast<uint32_t>(g) / static_cast<uint32_t>(a.n_paths);
  return g / a.n_paths;
}

// Forward mode: optional per-path record (score, exit step, exit point) for
// parity checks, in the caller's buffers.
template <int D, typename R>
__device__ __forceinline__ void dump_path(const PathArgs &a, uint64_t slot, R s, int32_t st,
                                          const R *xe) {
  if (a.dump_score) a.dump_score[slot] = static_cast<double>(s);
  if (a.steps) a.steps[slot] = st;
  if (a.dump_exit) {
#pragma unroll
    for (int d = 0; d < D; ++d) a.dump_exit[slot * D + d] = static_cast<double>(xe[d]);
  }
}

// The log2 of fast_unit's bound: 2^23 + (bits of U >> 8) as a float.
__device__ __forceinline__ float unif_log_bits(float U) {
  return __uint_as_float(__byte_perm(__float_as_uint(U), 0x4b000000u, 0x7321u));
}

// Distance bound of a point (binary32 also for binary64 paths: path_step_args'
// margin covers the rounding).
template <class Geom, typename R>
__device__ __forceinline__ float path_edge(const R *X) {
  float x[Geom::D];
#pragma unroll
  for (int d = 0; d < Geom::D; ++d) x[d] = static_cast<float>(X[d]);
  return Geom::edge(x);
}

// The four steps of the unit at step n (em_step's arithmetic), without exit
// tests: returns whether any step may have been an exit (the unit is then not
// taken).  e: path_edge of X, advanced with it.  n < 2^24 - 4
template <class Model, class Geom, typename R>
__device__ __forceinline__ bool fast_unit(const ModelConst &mc, const StepConst<R> &k, const R *z,
                                          const uint32_t *u, int32_t n, R *X, R &Y, R &Z,
                                          float &e) {
  constexpr int D = Model::D;
  bool maybe = false;
  const float nf = static_cast<float>(n);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    R b[D], Xn[D];
    R f = R(0);
#pragma unroll
    for (int d = 0; d < D; ++d) b[d] = R(0);
    if constexpr (Model::kDrift || Model::kSource) Model::coeffs(mc, X, b, f);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      if ((Model::kDriftAxes >> d) & 1u)
        Xn[d] = X[d] + b[d] * k.dt + k.sdt * z[D * j + d];
      else
        Xn[d] = X[d] + k.sdt * z[D * j + d];
    }
    if constexpr (Model::kSource) Z = Z + f * Y * k.dt;
    if constexpr (Model::kKill == 1) {
      if constexpr (sizeof(R) == 4) Y = k.kill_f(nf + static_cast<float>(j + 1));
      else Y = k.kill(Y, n + j + 1);
    }
    const float en = path_edge<Geom, R>(Xn);
    maybe |= !(unif_log_bits(unif_f(u[j])) >= fmaf(k.edge_c1, e * en, k.edge_c0));
    e = en;
#pragma unroll
    for (int d = 0; d < D; ++d) X[d] = Xn[d];
  }
  return maybe;
}

// The unit at step n again, a step at a time with the exact tests (em_step)
// and the step cap; its random numbers are shifted down by static indices so
// that one copy of the step serves all four.
template <class Model, class Geom, typename R, class Env>
__device__ __forceinline__ int exact_steps(const Env &env, const StepConst<R> &k, int32_t max_steps,
                                           R *z, uint32_t *u, R *X, R &Y, R &Z, int32_t &n, R *Xn) {
  constexpr int D = Model::D;
  int code = kStepContinue;
#pragma unroll 1
  for (int j = 0; j < 4; ++j) {
    code = em_step<Model, Geom, R, false>(env, k, X, Y, Z, z, u[0], n, Xn, static_cast<R *>(nullptr));
    ++n;
    if (code != kStepContinue || n >= max_steps) break;
#pragma unroll
    for (int i = 0; i < 3 * D; ++i) z[i] = z[i + D];
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i] = u[i + 1];
  }
  return code;
}

// Score (s, exit point xe) of a path that left with the code, or was capped:
// then at the projection of its last point on the nearest face.
template <class Model, class Geom, typename R>
__device__ __forceinline__ R end_score(const ModelConst &mc, int code, bool capped, const R *X,
                                       const R *Xn, R Y, R Z, R *xe) {
  if (!capped) return exit_score<Model, Geom, R>(mc, code, X, Xn, Y, Z, xe);
#pragma unroll
  for (int d = 0; d < Model::D; ++d) xe[d] = X[d];
  Geom::project(Geom::nearest_face(X), xe);
  return Model::g(mc, xe) * Y + Z;
}

// Paths at the start of a unit, N of them, in shared memory.  A path's
// killing weight Y is a function of n in binary32 (and 1 without killing):
// only binary64 paths with killing keep it.
template <int D, typename R, bool kY, int N>
struct PathStash {
  unsigned long long id[N];     // the path (Work)
  uint32_t w0[N], w1[N];        // PhiloxPath words (tag 0)
  int32_t n[N];                 // steps taken
  R x[D][N], z[N];
  R y[kY ? N : 1];
};
// Per warp: the paths to take (a stack) and the units to recheck (a ring).
// The ring holds at most 31 + 32 units (32 are taken out whenever there are as
// many).  New paths come in 32 at a time, only into an empty stack, beside at
// most 31 busy lanes and 31 parked units: so a warp never holds more than 94
// paths, and the stack never more than that.
constexpr int kStashCap = 96, kCheckCap = 64;
template <int D, typename R, bool kY>
struct ForwardStage {
  PathStash<D, R, kY, kStashCap> start;
  PathStash<D, R, kY, kCheckCap> check;
};
// At the wave's end lanes idle, and what is left is the longest paths' chain: a
// warp's last paths are finished with several lanes to each (finish_together).
// Before, parked units are rerun once they are as many as the busy lanes: neither
// are the others held up at every unit nor the parked ones for long.
// Binary64 paths are bound by the FP64 pipe to the end, so a warp with at most
// kDonate of them left leaves them (in its own stash, `given` of them) to the
// block's other warps and ends: fewer, fuller warps, the last of which finishes
// its paths as above (16 x 10^4 FP64 paths: 2.06 ms, 2.37 without).  Binary32
// paths are bound by latency there, and fuller warps only hold each other up.  A
// warp that leaves publishes its paths before it lowers `alive`; the warp that
// brings `alive` to zero looks for published paths once more before it ends,
// so none is lost.
constexpr int kDonate = 24;
template <typename R>
constexpr bool kCompact = sizeof(R) == 8;
struct DonorBoard {
  int given[kForwardBlock / 32], taken[kForwardBlock / 32];
  int alive;
};

template <class Model, typename R>
constexpr bool kKeepY = Model::kKill == 1 && sizeof(R) == 8;

// Y of a path that has taken n steps.
template <class Model, typename R>
__device__ __forceinline__ R path_weight(const StepConst<R> &k, int32_t n, R kept) {
  if constexpr (kKeepY<Model, R>) return kept;
  else if constexpr (Model::kKill == 1) return k.kill(R(1), n);  // e^0 = 1 exactly
  else return R(1);
}

// What a launch's warps work through.  A Work type gives the streams and sums
// (rk, normal_tables, max_steps, fix, counters), claims paths 32 at a time
// (claim: lane's path id, node, Philox words and start point; false when the
// lane has none), and per path id its node, model constants (env) and step
// constants.  PathWork: every node with the same number of paths and the same
// constants; the id is the index in the wave.
struct PathEnv {
  const ModelConst &mc;
  int32_t bridge;
};
template <int D, typename R>
struct PathWork {
  using Env = PathEnv;
  static constexpr bool kOwnConsts = false;  // step constants per path
  const PathArgs &a;
  const RoundKeys &rk;
  const double2 *normal_tables;
  NodeFix *fix;
  unsigned long long *counters;
  int32_t max_steps;
  unsigned long long span;
  __device__ __forceinline__ explicit PathWork(const PathArgs &p)
      : a(p), rk(p.rk), normal_tables(p.normal_tables), fix(p.fix), counters(p.counters),
        max_steps(p.max_steps), span(p.end - p.begin) {}
  __device__ __forceinline__ Env env(unsigned long long) const { return Env{a.mc, a.bridge}; }
  __device__ __forceinline__ StepConst<R> consts(unsigned long long) const { return StepConst<R>(a); }
  __device__ __forceinline__ uint64_t node(unsigned long long id) const {
    return path_node(a, a.begin + id);
  }
  __device__ __forceinline__ bool first(unsigned long long) const { return true; }
  __device__ __forceinline__ bool claim(bool &exhausted, unsigned long long &id, uint64_t &node,
                                        PhiloxPath &pp, R *x) const {
    const unsigned lane = threadIdx.x & 31u;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(a.cursor, 32ull);
    base = __shfl_sync(kFull, base, 0);
    if (base + 32 >= span) exhausted = true;
    id = base + lane;
    if (id >= span) return false;
    const unsigned long long g = a.begin + id;
    node = path_node(a, g);
    const uint64_t path = g - node * a.n_paths + a.path_offset;
    pp = philox_path(static_cast<uint32_t>(path), static_cast<uint32_t>(node) + a.node_offset, 0u,
                     a.rk);
#pragma unroll
    for (int d = 0; d < D; ++d) x[d] = static_cast<R>(a.nodes[node * D + d]);
    return true;
  }
  __device__ __forceinline__ void dump(unsigned long long id, R s, int32_t st, const R *xe) const {
    dump_path<D, R>(a, id, s, st, xe);
  }
};

// Called by all 32 lanes with an empty stash: claim up to 32 paths, score at
// once the ones that start on the boundary (tau = 0, u = g, Eq. 2.1) or
// outside the closed domain (invalid input: NaN, counted), and stash the
// interior ones.  Returns how many (warp-uniform).
template <class Model, class Geom, typename R, class Work, class Stash>
__device__ __forceinline__ int stash_starts(const Work &a, Stash &st, bool &exhausted,
                                            unsigned long long &my_bad) {
  constexpr int D = Model::D;
  const unsigned lane = threadIdx.x & 31u;
  __syncwarp();  // earlier reads of the stash are done
  bool interior = false;
  R x[D];
  PhiloxPath pp{0, 0, 0};
  unsigned long long id = 0;
  uint64_t node = 0;
  R s0 = R(0);
  const bool has = a.claim(exhausted, id, node, pp, x);
  if (has) {
    interior = Geom::inside_open(x);
    if (!interior) {
      s0 = Model::g(a.env(id).mc, x);
      if (!Geom::inside_closed(x)) {
        s0 = R(NAN);
        if (a.first(id)) ++my_bad;
      }
      a.dump(id, s0, 0, x);
    }
  }
  // starts on the boundary (u = g, tau = 0) or outside the closed domain (NaN)
  // go straight into the node's sums
  const bool at_bnd = has && !interior;
  if (__any_sync(kFull, at_bnd)) fix_commit<R>(a.fix, at_bnd, node, s0, false, true);
  const unsigned im = __ballot_sync(kFull, interior);
  if (interior) {
    const int e = __popc(im & ((1u << lane) - 1u));
    st.id[e] = id;
    st.w0[e] = pp.r0_w0;
    st.w1[e] = pp.r0_w1;
    st.n[e] = 0;
    st.z[e] = R(0);
    if constexpr (kKeepY<Model, R>) st.y[e] = R(1);
#pragma unroll
    for (int d = 0; d < D; ++d) st.x[d][e] = x[d];
  }
  __syncwarp();
  return __popc(im);
}

// Called by all 32 lanes: the cnt (<= 32) oldest parked units (from ring
// position head) run with the exact tests, one per lane.  Paths that end are
// scored and added to their nodes' sums; the others are pushed on the stash
// (n_start of it filled).
template <class Model, class Geom, typename R, class Work, class Stage>
__device__ __forceinline__ void recheck_units(const Work &a, Stage &st, int head, int cnt, int &n_start,
                                              unsigned long long &my_steps,
                                              unsigned long long &my_capped) {
  constexpr int D = Model::D;
  const int lane = static_cast<int>(threadIdx.x & 31u);
  __syncwarp();
  const bool has = lane < cnt;
  bool ends = false, capped = false;
  R s = R(0), X[D], Xn[D], Y = R(1), Z = R(0);
  PhiloxPath pp{0, 0, 0};
  unsigned long long id = 0;
  uint64_t node = 0;
  int32_t n = 0;
  if (has) {
    const int e = (head + lane) & (kCheckCap - 1);
    id = st.check.id[e];
    pp.r0_w0 = st.check.w0[e];
    pp.r0_w1 = st.check.w1[e];
    n = st.check.n[e];
    Z = st.check.z[e];
    const StepConst<R> k = a.consts(id);
    const typename Work::Env env = a.env(id);
    R y = R(1);
    if constexpr (kKeepY<Model, R>) y = st.check.y[e];
    Y = path_weight<Model, R>(k, n, y);
#pragma unroll
    for (int d = 0; d < D; ++d) X[d] = st.check.x[d][e];
    R z[4 * D];
    uint32_t u[4];
    path_randoms<D, R>(a.rk, a.normal_tables, n, pp, z, u);
    const int code = exact_steps<Model, Geom, R>(env, k, a.max_steps, z, u, X, Y, Z, n, Xn);
    capped = code == kStepContinue && n >= a.max_steps;
    ends = capped || code != kStepContinue;
    if (ends) {
      R xe[D];
      s = end_score<Model, Geom, R>(env.mc, code, capped, X, Xn, Y, Z, xe);
      if (capped) ++my_capped;
      my_steps += static_cast<unsigned long long>(n);
      node = a.node(id);
      a.dump(id, s, capped ? -a.max_steps : n, xe);
    }
  }
  const unsigned back = __ballot_sync(kFull, has && !ends);
  if (has && !ends) {
    const int e = n_start + __popc(back & ((1u << lane) - 1u));
    st.start.id[e] = id;
    st.start.w0[e] = pp.r0_w0;
    st.start.w1[e] = pp.r0_w1;
    st.start.n[e] = n;
    st.start.z[e] = Z;
    if constexpr (kKeepY<Model, R>) st.start.y[e] = Y;
#pragma unroll
    for (int d = 0; d < D; ++d) st.start.x[d][e] = X[d];
  }
  n_start += __popc(back);
  fix_commit<R>(a.fix, ends, node, s, capped, false);
  __syncwarp();
}

// Called by all 32 lanes with cnt <= kTogether paths at a unit's start in the
// stash: runs them to their ends, G = 32 / (the next power of two) lanes to a
// path.  Random numbers are most of a unit's work (about three quarters) and do
// not depend on the path, so each of a path's lanes forms those of another of
// its next G units; then all of them take the units together, the random
// numbers handed round by shuffles, and a unit that may hold an exit at once with
// the exact tests.  Kept out of line: the main loop's registers are its own.
// With at most 16 paths to a warp (8: the L-shape 2 % slower): 16 x 2000 paths
// of the square 141 -> 102 us, 16 x 10^4 FP64 paths with both stages 3.00 ->
// 2.06 ms.
constexpr int kTogether = 16;
struct PathCounts {
  unsigned long long steps, capped;
};
template <class Model, class Geom, typename R, class Work, class Stage>
__device__ __noinline__ PathCounts finish_together(const Work a, Stage &st, int cnt, int32_t last_fast) {
  constexpr int D = Model::D;
  const unsigned lane = threadIdx.x & 31u;
  StepConst<R> k = a.consts(0);
  PathCounts mine{0, 0};
  while (cnt > 0) {
    int lg = 5;  // log2 G
    while (lg > 0 && (32 >> lg) < cnt) --lg;
    const unsigned g = lane & ((1u << lg) - 1u), p = lane >> lg;
    __syncwarp();
    bool alive = static_cast<int>(p) < cnt;
    const int i = alive ? static_cast<int>(p) : 0;
    const unsigned long long id = st.start.id[i];
    if constexpr (Work::kOwnConsts) k = a.consts(id);
    const PhiloxPath pp{st.start.w0[i], st.start.w1[i], 0u};
    int32_t n = st.start.n[i];
    R X[D], Xn[D], Z = st.start.z[i], y = R(1);
    if constexpr (kKeepY<Model, R>) y = st.start.y[i];
    R Y = path_weight<Model, R>(k, n, y);
#pragma unroll
    for (int d = 0; d < D; ++d) X[d] = st.start.x[d][i];
    float e = path_edge<Geom, R>(X);
    const typename Work::Env env = a.env(id);
    __syncwarp();
    int left = cnt;
    do {
      R zg[4 * D];
      uint32_t ug[4];
      path_randoms<D, R>(a.rk, a.normal_tables,
                         static_cast<int32_t>(static_cast<uint32_t>(n) + 4u * g), pp, zg, ug);
      bool ends = false, capped = false;
      R s = R(0);
#pragma unroll 1
      for (int q = 0; q < (1 << lg); ++q) {
        const int from = static_cast<int>(lane - g) + q;
        R z[4 * D];
        uint32_t u[4];
#pragma unroll
        for (int j = 0; j < 4 * D; ++j) z[j] = __shfl_sync(kFull, zg[j], from);
#pragma unroll
        for (int j = 0; j < 4; ++j) u[j] = __shfl_sync(kFull, ug[j], from);
        if (!alive) continue;
        R X0[D], Y0 = Y, Z0 = Z;
#pragma unroll
        for (int d = 0; d < D; ++d) X0[d] = X[d];
        const bool maybe = fast_unit<Model, Geom, R>(env.mc, k, z, u, n, X, Y, Z, e);
        if (!maybe && n <= last_fast) {
          n += 4;
          continue;
        }
#pragma unroll
        for (int d = 0; d < D; ++d) X[d] = X0[d];
        Y = Y0;
        Z = Z0;
        const int code = exact_steps<Model, Geom, R>(env, k, a.max_steps, z, u, X, Y, Z, n, Xn);
        capped = code == kStepContinue && n >= a.max_steps;
        ends = capped || code != kStepContinue;
        if (ends) {
          R xe[D];
          s = end_score<Model, Geom, R>(env.mc, code, capped, X, Xn, Y, Z, xe);
          if (g == 0) {
            a.dump(id, s, capped ? -a.max_steps : n, xe);
            mine.steps += static_cast<unsigned long long>(n);
            mine.capped += capped ? 1u : 0u;
          }
          alive = false;
        } else {
          e = path_edge<Geom, R>(X);
        }
      }
      const bool has = ends && g == 0;
      if (__any_sync(kFull, has)) fix_commit<R>(a.fix, has, has ? a.node(id) : 0, s, capped, false);
      left = __popc(__ballot_sync(kFull, alive && g == 0));
    } while (left > 0 && (left > 32 >> (lg + 1) || lg == 5));
    // fewer paths than half the groups: more lanes to each
    const unsigned am = __ballot_sync(kFull, alive && g == 0);
    if (alive && g == 0) {
      const int o = __popc(am & ((1u << lane) - 1u));
      st.start.id[o] = id;
      st.start.w0[o] = pp.r0_w0;
      st.start.w1[o] = pp.r0_w1;
      st.start.n[o] = n;
      st.start.z[o] = Z;
      if constexpr (kKeepY<Model, R>) st.start.y[o] = Y;
#pragma unroll
      for (int d = 0; d < D; ++d) st.start.x[d][o] = X[d];
    }
    cnt = left;
  }
  __syncwarp();
  return mine;
}

// The block's paths, from a Work.
template <class Model, class Geom, typename R, class Work>
__device__ __forceinline__ void forward_paths(const Work &a) {
  constexpr int D = Model::D;
  using Stage = ForwardStage<D, R, kKeepY<Model, R>>;
  __shared__ Stage stage_all[kForwardBlock / 32];
  Stage &stage = stage_all[threadIdx.x >> 5];
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt_mask = (1u << lane) - 1u;
  StepConst<R> k = a.consts(0);
  // the last unit start that ends below the step cap (and below the step counts
  // that binary32 does not hold)
  const int32_t last_fast = (a.max_steps < (1 << 24) ? a.max_steps : 1 << 24) - 5;
  R X[D], Y = R(1), Z = R(0);
  float e = 0.0f;
  PhiloxPath pp{0, 0, 0};
  unsigned long long id = 0;
  int32_t n = 0;
  bool active = false;
  int n_start = 0;              // stash fill; parked units and the oldest (warp-uniform)
  int n_check = 0, head = 0;
  bool exhausted = false;       // the wave's indices are all claimed (warp-uniform)
  bool last = false;            // the block's last warp (warp-uniform)
  unsigned long long my_steps = 0, my_capped = 0, my_bad = 0;
  constexpr int kWarps = kForwardBlock / 32;
  __shared__ DonorBoard board;
  if (threadIdx.x < kWarps) board.given[threadIdx.x] = board.taken[threadIdx.x] = 0;
  if (threadIdx.x == 0) board.alive = kWarps;
  __syncthreads();

  // entry i of a stash becomes the lane's path
  auto load = [&](const auto &st, int i) {
    id = st.id[i];
    if constexpr (Work::kOwnConsts) k = a.consts(id);
    pp.r0_w0 = st.w0[i];
    pp.r0_w1 = st.w1[i];
    pp.tag = 0u;
    n = st.n[i];
    Z = st.z[i];
    R y = R(1);
    if constexpr (kKeepY<Model, R>) y = st.y[i];
    Y = path_weight<Model, R>(k, n, y);
#pragma unroll
    for (int d = 0; d < D; ++d) X[d] = st.x[d][i];
    e = path_edge<Geom, R>(X);
    active = true;
  };
  // entry i of a stash from the start of the lane's unit
  auto store = [&](auto &st, int i, int32_t n0, const R *X0, R Y0, R Z0) {
    st.id[i] = id;
    st.w0[i] = pp.r0_w0;
    st.w1[i] = pp.r0_w1;
    st.n[i] = n0;
    st.z[i] = Z0;
    if constexpr (kKeepY<Model, R>) st.y[i] = Y0;
#pragma unroll
    for (int d = 0; d < D; ++d) st.x[d][i] = X0[d];
    active = false;
  };
  // idle lanes take published paths, this warp's own first (the last warp's);
  // returns the lanes still idle
  auto adopt = [&](unsigned need) -> unsigned {
    volatile DonorBoard &vb = board;
    const unsigned from = __ballot_sync(kFull, lane < kWarps && vb.taken[lane % kWarps] < vb.given[lane % kWarps]);
    if (!from) return need;
    for (int q = 0; need && q < kWarps; ++q) {
      const int w = (static_cast<int>(threadIdx.x >> 5) + q) % kWarps;
      if (!((from >> w) & 1u)) continue;
      int at = 0;
      if (lane == 0) at = atomicAdd(&board.taken[w], __popc(need));
      at = __shfl_sync(kFull, at, 0);
      __threadfence_block();
      const int i = at + __popc(need & lt_mask);
      if (!active && i < vb.given[w]) load(stage_all[w].start, i);
      need = __ballot_sync(kFull, !active);
    }
    return need;
  };

  // every path that the warp holds into its stash (empty before); returns how many
  auto gather = [&](unsigned need) -> int {
    const int busy = 32 - __popc(need);
    if (active) store(stage.start, __popc(~need & lt_mask), n, X, Y, Z);
    if (static_cast<int>(lane) < n_check) {  // parked units are paths at a unit's start
      const int i = (head + static_cast<int>(lane)) & (kCheckCap - 1), o = busy + static_cast<int>(lane);
      stage.start.id[o] = stage.check.id[i];
      stage.start.w0[o] = stage.check.w0[i];
      stage.start.w1[o] = stage.check.w1[i];
      stage.start.n[o] = stage.check.n[i];
      stage.start.z[o] = stage.check.z[i];
      if constexpr (kKeepY<Model, R>) stage.start.y[o] = stage.check.y[i];
#pragma unroll
      for (int d = 0; d < D; ++d) stage.start.x[d][o] = stage.check.x[d][i];
    }
    const int all = busy + n_check;
    n_check = 0;
    __syncwarp();
    return all;
  };
  // the oldest cnt parked units
  auto recheck = [&](int cnt) {
    recheck_units<Model, Geom, R>(a, stage, head, cnt, n_start, my_steps, my_capped);
    head = (head + cnt) & (kCheckCap - 1);
    n_check -= cnt;
  };
  // one unit of the lane's path; a unit that may hold an exit, or reach the
  // step cap, is parked as it started
  auto advance = [&]() {
    bool park = false;
    R X0[D], Z0 = Z, Y0 = Y;
#pragma unroll
    for (int d = 0; d < D; ++d) X0[d] = X[d];
    if (active) {
      R z[4 * D];
      uint32_t u[4];
      path_randoms<D, R>(a.rk, a.normal_tables, n, pp, z, u);
      park = fast_unit<Model, Geom, R>(a.env(id).mc, k, z, u, n, X, Y, Z, e) || n > last_fast;
      n += 4;
    }
    const unsigned pm = __ballot_sync(kFull, park);
    if (pm) {
      if (park) store(stage.check, (head + n_check + __popc(pm & lt_mask)) & (kCheckCap - 1), n - 4, X0, Y0, Z0);
      n_check += __popc(pm);
    }
  };

  // ---- while the wave has paths: every lane busy, parked units 32 together
  for (;;) {
    if (n_check >= 32) recheck(32);
    unsigned need = __ballot_sync(kFull, !active);
    while (need) {  // idle lanes take stashed paths; an empty stash is refilled
      if (n_start == 0) {
        if (exhausted) break;
        n_start = stash_starts<Model, Geom, R>(a, stage.start, exhausted, my_bad);
        continue;
      }
      const int r = __popc(need & lt_mask), cnt = __popc(need);
      const int take = cnt < n_start ? cnt : n_start;
      if (!active && r < take) load(stage.start, n_start - 1 - r);
      n_start -= take;
      need = __ballot_sync(kFull, !active);
    }
    if (need) break;
    advance();
  }

  // ---- the wave's end: lanes idle (see DonorBoard)
#pragma unroll 1
  for (;;) {
    unsigned need = __ballot_sync(kFull, !active);
    if (need && n_start > 0) {
      const int r = __popc(need & lt_mask), cnt = __popc(need);
      const int take = cnt < n_start ? cnt : n_start;
      if (!active && r < take) load(stage.start, n_start - 1 - r);
      n_start -= take;
      need = __ballot_sync(kFull, !active);
    }
    if (need && 32 - __popc(need) + n_check <= kTogether && (!kCompact<R> || last)) {
      if constexpr (kCompact<R>) need = adopt(need);
      if (32 - __popc(need) + n_check <= kTogether) {
        const PathCounts c = finish_together<Model, Geom, R>(a, stage, gather(need), last_fast);
        my_steps += c.steps;
        my_capped += c.capped;
        break;
      }
    }
    if (n_check > 0 && (n_check >= 32 || n_check >= 32 - __popc(need))) {
      recheck(n_check < 32 ? n_check : 32);
      continue;
    }
    if (need) {
      if constexpr (kCompact<R>) {
        need = adopt(need);
        const int left = 32 - __popc(need), all = left + n_check;
        if (all <= kDonate && !last) {
          gather(need);
          __threadfence_block();
          __syncwarp();
          int before = 0;
          if (lane == 0) {
            volatile DonorBoard &vb = board;
            vb.given[threadIdx.x >> 5] = all;
            __threadfence_block();
            before = atomicSub(&board.alive, 1);
            if (before == 1) board.alive = 1;  // the last warp stays while there are paths
          }
          before = __shfl_sync(kFull, before, 0);
          if (before > 1) break;
          last = true;
          need = adopt(kFull);
        }
      }
      if (need == kFull) break;
    }
    advance();
  }

  // ---- per-warp totals
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    my_steps += __shfl_xor_sync(kFull, my_steps, m);
    my_capped += __shfl_xor_sync(kFull, my_capped, m);
    my_bad += __shfl_xor_sync(kFull, my_bad, m);
  }
  if (lane == 0) {
    if (my_steps) atomicAdd(&a.counters[0], my_steps);
    if (my_capped) atomicAdd(&a.counters[1], my_capped);
    if (my_bad) atomicAdd(&a.counters[2], my_bad);
  }
}

// Blocks per SM the registers are held to: 72 registers for binary32 (seven
// blocks: the 3-D solve 762 ms, 773 at 78 registers and six), 64 for the 2-D
// family with drift (eight: its forward pass 1.5 % faster; the Laplace family's
// small calls were 4 % slower so), 128 and 168 for binary64 without and with
// drift (spills below).
template <class Model, typename R>
constexpr int kForwardBlocks = sizeof(R) == 4 ? (Model::kDrift && Model::D == 2 ? 8 : 7)
                                              : (Model::kDrift ? 3 : 4);

// Of the bps blocks that fit an SM, those that a launch over `paths` paths uses:
// more warps hide more latency, but the longest paths' chain at the end runs from
// the moment the paths are all claimed, and the fewer paths a lane gets the larger
// its share (and the slower each of the chain's steps, beside more warps).  P
// paths per lane and block of an SM: about sqrt(P) / 1.6 blocks, at least two.
// Cube, dt = 10^-3, blocks 2 .. 7: 275 275 291 312 343 377 us (P = 13), 523 484 486
// 493 509 522 us (41), 762 685 666 664 670 683 us (66), 1519 1258 1172 1144 1137 1150
// us (154), 2852 2319 2122 2028 1993 1986 us (308); the square and the L-shape, the
// gradient's and the reflecting paths alike.  (Binary64 absorbing paths, bound by
// the FP64 pipe from two blocks on, are within 2 % at any number.)
inline int blocks_for_paths(int bps, uint64_t paths, int num_sms, int block) {
  const double P = static_cast<double>(paths) / (static_cast<double>(num_sms) * block);
  const double k = std::sqrt(P) / 1.6 + 0.5;
  return k >= bps ? bps : std::min(bps, std::max(2, static_cast<int>(k)));
}

template <class Model, class Geom, typename R>
__global__ void __launch_bounds__(kForwardBlock, kForwardBlocks<Model, R>)
path_kernel(const __grid_constant__ PathArgs a) {
  forward_paths<Model, Geom, R>(PathWork<Model::D, R>(a));
}

}  // namespace pdd
