// reflect.cu -- interface paths with reflecting faces: the mixed BVP of
// Eq. 2.4 (Robin data du/dN = phi u + psi on the reflecting part of the
// boundary) through the local-time system of Eq. 2.9: X is pushed back into
// the domain by the local time xi (dX = ... - N dxi), Y gains phi Y dxi and
// Z gains psi Y dxi.
//
// A step is the Euler-Maruyama step of the path kernel (same streams, tag 0)
// followed, for every reflecting face within bridge reach, by Lepingle's
// half-space reflection: with distances y (start) and y' (free end), the
// Brownian bridge's minimum is m = (y + y' - sqrt((y' - y)^2 - 2 sigma^2 dt
// ln U')) / 2, the local time L = max(0, -m), and the end point moves in by
// L.  U' for axis k comes from the tag-4 stream Philox((b, p, i, 4)): in 3-D
// word k of block b = n; in 2-D word 2 (n mod 2) + k of block b = n / 2, so
// one block serves two steps.  It matters only when a reflecting face is
// within reach (2 y y' / (sigma^2 dt) < 18; beyond, L = 0 for every
// U' >= 2^-24).  Along the local time the weights are integrated
// exactly with psi frozen at the end point's projection: Z += psi Y (e^{phi
// L} - 1) / phi, Y *= e^{phi L}; then the time part as in the path kernel
// (left point).  Absorbing faces keep the hard-exit and bridge tests.
// Y is formed as exp(n c dt + sum phi L) so binary32 rounding does not
// accumulate along the path.
//
// What bounds it: instruction issue, above all Philox's wide multiplies (1.25
// blocks per 2-D step, with the tag-4 stream).  The kernel works as the path
// kernel does: units of four steps without an exit test, screened by one bound
// over the absorbing faces (the smallest d d' against the bits of U,
// edge_bound) and redone 32 at a time with the exact tests where they may hold
// an exit.  A reflection moves the path at once, but its weight (two
// exponentials, expm1, the Robin data) does not act on the path: it is queued
// and formed with those of the other lanes, and each lane adds its own in order
// (bit-identical sums).  16 nodes of the square, two reflecting faces, 10^6
// paths each: 51.3 ms with weights and exit tests where they occur (21.8 of 32
// lanes), 40.6 ms now; in binary64, 2 x 10^4 paths, 130 -> 66 ms (the normals
// from tables).
#include <cmath>
#include <cstring>

#include "ctx.hpp"
#include "models.cuh"
#include "path_kernel.cuh"
#include "reduce.cuh"

namespace pdd {

struct ReflectArgs {
  const double *nodes;
  uint64_t n_paths, path_offset, begin, end;
  uint32_t node_offset;          // stream index of node 0
  unsigned long long *cursor;
  unsigned long long *counters;  // [0] steps, [1] capped, [2] bad nodes
  void *score;
  int32_t *steps;
  int32_t *flags;                // per-node flags or null (rare events, atomicOr)
  double *exit;                  // exit point per path [end - begin][D] or null
  RoundKeys rk;
  double dt, sdt, s2dt, cdt, phi;  // dt, sigma sqrt(dt), sigma^2 dt, c dt, Robin phi
  // the binary32 step constants, rounded on the host (dt, sdt, s2dt, cdt, phi,
  // 1 / s2dt, b2, boff of ReflectConst): formed in the kernel from the FP64
  // fields, they were re-formed inside the step loop on the FP64 pipe
  float kf[8];
  // the reflecting faces in order: axis, and x -> rs x + ro the distance; the
  // range [rlo, rhi] that a reflected coordinate is clamped to
  int32_t n_refl, r_face[6];
  float rs[6], ro[6], rlo[6], rhi[6];
  float add[6];                    // 0 for an absorbing face, large for a reflecting one
  float edge_c0, edge_c1;          // screening bound over the absorbing faces (edge_bound)
  const double2 *normal_tables;    // FP64 paths: NormalTables
  int32_t mask;                    // bit j: face j reflects
  int32_t max_steps, bridge;
  ModelConst mc;
};

// Optional per-path exit point (parity checks).
template <int D, typename R>
__device__ __forceinline__ void dump_exit_point(double *exit, uint64_t slot, const R *x) {
  if (exit) {
#pragma unroll
    for (int d = 0; d < D; ++d) exit[slot * D + d] = static_cast<double>(x[d]);
  }
}

// Special functions of the reflections' weights: binary32 takes the hardware
// approximations (relative errors of order 1e-7 against the 1e-4 per-path and
// 1e-5 per-node parity bars), binary64 the accurate library functions.  expm1
// stays accurate: its argument phi L is small, where exp(v) - 1 would cancel.
__device__ __forceinline__ float rb_exp(float x) { return exp_fast(x); }
__device__ __forceinline__ double rb_exp(double x) { return exp(x); }
__device__ __forceinline__ float rb_cos(float x) { return cos_approx(x); }   // |x| <= 1 here
__device__ __forceinline__ double rb_cos(double x) { return cos(x); }
__device__ __forceinline__ float rb_sin(float x) { return sin_approx(x); }
__device__ __forceinline__ double rb_sin(double x) { return sin(x); }
__device__ __forceinline__ float rb_sinpi(float x) { return sin_approx(3.14159265358979324f * x); }
__device__ __forceinline__ double rb_sinpi(double x) { return sinpi(x); }
__device__ __forceinline__ float rb_cospi(float x) { return cos_approx(3.14159265358979324f * x); }
__device__ __forceinline__ double rb_cospi(double x) { return cospi(x); }

// Outward-normal derivative of the family's exact solution on face j.
template <class Model> struct RobinData;
template <> struct RobinData<LaplaceExpCos> {
  template <typename R>
  __device__ static R dudn(int j, const R *x) {
    const R e = rb_exp(x[0]);
    const R g = (j >> 1) == 0 ? e * rb_cos(x[1]) : -e * rb_sin(x[1]);
    return (j & 1) ? g : -g;
  }
  template <typename R>
  __device__ static R u(const R *x) { return rb_exp(x[0]) * rb_cos(x[1]); }
};
template <> struct RobinData<EllipticManufactured> {
  template <typename R>
  __device__ static R dudn(int j, const R *x) {
    constexpr double kPi = 3.14159265358979323846;
    const int k = j >> 1;
    const R ez = rb_exp(x[2]);
    R g;
    if (k == 0) g = R(kPi) * rb_cospi(x[0]) * rb_sinpi(x[1]) * ez;
    else if (k == 1) g = R(kPi) * rb_sinpi(x[0]) * rb_cospi(x[1]) * ez;
    else g = rb_sinpi(x[0]) * rb_sinpi(x[1]) * ez;
    return (j & 1) ? g : -g;
  }
  template <typename R>
  __device__ static R u(const R *x) { return rb_sinpi(x[0]) * rb_sinpi(x[1]) * rb_exp(x[2]); }
};

template <typename R> __device__ __forceinline__ R r_exp(R v);
template <> __device__ __forceinline__ float r_exp<float>(float v) { return exp_fast(v); }
template <> __device__ __forceinline__ double r_exp<double>(double v) { return exp(v); }
template <typename R> __device__ __forceinline__ R r_expm1(R v);
template <> __device__ __forceinline__ float r_expm1<float>(float v) { return expm1f(v); }
template <> __device__ __forceinline__ double r_expm1<double>(double v) { return expm1(v); }
template <typename R> __device__ __forceinline__ R r_log(R v);
template <> __device__ __forceinline__ float r_log<float>(float v) {
  return 0.6931471805599453f * lg2_approx(v);
}
template <> __device__ __forceinline__ double r_log<double>(double v) { return log(v); }
__device__ __forceinline__ float r_sqrt(float v) { return sqrt_approx(fmaxf(v, 0.0f)); }
__device__ __forceinline__ double r_sqrt(double v) { return sqrt(v); }

// Step constants of the reflecting kernel in the path precision.
template <typename R>
struct ReflectConst {
  R dt, sdt, s2dt, cdt, phi, inv_s2dt;
  R b2;    // -2 log2(e) / (sigma^2 dt): exp(-2 m / (sigma^2 dt)) = 2^(b2 m)
  R boff;  // log2(2D) + 2^-12 with the bridge test, -inf without
};

// Bound on the absorbing faces' crossing probability of a step whose smallest
// d d' over them is m: P = 1 - prod (1 - p_j) <= sum p_j <= 2D exp(-2 m /
// (sigma^2 dt)), raised by 2^(2^-12) for the rounding of the exponents.
__device__ __forceinline__ float reflect_bound(const ReflectConst<float> &k, float m) {
  return ex2_approx(fmaf(k.b2, m, k.boff));
}
__device__ __forceinline__ double reflect_bound(const ReflectConst<double> &k, double m) {
  return exp2(k.b2 * m + k.boff);
}

// One step of a reflecting path from X (Zs, Zr, sphil and n its running sums:
// source and boundary part of Z, phi times the local time, steps):
// the Euler-Maruyama move with normals xi, Lepingle's reflection on the
// reflecting faces within reach (axis k's uniform word: word wo + k of the
// tag-4 block rw), and the absorbing exit tests with the bridge uniform word
// wu.  Returns true when the path left through an absorbing
// face (xe its exit point); X advances otherwise, Zs and Zr in both cases.
template <class Model, typename R>
__device__ __forceinline__ bool reflect_step(const ReflectArgs &a, const ReflectConst<R> &k,
                                             const uint4 &rw, int wo, R *X, R &Zs, R &Zr, R &sphil,
                                             int32_t n, const R *xi, uint32_t wu, R *xe) {
  constexpr int D = Model::D;
  using G = Box<D>;
  R b[3] = {R(0), R(0), R(0)}, f = R(0);
  Model::template coeffs<R>(a.mc, X, b, f);
  // Y at the step's start; needed every step only with a source term
  constexpr bool kYStep = Model::kSource;
  const R Y = kYStep ? r_exp<R>(static_cast<R>(n) * k.cdt + sphil) : R(0);
  R Xn[3];
#pragma unroll
  for (int q = 0; q < D; ++q) Xn[q] = X[q] + b[q] * k.dt + k.sdt * xi[q];

  // ---- reflection on the reflecting faces within reach.  The bridge
  // minimum is formed for every reflecting face and step (full lanes: paths
  // linger near these faces, so a branch on reach would run, diverged, at
  // most warp-steps); only an actual reflection (L > 0) branches.
  R zr = R(0), yr = Y;
  bool have_y = kYStep;
#pragma unroll
  for (int j = 0; j < 2 * D; ++j) {
    if (!((a.mask >> j) & 1)) continue;
    const R y0 = G::template face_dist<R>(j, X), y1 = G::template face_dist<R>(j, Xn);
    const bool reach = R(2) * y0 * y1 * k.inv_s2dt < R(18);
    const int q = j >> 1;
    const int w = wo + q;
    const uint32_t wk = w == 0 ? rw.x : w == 1 ? rw.y : w == 2 ? rw.z : rw.w;
    const R dy = y1 - y0;
    const R mn = R(0.5) * (y0 + y1 - r_sqrt(dy * dy - R(2) * k.s2dt * r_log<R>(unif<R>(wk))));
    const R L = (reach && mn < R(0)) ? -mn : R(0);
    if (L > R(0)) {
      if (j & 1) Xn[q] = fmin(Xn[q] - L, R(1));
      else Xn[q] = fmax(Xn[q] + L, R(0));
      R xp[3] = {Xn[0], Xn[1], Xn[2]};
      xp[q] = R(j & 1);
      const R psi = RobinData<Model>::template dudn<R>(j, xp) - k.phi * RobinData<Model>::template u<R>(xp);
      if (!have_y) {
        yr = r_exp<R>(static_cast<R>(n) * k.cdt + sphil);
        have_y = true;
      }
      const R g1 = k.phi != R(0) ? r_expm1<R>(k.phi * L) / k.phi : L;
      zr += psi * yr * g1;
      yr *= r_exp<R>(k.phi * L);
      sphil += k.phi * L;
    }
  }
  if (kYStep) Zs += f * Y * k.dt;
  Zr += zr;

  // ---- exit through absorbing faces.  am > 0 puts X' strictly inside the
  // absorbing faces (the reflecting ones keep it in [0, 1]); above the bound
  // no absorbing crossing is possible.  Below, the exact tests.
  R am = R(1);
#pragma unroll
  for (int j = 0; j < 2 * D; ++j)
    if (!((a.mask >> j) & 1))
      am = fmin(am, G::template face_dist<R>(j, X) * G::template face_dist<R>(j, Xn));
  const R U = unif<R>(wu);
  bool out = false;
  if (!(am > R(0)) || U < reflect_bound(k, am)) {
#pragma unroll
    for (int q = 0; q < D; ++q) xe[q] = Xn[q];
    if (!G::template inside_closed<R>(Xn)) {
      G::template segment_exit<R>(X, Xn, xe);
      out = true;
    } else if (a.bridge) {
      R P = R(0), pb = R(-1);
      int jb = -1;
#pragma unroll
      for (int j = 0; j < 2 * D; ++j) {
        if ((a.mask >> j) & 1) continue;
        const R e = R(2) * G::template face_dist<R>(j, X) * G::template face_dist<R>(j, Xn) * k.inv_s2dt;
        if (e < R(18)) {
          const R p = r_exp<R>(-e);
          P = P + p * (R(1) - P);
          if (p > pb) {
            pb = p;
            jb = j;
          }
        }
      }
      if (jb >= 0 && U < P) {
#pragma unroll
        for (int j = 0; j < 2 * D; ++j)
          if (j == jb) G::template project<R>(j, xe);
        out = true;
      }
    }
  }
  if (out) return true;
#pragma unroll
  for (int q = 0; q < D; ++q) X[q] = Xn[q];
  return false;
}

// A reflection whose weight is still to be added: the tangential coordinates of
// its point, its local time L, the exponent of Y before it and its code, 1 + face
// + 8 times its place among the step's reflections.
template <int D, typename R>
struct ReflectEvents {
  static constexpr int kCap = 8;  // per lane
  struct alignas(16) Event {
    R t, L, y, code;
  };
  Event e[kCap][32];
  R t2[D == 3 ? kCap : 1][32];
  uint16_t map[kCap * 32];
};

// The same step without a branch: reflections are applied and queued in ev
// (cnt of them so far; more than kCap: the step has to be redone).  Returns true
// when the step may leave through an absorbing face.
template <class Model, typename R, int NR>
__device__ __forceinline__ bool reflect_fast(const ReflectArgs &a, const ReflectConst<R> &k,
                                             const uint4 &rw, int wo, R *X, R &Zs, R &sphil, int32_t n,
                                             const R *xi, uint32_t wu, int &cnt,
                                             ReflectEvents<Model::D, R> &ev) {
  constexpr int D = Model::D;
  using G = Box<D>;
  using Ev = ReflectEvents<D, R>;
  const unsigned lane = threadIdx.x & 31u;
  R b[3] = {R(0), R(0), R(0)}, f = R(0);
  Model::template coeffs<R>(a.mc, X, b, f);
  if constexpr (Model::kSource)
    Zs += f * r_exp<R>(static_cast<R>(n) * k.cdt + sphil) * k.dt;
  R Xn[3];
#pragma unroll
  for (int q = 0; q < D; ++q) Xn[q] = X[q] + b[q] * k.dt + k.sdt * xi[q];
  const int nr = NR ? NR : a.n_refl;
  R place = R(1);  // 1 + 8 times the step's reflections so far
#pragma unroll
  for (int r = 0; r < (NR ? NR : 2 * D); ++r) {
    if (r >= nr) break;
    const int j = a.r_face[r], q = j >> 1;
    const R sg = static_cast<R>(a.rs[r]), of = static_cast<R>(a.ro[r]);
    const R x0 = q == 0 ? X[0] : (D == 2 || q == 1 ? X[1] : X[2]);
    const R x1 = q == 0 ? Xn[0] : (D == 2 || q == 1 ? Xn[1] : Xn[2]);
    const R y0 = fma(sg, x0, of), y1 = fma(sg, x1, of);
    const bool reach = R(2) * y0 * y1 * k.inv_s2dt < R(18);
    const uint32_t wk = D == 3 ? (q == 0 ? rw.x : q == 1 ? rw.y : rw.z)
                               : (q == 0 ? (wo ? rw.z : rw.x) : (wo ? rw.w : rw.y));
    const R dy = y1 - y0;
    const R mn = R(0.5) * (y0 + y1 - r_sqrt(dy * dy - R(2) * k.s2dt * r_log<R>(unif<R>(wk))));
    if (reach && mn < R(0)) {
      const R L = -mn;
      const R in = fmin(fmax(x1 + sg * L, static_cast<R>(a.rlo[r])), static_cast<R>(a.rhi[r]));
      if (q == 0) Xn[0] = in;
      else if (D == 2 || q == 1) Xn[1] = in;
      else Xn[2] = in;
      if (cnt < Ev::kCap) {
        ev.e[cnt][lane] = {q == 0 ? Xn[1] : Xn[0], L, static_cast<R>(n) * k.cdt + sphil,
                           place + static_cast<R>(j)};
        if constexpr (D == 3) ev.t2[cnt][lane] = q == 2 ? Xn[1] : Xn[2];
      }
      ++cnt;
      place += R(8);
      sphil += k.phi * L;
    }
  }
  R am = R(1);
#pragma unroll
  for (int j = 0; j < 2 * D; ++j)
    am = fmin(am, fma(G::template face_dist<R>(j, X), G::template face_dist<R>(j, Xn),
                      static_cast<R>(a.add[j])));
#pragma unroll
  for (int q = 0; q < D; ++q) X[q] = Xn[q];
  return !(am > R(0) && unif_log_bits(unif_f(wu)) >= fmaf(a.edge_c1, static_cast<float>(am), a.edge_c0));
}

// Paths at the start of a unit, N of them, in shared memory.
template <class Model, typename R, int N>
struct ReflectStash {
  unsigned long long id[N];
  uint32_t w0[N], w1[N];
  int32_t n[N];
  R x[Model::D][N], zr[N], sphil[N], zs[Model::kSource ? N : 1];
};
template <class Model, typename R>
struct ReflectStage {
  ReflectStash<Model, R, 96> start;  // (capacities: see path_kernel.cuh, ForwardStage)
  ReflectStash<Model, R, 64> check;
  ReflectEvents<Model::D, R> ev;
};
// Threads per block (within 48 KB of stages).
template <class Model, typename R>
constexpr int kReflectBlock = sizeof(R) == 4 && Model::D == 2 ? 128 : 64;

// NR: the number of reflecting faces, or 0 for any.
template <class Model, typename R, int NR>
__global__ void __launch_bounds__(kReflectBlock<Model, R>) reflect_kernel(const __grid_constant__ ReflectArgs a) {
  constexpr int D = Model::D;
  using G = Box<D>;
  using Ev = ReflectEvents<D, R>;
  __shared__ ReflectStage<Model, R> stage_all[kReflectBlock<Model, R> / 32];
  ReflectStage<Model, R> &st = stage_all[threadIdx.x >> 5];
  const unsigned lane = threadIdx.x & 31u, lt_mask = (1u << lane) - 1u;
  ReflectConst<R> k;
  if constexpr (sizeof(R) == 4) {
    k.dt = a.kf[0];
    k.sdt = a.kf[1];
    k.s2dt = a.kf[2];
    k.cdt = a.kf[3];
    k.phi = a.kf[4];
    k.inv_s2dt = a.kf[5];
    k.b2 = a.kf[6];
    k.boff = a.kf[7];
  } else {
    k.dt = a.dt;
    k.sdt = a.sdt;
    k.s2dt = a.s2dt;
    k.cdt = a.cdt;
    k.phi = a.phi;
    k.inv_s2dt = 1.0 / k.s2dt;
    k.b2 = -2.0 * 1.4426950408889634 / a.s2dt;
    k.boff = a.bridge ? (D == 2 ? 2.0 : 2.584962500721156) + 2.44140625e-4 : -INFINITY;
  }
  const int32_t last_fast = min(a.max_steps, 1 << 24) - 5;
  R X[3] = {R(0), R(0), R(0)};
  R Zs = R(0), Zr = R(0), sphil = R(0);  // source and boundary sums; phi times the local time
  PhiloxPath pp{0, 0, 0u};
  unsigned long long id = 0;
  int32_t n = 0;
  int cnt = 0;  // the lane's queued reflections
  bool active = false, exhausted = false;
  int n_start = 0, n_check = 0, head = 0;  // warp-uniform
  unsigned long long my_steps = 0, my_capped = 0, my_bad = 0;
  R *score = static_cast<R *>(a.score);
  const unsigned long long total = a.end - a.begin;

  auto node_of = [&](unsigned long long g) -> unsigned long long {
    if (a.end <= 0xffffffffull && a.n_paths <= 0xffffffffull)
      return static_cast<uint32_t>(g) / static_cast<uint32_t>(a.n_paths);
    return g / a.n_paths;
  };
  auto load = [&](const auto &q, int i) {
    id = q.id[i];
    pp.r0_w0 = q.w0[i];
    pp.r0_w1 = q.w1[i];
    n = q.n[i];
#pragma unroll
    for (int d = 0; d < D; ++d) X[d] = q.x[d][i];
    Zr = q.zr[i];
    sphil = q.sphil[i];
    if constexpr (Model::kSource) Zs = q.zs[i];
  };
  auto store = [&](auto &q, int i, int32_t n0, const R *x, R zs, R zr, R sp) {
    q.id[i] = id;
    q.w0[i] = pp.r0_w0;
    q.w1[i] = pp.r0_w1;
    q.n[i] = n0;
#pragma unroll
    for (int d = 0; d < D; ++d) q.x[d][i] = x[d];
    q.zr[i] = zr;
    q.sphil[i] = sp;
    if constexpr (Model::kSource) q.zs[i] = zs;
  };
  // the tag-4 blocks of a unit's steps: one per two steps in 2-D, one per step
  // in 3-D
  auto refl_block = [&](int32_t step) {
    const PhiloxPath p4{pp.r0_w0, pp.r0_w1, 4u};
    return philox10_path(static_cast<uint32_t>(D == 3 ? step : step >> 1), p4, a.rk);
  };

  // ---- claim 32 paths into the empty stash; starts on an absorbing face or
  // outside are scored at once
  auto claim = [&]() {
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(a.cursor, 32ull);
    base = __shfl_sync(kFull, base, 0);
    if (base + 32 >= total) exhausted = true;
    const unsigned long long q = base + lane, id0 = id;
    const PhiloxPath pp0 = pp;
    bool in = false;
    R x[3] = {R(0), R(0), R(0)};
    if (q < total) {
      const unsigned long long g = a.begin + q, node = node_of(g);
      pp = philox_path(static_cast<uint32_t>(g - node * a.n_paths + a.path_offset),
                       static_cast<uint32_t>(node) + a.node_offset, 0u, a.rk);
      id = q;
#pragma unroll
      for (int d = 0; d < D; ++d) x[d] = static_cast<R>(a.nodes[node * D + d]);
      const bool bad = !G::template inside_closed<R>(x);
      bool on_abs = bad;
#pragma unroll
      for (int d = 0; d < D; ++d)
        on_abs = on_abs || (x[d] <= R(0) && !((a.mask >> (2 * d)) & 1)) ||
                 (x[d] >= R(1) && !((a.mask >> (2 * d + 1)) & 1));
      in = !on_abs;
      if (on_abs) {
        score[q] = bad ? R(NAN) : Model::template g<R>(a.mc, x);
        if (a.steps) a.steps[q] = 0;
        dump_exit_point<D>(a.exit, q, x);
        if (a.flags) atomicOr(a.flags + node, bad ? kNodeOutside : kNodeOnBoundary);
        if (bad) ++my_bad;
      }
    }
    const unsigned im = __ballot_sync(kFull, in);
    if (in) store(st.start, __popc(im & lt_mask), 0, x, R(0), R(0), R(0));
    id = id0;
    pp = pp0;
    __syncwarp();
    n_start = __popc(im);
  };

  // ---- the queued reflections' weights, one per lane, then each lane adds its
  // own in order
  auto flush = [&]() {
    __syncwarp();
    int inc = cnt;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const int v = __shfl_up_sync(kFull, inc, s);
      if (static_cast<int>(lane) >= s) inc += v;
    }
    const int all = __shfl_sync(kFull, inc, 31);
    if (all == 0) return;
    const int most = __reduce_max_sync(kFull, cnt), off = inc - cnt;
    for (int i = 0; i < most; ++i)
      if (i < cnt) st.ev.map[off + i] = static_cast<uint16_t>(lane | static_cast<unsigned>(i) << 5);
    __syncwarp();
    for (int i0 = 0; i0 < all; i0 += 32) {
      const int i = i0 + static_cast<int>(lane);
      if (i < all) {
        const unsigned m = st.ev.map[i], el = m & 31u, ei = m >> 5;
        const typename Ev::Event E = st.ev.e[ei][el];
        const int code = static_cast<int>(E.code) - 1, j = code & 7, q = j >> 1;
        const R edge = R(j & 1);
        R xp[3] = {q == 0 ? edge : E.t, q == 1 ? edge : (q == 0 ? E.t : R(0)), R(0)};
        if constexpr (D == 3) {
          // tangential coordinates in axis order
          const R t2 = st.ev.t2[ei][el];
          xp[1] = q == 1 ? edge : (q == 0 ? E.t : t2);
          xp[2] = q == 2 ? edge : t2;
        }
        const R psi = RobinData<Model>::template dudn<R>(j, xp) - k.phi * RobinData<Model>::template u<R>(xp);
        const R g1 = k.phi != R(0) ? r_expm1<R>(k.phi * E.L) / k.phi : E.L;
        const int before = code >> 3;  // reflections of the same step before this one
        if (before == 0) {
          st.ev.e[ei][el].t = psi * r_exp<R>(E.y) * g1;
        } else {
          R y = r_exp<R>(st.ev.e[ei - before][el].y);
          for (int b = before; b > 0; --b) y *= r_exp<R>(k.phi * st.ev.e[ei - b][el].L);
          st.ev.e[ei][el].t = psi * y;
          st.ev.e[ei][el].code = -g1;
        }
      }
    }
    __syncwarp();
    R zr = R(0);  // a step's sum
    for (int i = 0; i < most; ++i)
      if (i < cnt) {
        const R t = st.ev.e[i][lane].t, c = st.ev.e[i][lane].code;
        if (c > R(0)) {
          Zr += zr;
          zr = t;
        } else {
          zr = fma(t, -c, zr);
        }
      }
    Zr += zr;
    cnt = 0;
    __syncwarp();
  };

  // ---- the c oldest parked units, one per lane, with the exact tests
  auto recheck = [&](int c) {
    __syncwarp();
    const bool has = static_cast<int>(lane) < c;
    // the lane's own path waits in registers
    const R X0[3] = {X[0], X[1], X[2]}, Zs0 = Zs, Zr0 = Zr, sphil0 = sphil;
    const unsigned long long id0 = id;
    const PhiloxPath pp0 = pp;
    const int32_t n0 = n;
    bool fin = false;
    if (has) {
      load(st.check, (head + static_cast<int>(lane)) & 63);
      R z[4 * D];
      uint32_t u[4];
      path_randoms<D, R>(a.rk, a.normal_tables, n, pp, z, u);
      uint4 rw = make_uint4(0u, 0u, 0u, 0u);
      R xe[3] = {R(0), R(0), R(0)};
      bool out = false, capped = false;
#pragma unroll 1
      for (int j = 0; j < 4; ++j) {
        if (D == 3 || (j & 1) == 0) rw = refl_block(n);
        out = reflect_step<Model, R>(a, k, rw, D == 2 ? 2 * (j & 1) : 0, X, Zs, Zr, sphil, n, z, u[0], xe);
        ++n;
        if (out) break;
        if (n >= a.max_steps) {
          capped = true;
          break;
        }
#pragma unroll
        for (int i = 0; i < 3 * D; ++i) z[i] = z[i + D];
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i] = u[i + 1];
      }
      fin = out || capped;
      if (fin) {
        if (capped) {
          // cap: score at the projection on the nearest absorbing face
          int jn = -1;
          R dn = R(1e30);
#pragma unroll
          for (int j = 0; j < 2 * D; ++j) {
            if ((a.mask >> j) & 1) continue;
            const R d = G::template face_dist<R>(j, X);
            if (d < dn) {
              dn = d;
              jn = j;
            }
          }
#pragma unroll
          for (int q = 0; q < D; ++q) xe[q] = X[q];
#pragma unroll
          for (int j = 0; j < 2 * D; ++j)
            if (j == jn) G::template project<R>(j, xe);
          if (a.flags) atomicOr(a.flags + node_of(a.begin + id), kNodeCapped);
          ++my_capped;
        }
        const R Yn = r_exp<R>(static_cast<R>(n) * k.cdt + sphil);
        const R Z = Model::kSource ? Zs + Zr : Zr;
        score[id] = Model::template g<R>(a.mc, xe) * Yn + Z;
        if (a.steps) a.steps[id] = capped ? -n : n;
        dump_exit_point<D>(a.exit, id, xe);
        my_steps += static_cast<unsigned long long>(n);
      }
    }
    const unsigned back = __ballot_sync(kFull, has && !fin);
    if (has && !fin) store(st.start, n_start + __popc(back & lt_mask), n, X, Zs, Zr, sphil);
    n_start += __popc(back);
    head = (head + c) & 63;
    n_check -= c;
#pragma unroll
    for (int d = 0; d < D; ++d) X[d] = X0[d];
    Zs = Zs0;
    Zr = Zr0;
    sphil = sphil0;
    id = id0;
    pp = pp0;
    n = n0;
    __syncwarp();
  };

  // ---- one unit without a branch; parked as it started if it may hold an exit
  auto advance = [&]() {
    bool park = false;
    const R X0[3] = {X[0], X[1], X[2]}, Zs0 = Zs, sphil0 = sphil;
    if (active) {
      R z[4 * D];
      uint32_t u[4];
      path_randoms<D, R>(a.rk, a.normal_tables, n, pp, z, u);
      uint4 rw[D == 3 ? 4 : 2];
#pragma unroll
      for (int j = 0; j < (D == 3 ? 4 : 2); ++j) rw[j] = refl_block(D == 3 ? n + j : n + 2 * j);
      const int cnt0 = cnt;
      bool maybe = false;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        maybe |= reflect_fast<Model, R, NR>(a, k, rw[D == 3 ? j : j >> 1], D == 2 ? 2 * (j & 1) : 0, X, Zs,
                                        sphil, n + j, z + D * j, u[j], cnt, st.ev);
      park = maybe || cnt > Ev::kCap || n > last_fast;
      if (park) cnt = cnt0;
      n += 4;
    }
    const unsigned pm = __ballot_sync(kFull, park);
    // a parked path takes its sum along; and a lane's queue holds three more, or
    // its next unit may have to be redone (four: 41.5, three: 41.3, two: 41.0 ms
    // on the case above, where it happens least)
    if (__any_sync(kFull, (park && cnt > 0) || cnt > Ev::kCap - 3)) flush();
    if (pm) {
      if (park) {
        store(st.check, (head + n_check + __popc(pm & lt_mask)) & 63, n - 4, X0, Zs0, Zr, sphil0);
        active = false;
      }
      n_check += __popc(pm);
    }
  };

  auto refill = [&](unsigned need) -> unsigned {
    const int c = __popc(need), take = c < n_start ? c : n_start;
    const int r = __popc(need & lt_mask);
    if (!active && r < take) {
      load(st.start, n_start - 1 - r);
      active = true;
    }
    n_start -= take;
    return __ballot_sync(kFull, !active);
  };

  // (as the multilevel kernel's loop: while there are paths to claim, parked
  // units go 32 together; at the end as soon as they are as many as the busy lanes)
#pragma unroll 1
  for (;;) {
    unsigned need = n_check < 32 ? __ballot_sync(kFull, !active) : 0u;
    while (need) {
      if (n_start == 0) {
        if (exhausted) break;
        claim();
        continue;
      }
      need = refill(need);
    }
    if (n_check >= 32 || (need && n_check > 0 && n_check >= 32 - __popc(need))) {
      recheck(n_check < 32 ? n_check : 32);
      continue;
    }
    if (need == kFull) break;
    advance();
  }
#pragma unroll
  for (int s2 = 16; s2 > 0; s2 >>= 1) {
    my_steps += __shfl_xor_sync(kFull, my_steps, s2);
    my_capped += __shfl_xor_sync(kFull, my_capped, s2);
    my_bad += __shfl_xor_sync(kFull, my_bad, s2);
  }
  if (lane == 0) {
    if (my_steps) atomicAdd(&a.counters[0], my_steps);
    if (my_capped) atomicAdd(&a.counters[1], my_capped);
    if (my_bad) atomicAdd(&a.counters[2], my_bad);
  }
}

template <class Model, typename R>
static pdd_status run_reflect(pdd_ctx *ctx, const double *d_nodes, int64_t n,
                              const pdd_mc_params *mc, double *d_mean, double *d_se,
                              int64_t *d_npaths, pdd_diag *diag) {
  const uint64_t N = static_cast<uint64_t>(mc->n_paths);
  const uint64_t total = static_cast<uint64_t>(n) * N;
  const uint64_t wave = std::min<uint64_t>(total, ctx->wave_max_paths);
  const size_t acc_off = 256;
  const uint64_t wave_nodes = std::min<uint64_t>(static_cast<uint64_t>(n), wave / N + 2);
  const int parts = reduce_parts(N, wave_nodes);
  const size_t part_off = align_up(acc_off + static_cast<size_t>(n) * sizeof(NodeAcc), 256);
  const size_t score_off = part_off + reduce_parts_bytes(wave_nodes, parts);
  const size_t table_off = align_up(score_off + wave * sizeof(R), 256);
  pdd_status st = ensure_scratch(ctx, table_off + (sizeof(R) == 8 ? kNormalEntries * sizeof(double2) : 0));
  if (st != PDD_OK) return st;
  char *base = static_cast<char *>(ctx->scratch);
  auto *counters = reinterpret_cast<unsigned long long *>(base);
  auto *acc = reinterpret_cast<NodeAcc *>(base + acc_off);
  R *score = reinterpret_cast<R *>(base + score_off);
  PDD_CUDA_TRY(ctx, cudaMemsetAsync(base, 0, score_off, ctx->stream));
  const ReduceParts rp = reduce_parts_at(base + part_off, wave_nodes, parts);
  int32_t *flags = diag ? diag->d_node_flags : nullptr;
  if (flags) PDD_CUDA_TRY(ctx, cudaMemsetAsync(flags, 0, static_cast<size_t>(n) * 4, ctx->stream));
  ReflectArgs a;
  std::memset(&a, 0, sizeof a);
  a.nodes = d_nodes;
  a.n_paths = N;
  a.path_offset = static_cast<uint64_t>(mc->path_offset);
  a.node_offset = static_cast<uint32_t>(mc->node_offset);
  a.cursor = counters + 4;
  a.counters = counters;
  a.score = score;
  a.rk = make_round_keys(mc->seed);
  const double sig = ctx->prob.sigma;
  a.dt = mc->dt;
  a.sdt = sig * std::sqrt(mc->dt);
  a.s2dt = sig * sig * mc->dt;
  a.cdt = constant_kill(ctx->prob.kind) * mc->dt;
  a.mask = static_cast<int32_t>(ctx->params[0]);
  a.phi = ctx->params[1];
  a.max_steps = static_cast<int32_t>(mc->max_steps);
  a.bridge = mc->bridge ? 1 : 0;
  {
    const float s2dt_f = static_cast<float>(a.s2dt);
    const float kf[8] = {static_cast<float>(a.dt), static_cast<float>(a.sdt), s2dt_f,
                         static_cast<float>(a.cdt), static_cast<float>(a.phi), 1.0f / s2dt_f,
                         static_cast<float>(-2.0 * 1.4426950408889634 / a.s2dt),
                         a.bridge ? static_cast<float>((Model::D == 2 ? 2.0 : 2.584962500721156) +
                                                       2.44140625e-4)
                                  : -INFINITY};
    for (int i = 0; i < 8; ++i) a.kf[i] = kf[i];
  }
  for (int j = 0; j < 2 * Model::D; ++j) {
    const bool hi = (j & 1) != 0;
    if (!((a.mask >> j) & 1)) continue;
    a.add[j] = 4.0f;  // (no product of two points within reach is below -2)
    a.r_face[a.n_refl] = j;
    a.rs[a.n_refl] = hi ? -1.0f : 1.0f;
    a.ro[a.n_refl] = hi ? 1.0f : 0.0f;
    a.rlo[a.n_refl] = hi ? -INFINITY : 0.0f;
    a.rhi[a.n_refl] = hi ? 1.0f : INFINITY;
    ++a.n_refl;
  }
  edge_bound(a.sdt, a.bridge != 0, std::max(1, 2 * Model::D - a.n_refl), &a.edge_c0, &a.edge_c1);
  if (sizeof(R) == 8) {
    auto *tables = reinterpret_cast<double2 *>(base + table_off);
    launch_normal_tables(tables, ctx->stream);
    PDD_CUDA_TRY(ctx, cudaGetLastError());
    a.normal_tables = tables;
  }
  a.mc = ctx->mc;
  a.flags = flags;
  constexpr int kBlock = kReflectBlock<Model, R>;
  auto kern = a.n_refl == 1 ? reflect_kernel<Model, R, 1>
            : a.n_refl == 2 ? reflect_kernel<Model, R, 2>
                            : reflect_kernel<Model, R, 0>;
  int bps = 0;
  PDD_CUDA_TRY(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, kBlock, 0));
  if (bps < 1) bps = 1;
  if (ctx->path_blocks_per_sm > 0) bps = std::min(bps, ctx->path_blocks_per_sm);
  else bps = blocks_for_paths(bps, wave, ctx->num_sms, kBlock);
  uint64_t grid = static_cast<uint64_t>(bps) * ctx->num_sms;
  grid = std::max<uint64_t>(1, std::min<uint64_t>(grid, (wave + kBlock - 1) / kBlock));
  for (uint64_t b0 = 0; b0 < total; b0 += wave) {
    const uint64_t b1 = std::min(total, b0 + wave);
    if (b0 > 0) PDD_CUDA_TRY(ctx, cudaMemsetAsync(a.cursor, 0, sizeof(unsigned long long), ctx->stream));
    a.begin = b0;
    a.end = b1;
    a.steps = (diag && diag->d_path_steps) ? diag->d_path_steps + b0 : nullptr;
    a.exit = (diag && diag->d_path_exit) ? diag->d_path_exit + b0 * Model::D : nullptr;
    const auto ev = prof_slot(ctx);
    if (ev.first) PDD_CUDA_TRY(ctx, cudaEventRecord(ev.first, ctx->stream));
    kern<<<static_cast<unsigned>(grid), kBlock, 0, ctx->stream>>>(a);
    PDD_CUDA_TRY(ctx, cudaGetLastError());
    if (ev.second) PDD_CUDA_TRY(ctx, cudaEventRecord(ev.second, ctx->stream));
    const uint64_t node_lo = b0 / N, node_hi = (b1 - 1) / N;
    reduce_wave_kernel<R><<<static_cast<unsigned>((node_hi - node_lo + 1) * parts), kReduceBlock, 0,
                            ctx->stream>>>(score, b0, b1, N, node_lo, acc, rp);
    PDD_CUDA_TRY(ctx, cudaGetLastError());
    if (diag && diag->d_path_score) {
      const uint64_t cnt = b1 - b0;
      const unsigned g = static_cast<unsigned>(std::min<uint64_t>((cnt + 255) / 256, 8192));
      widen_scores_kernel<R><<<g, 256, 0, ctx->stream>>>(score, diag->d_path_score + b0, cnt);
      PDD_CUDA_TRY(ctx, cudaGetLastError());
    }
  }
  finalize_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, ctx->stream>>>(
      acc, n, d_mean, d_se, d_npaths, flags);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  if (diag) {
    unsigned long long h[4] = {0, 0, 0, 0};
    PDD_CUDA_TRY(ctx, cudaMemcpyAsync(h, counters, sizeof h, cudaMemcpyDeviceToHost, ctx->stream));
    PDD_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    diag->path_steps = static_cast<int64_t>(h[0]);
    diag->capped = static_cast<int64_t>(h[1]);
    if (h[2]) return fail(ctx, PDD_EINVAL, "%llu paths started outside the closed domain", h[2]);
    if (h[1]) return fail(ctx, PDD_ECAP, "%llu paths hit max_steps", h[1]);
  }
  return PDD_OK;
}

pdd_status reflect_solve_impl(pdd_ctx *ctx, const double *d_nodes, int64_t n,
                              const pdd_mc_params *mc, double *d_mean, double *d_se,
                              int64_t *d_npaths, pdd_diag *diag) {
  const bool fp64 = mc->precision == PDD_FP64;
  switch (ctx->prob.kind) {
    case PDD_PROB_LAPLACE_EXPCOS:
      return fp64 ? run_reflect<LaplaceExpCos, double>(ctx, d_nodes, n, mc, d_mean, d_se, d_npaths, diag)
                  : run_reflect<LaplaceExpCos, float>(ctx, d_nodes, n, mc, d_mean, d_se, d_npaths, diag);
    case PDD_PROB_ELLIPTIC_MANUFACTURED:
      return fp64 ? run_reflect<EllipticManufactured, double>(ctx, d_nodes, n, mc, d_mean, d_se, d_npaths, diag)
                  : run_reflect<EllipticManufactured, float>(ctx, d_nodes, n, mc, d_mean, d_se, d_npaths, diag);
    default:
      return fail(ctx, PDD_EINVAL, "reflecting faces need the Laplace or the 3-D manufactured family");
  }
}

}  // namespace pdd
