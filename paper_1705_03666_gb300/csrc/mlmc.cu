// mlmc.cu -- one level of the multilevel Monte Carlo estimator (Sec. 2.1
// names Giles' multilevel method as the next acceleration of the Euler
// scheme):  E[P_L] = E[P_0] + sum_{l=1..L} E[P_l - P_{l-1}],  P_l the score of
// the Euler-Maruyama path with step dt_l = dt_0 / R^l.
//
// A lane owns one coupled pair: the fine path (step dt_l) and the coarse path
// (step dt_{l-1} = R dt_l) driven by the same Brownian motion -- the coarse
// increment is the sum of the R fine increments -- each stopping at its own
// exit (hard exit at the segment crossing, or the half-space bridge test over
// the faces within reach, exit at the end of the step).  Fine step k of pair
// p at node i reads Philox(seed, (k, p, i, 16 + l)): normals BM(w0, w1) and
// the bridge uniform U(w2); the coarse step closing a group of R fine steps
// takes the uniform of the group's last fine step (independent of every
// normal, so each path has exactly the law of the plain scheme at its step,
// and the shared uniform couples the exit decisions).  Level 0 is the plain
// scheme (fine path only).  Left point for Y and Z.  Dimensions 1 and 2.
//
// What bounds it: instruction issue.  The kernel works as the path kernel
// does (path_kernel.cuh): a unit of steps (four fine ones at level 0 and for R = 2,
// else R) runs without a branch under one conservative distance bound per
// step and walk, and a unit that may hold an exit is parked and rerun with
// the exact tests, 32 at a time.  Finished pairs are queued and added to the
// exact sums of the difference, the fine and the coarse score 32 at a time
// (no score is stored).  Four levels of 16 nodes (4e5 .. 5e4 pairs, dt 4e-3 ..
// 5e-4): 9.7 ms with the exits tested where they occur (15-17 of 32 lanes busy)
// and three reductions of 16 blocks per level; 5.5 ms now.
#include <cmath>
#include <cstring>

#include "branch_kernel.cuh"
#include "ctx.hpp"
#include "mlmc_pair.cuh"
#include "models.cuh"
#include "path_kernel.cuh"

namespace pdd {

// Threads per block (binary64 stages of four warps would not fit in the static
// shared memory).
template <typename R>
constexpr int kMlmcBlock = sizeof(R) == 4 ? 128 : 64;

struct MlmcArgs {
  const double *nodes;
  uint64_t n_paths, total;
  unsigned long long *cursor;
  unsigned long long *counters;  // [0] fine steps, [1] capped walks, [2] bad nodes
  NodeFix *fix;                  // [3][n]: difference, fine, coarse (level 0: [0] alone)
  int64_t n;
  double *dump_diff;             // [total] or null
  int32_t *steps;                // [total] or null
  double *aux;                   // [total][8] per-walk records, or null
  RoundKeys rk;
  double dtf, sdtf, s2;          // fine step, sqrt(fine step), sigma^2
  double scale;                  // of the scores in the sums (mlmc_scale)
  float edge[2][2];              // (c0, c1) of the screening bound: fine, coarse
  int32_t level, refine, max_steps, bridge;
  // x / n_paths for 32-bit x by one multiply-high and shifts
  uint32_t nt_m;
  int32_t nt_s1, nt_s2;
  ModelConst mc;
};

// Constants of one walk's step: length dt, sigma, 1 / (sigma^2 dt) and the
// screening bound's exponent scale -2 log2(e) / (sigma^2 dt) and offset
// (log2 of the face count + 2^-12 with the bridge test, -inf without).
template <typename R>
struct MlmcStep {
  R dt, sig, inv, b2, boff;
};
template <typename R>
__device__ __forceinline__ MlmcStep<R> mlmc_step_const(double dt, double s2, int faces, bool bridge) {
  MlmcStep<R> c;
  c.dt = static_cast<R>(dt);
  c.sig = static_cast<R>(sqrt(s2));
  c.inv = R(1) / (static_cast<R>(s2) * c.dt);
  c.b2 = static_cast<R>(-2.0 * 1.4426950408889634 / (s2 * dt));
  c.boff = bridge ? static_cast<R>(log2(static_cast<double>(faces)) + 2.44140625e-4)
                  : static_cast<R>(-INFINITY);
  return c;
}
// Bound on the step's crossing probability over all faces (the union bound
// at the smallest d d' m, raised by 2^(2^-12) for the exponents' rounding).
__device__ __forceinline__ float mlmc_bound(const MlmcStep<float> &c, float m) {
  return ex2_approx(fmaf(c.b2, m, c.boff));
}
__device__ __forceinline__ double mlmc_bound(const MlmcStep<double> &c, double m) {
  return exp2(c.b2 * m + c.boff);
}

// One walk of a pair (Y = 1: the 2-D families have no killing).
template <typename R>
struct MlmcWalk {
  R X[2], Z, s;  // s: the score once done
  bool done;
};

// X' of an Euler step with the (unscaled-by-sigma) increment dW.
template <class Model, typename R>
__device__ __forceinline__ void mlmc_move(const MlmcArgs &a, const MlmcStep<R> &c, const R *X, R Z,
                                          const R *dW, R *Xn, R &Zn) {
  constexpr int D = Model::D;
  R b[2] = {R(0), R(0)}, f = R(0);
  if constexpr (Model::kDrift || Model::kSource) Model::coeffs(a.mc, X, b, f);
  Xn[0] = X[0];
  Xn[1] = X[1];
#pragma unroll
  for (int k = 0; k < D; ++k) Xn[k] = X[k] + b[k] * c.dt + c.sig * dW[k];
  Zn = Model::kSource ? Z + f * R(1) * c.dt : Z;
}

// One step with the exact tests.  A lower bound on the smallest d d' (> 0: X'
// inside) and the union bound screen the step; below the bound, hard exit or
// the bridge over every face within reach.  xe: the exit point of a walk that
// ends.
template <class Model, class Geom, typename R>
__device__ __forceinline__ void mlmc_step(const MlmcArgs &a, const MlmcStep<R> &c,
                                          MlmcWalk<R> &w, const R *dW, R U, R *xe) {
  R Xn[2], Zn;
  mlmc_move<Model, R>(a, c, w.X, w.Z, dW, Xn, Zn);
  const R mn = Geom::screen_lb(w.X, Xn);
  if (!(mn > R(0)) || U < mlmc_bound(c, mn)) {
    if (!Geom::inside_closed(Xn)) {
      Geom::segment_exit(w.X, Xn, xe);
      w.s = Model::g(a.mc, xe) * R(1) + Zn;
      w.done = true;
      return;
    }
    if (a.bridge) {
      R P = R(0), pb = R(-1);
      int jb = -1;
#pragma unroll
      for (int j = 0; j < Geom::kFaces; ++j) {
        const R e = R(2) * Geom::face_dist(j, w.X) * Geom::face_dist(j, Xn) * c.inv;
        if (e < R(18)) {
          const R p = exp_fast(-e);
          P = P + p * (R(1) - P);
          if (p > pb) {
            pb = p;
            jb = j;
          }
        }
      }
      if (jb >= 0 && U < P) {
        xe[0] = Xn[0];
        xe[1] = Xn[1];
#pragma unroll
        for (int j = 0; j < Geom::kFaces; ++j)
          if (j == jb) Geom::project(j, xe);
        w.s = Model::g(a.mc, xe) * R(1) + Zn;
        w.done = true;
        return;
      }
    }
  }
  w.X[0] = Xn[0];
  w.X[1] = Xn[1];
  w.Z = Zn;
}
template <class Model, class Geom, typename R>
__device__ __forceinline__ void mlmc_cap(const MlmcArgs &a, MlmcWalk<R> &w, R *xe) {
  xe[0] = w.X[0];
  xe[1] = w.X[1];
  const int jn = Geom::nearest_face(w.X);
#pragma unroll
  for (int j = 0; j < Geom::kFaces; ++j)
    if (j == jn) Geom::project(j, xe);
  w.s = Model::g(a.mc, xe) * R(1) + w.Z;
  w.done = true;
}

// The same step without exit tests: returns whether it may be an exit (the
// bound of path_step_args on e e', e the distance bound of X, advanced).
template <class Model, class Geom, typename R>
__device__ __forceinline__ bool mlmc_fast(const MlmcArgs &a, const MlmcStep<R> &c, const float *edge,
                                          MlmcWalk<R> &w, const R *dW, float logu, float &e) {
  R Xn[2], Zn;
  mlmc_move<Model, R>(a, c, w.X, w.Z, dW, Xn, Zn);
  const float en = path_edge<Geom, R>(Xn);
  const bool maybe = !(logu >= fmaf(edge[1], e * en, edge[0]));
  e = en;
  w.X[0] = Xn[0];
  w.X[1] = Xn[1];
  w.Z = Zn;
  return maybe;
}

// Pairs at the start of a unit, N of them, and finished pairs, in shared memory.
template <typename R, int N>
struct PairStash {
  unsigned long long id[N];
  uint32_t w0[N], w1[N];
  uint32_t state[N];           // PairState
  R fx[2][N], fz[N], cx[2][N], cz[N];  // a walk that is done keeps its score in its z
};
template <typename R>
struct MlmcStage {
  PairStash<R, 96> start;      // (capacities: see path_kernel.cuh, ForwardStage)
  PairStash<R, 64> check;
  unsigned long long did[64];
  R df[64], dc[64];
  // running sums of the difference, the fine and the coarse score (FixAccum)
  long long sum[3][32];
  uint64_t sum_node[3];
};

__device__ __forceinline__ uint64_t mlmc_node(const MlmcArgs &a, uint64_t g) {
  if (a.total <= 0xffffffffull) {
    const uint32_t x = static_cast<uint32_t>(g), t = __umulhi(a.nt_m, x);
    return (t + ((x - t) >> a.nt_s1)) >> a.nt_s2;
  }
  return g / a.n_paths;
}

// kMode 0: level 0 (no coarse walk), units of four steps; 2: R = 2, units of
// four fine and two coarse steps; 1: any R, units of R fine steps and one
// coarse step.
template <class Model, class Geom, typename R, int kMode>
__global__ void __launch_bounds__(kMlmcBlock<R>, sizeof(R) == 4 ? (Model::kDrift ? 4 : 6) : 4)
mlmc_kernel(const __grid_constant__ MlmcArgs a) {
  constexpr int D = Model::D;
  __shared__ MlmcStage<R> stage_all[kMlmcBlock<R> / 32];
  MlmcStage<R> &st = stage_all[threadIdx.x >> 5];
  const unsigned lane = threadIdx.x & 31u, lt_mask = (1u << lane) - 1u;
  const R sdtf = static_cast<R>(a.sdtf);
  const MlmcStep<R> cf = mlmc_step_const<R>(a.dtf, a.s2, Geom::kFaces, a.bridge != 0);
  const MlmcStep<R> cc = mlmc_step_const<R>(static_cast<double>(static_cast<R>(a.dtf) *
                                                                static_cast<R>(a.refine)),
                                            a.s2, Geom::kFaces, a.bridge != 0);
  const int unit = kMode == 1 ? a.refine : 4;
  const int32_t last_fast = a.max_steps - unit - 1;
  MlmcWalk<R> fw{}, cw{};
  float ef = 0.f, ec = 0.f;
  PhiloxPath pp{0, 0, 16u + static_cast<uint32_t>(a.level)};
  unsigned long long id = 0;
  int32_t k = 0;
  bool active = false, exhausted = false;
  int n_start = 0, n_check = 0, head = 0, n_done = 0;  // warp-uniform
  unsigned long long my_steps = 0, my_capped = 0, my_bad = 0;
  for (int p = 0; p < 3; ++p) {
    st.sum[p][lane] = 0;
    if (lane == 0) st.sum_node[p] = ~0ull;
  }

  auto load = [&](const auto &q, int i) {
    id = q.id[i];
    pp.r0_w0 = q.w0[i];
    pp.r0_w1 = q.w1[i];
    const PairState p = pair_unpack(q.state[i], unit);
    k = p.steps;
    fw.done = p.fine_done;
    cw.done = p.coarse_done;
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      fw.X[d] = q.fx[d][i];
      cw.X[d] = q.cx[d][i];
    }
    fw.Z = fw.s = q.fz[i];
    cw.Z = cw.s = q.cz[i];
    ef = path_edge<Geom, R>(fw.X);
    ec = path_edge<Geom, R>(cw.X);
  };
  auto store = [&](auto &q, int i, int32_t k0, const MlmcWalk<R> &f, const MlmcWalk<R> &c) {
    q.id[i] = id;
    q.w0[i] = pp.r0_w0;
    q.w1[i] = pp.r0_w1;
    q.state[i] = pair_pack(k0, unit, f.done, c.done);
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      q.fx[d][i] = f.X[d];
      q.cx[d][i] = c.X[d];
    }
    q.fz[i] = f.done ? f.s : f.Z;
    q.cz[i] = c.done ? c.s : c.Z;
  };
  // the normals and the bridge uniform of fine step kk
  auto randoms = [&](int32_t kk, R *dW, R &U) {
    const uint4 w = philox10_path(static_cast<uint32_t>(kk), pp, a.rk);
    R z0, z1;
    box_muller<R>(w.x, w.y, z0, z1);
    dW[0] = sdtf * z0;
    dW[1] = D > 1 ? sdtf * z1 : R(0);
    U = unif<R>(w.z);
  };
  // finished pairs (first cnt of the queue from `from`) into the sums
  const R scale = static_cast<R>(a.scale);
  auto commit = [&](int from, int cnt) {
    __syncwarp();
    const bool has = static_cast<int>(lane) < cnt;
    R f = R(0), c = R(0), df = R(0);
    uint64_t node = 0;
    if (has) {
      f = st.df[from + lane];
      c = st.dc[from + lane];
      df = kMode == 0 ? f : f - c;
      const unsigned long long q = st.did[from + lane];
      node = mlmc_node(a, q);
      if (a.dump_diff) a.dump_diff[q] = static_cast<double>(df);
    }
#pragma unroll 1
    for (int p = 0; p < (kMode == 0 ? 1 : 3); ++p) {
      FixAccum acc;
      acc.v = st.sum[p][lane];
      acc.node = st.sum_node[p];
      __syncwarp();
      acc.add<R>(a.fix + p * a.n, has, node, scale * (p == 0 ? df : (p == 1 ? f : c)), false);
      st.sum[p][lane] = acc.v;
      if (lane == 0) st.sum_node[p] = acc.node;
    }
    __syncwarp();
  };
  // lanes with `fin` queue their pair (id, f, c)
  auto finish = [&](bool fin, R f, R c) {
    const unsigned m = __ballot_sync(kFull, fin);
    if (!m) return;
    if (fin) {
      const int i = n_done + __popc(m & lt_mask);
      st.did[i] = id;
      st.df[i] = f;
      st.dc[i] = c;
    }
    n_done += __popc(m);
    if (n_done >= 32) {
      n_done -= 32;
      commit(n_done, 32);
    }
  };
  auto aux_walk = [&](unsigned long long q, int which, R s, int32_t steps, const R *xe) {
    if (!a.aux) return;
    double *o = a.aux + 8 * q;
    o[which] = static_cast<double>(s);
    o[2 + which] = static_cast<double>(steps);
    o[4 + 2 * which] = static_cast<double>(xe[0]);
    o[5 + 2 * which] = static_cast<double>(xe[1]);
  };

  // ---- claim 32 pairs into the empty stash; starts on the boundary or outside
  // are finished at once
  auto claim = [&]() {
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(a.cursor, 32ull);
    base = __shfl_sync(kFull, base, 0);
    if (base + 32 >= a.total) exhausted = true;
    const unsigned long long q = base + lane;
    const bool has = q < a.total;
    bool in = false;
    MlmcWalk<R> f{}, c{};
    const unsigned long long id0 = id;
    const PhiloxPath pp0 = pp;
    R g0 = R(0);
    if (has) {
      const uint64_t node = mlmc_node(a, q);
      pp = philox_path(static_cast<uint32_t>(q - node * a.n_paths), static_cast<uint32_t>(node), pp.tag,
                       a.rk);
      f.X[0] = static_cast<R>(a.nodes[node * D]);
      f.X[1] = D > 1 ? static_cast<R>(a.nodes[node * D + (D > 1 ? 1 : 0)]) : R(0);
      f.Z = R(0);
      f.done = false;
      c = f;
      c.done = kMode == 0;
      id = q;
      const bool closed = Geom::inside_closed(f.X);
      in = closed && Geom::inside_open(f.X);
      if (!in) {
        g0 = closed ? Model::g(a.mc, f.X) : R(NAN);
        if (!closed) ++my_bad;
        if (a.steps) a.steps[q] = 0;
        aux_walk(q, 0, g0, 0, f.X);
        const R zero[2] = {R(0), R(0)};
        aux_walk(q, 1, kMode == 0 ? R(0) : g0, 0, kMode == 0 ? zero : f.X);
      }
    }
    finish(has && !in, g0, kMode == 0 ? R(0) : g0);
    const unsigned im = __ballot_sync(kFull, in);
    if (in) store(st.start, __popc(im & lt_mask), 0, f, c);
    id = id0;
    pp = pp0;
    __syncwarp();
    n_start = __popc(im);
  };

  // ---- the cnt oldest parked units, one per lane, with the exact tests
  auto recheck = [&](int cnt) {
    __syncwarp();
    const bool has = static_cast<int>(lane) < cnt;
    // the lane's own pair waits in registers
    const MlmcWalk<R> f0 = fw, c0 = cw;
    const float ef0 = ef, ec0 = ec;
    const unsigned long long id0 = id;
    const PhiloxPath pp0 = pp;
    const int32_t k0 = k;
    bool fin = false;
    if (has) {
      load(st.check, (head + static_cast<int>(lane)) & 63);
      R dWc[2] = {R(0), R(0)};
      int kc = 0;
#pragma unroll 1
      for (int j = 0; j < unit; ++j) {
        R dW[2], U, xe[2];
        randoms(k, dW, U);
        if (!fw.done) {
          mlmc_step<Model, Geom, R>(a, cf, fw, dW, U, xe);
          if (fw.done) aux_walk(id, 0, fw.s, k + 1, xe);
        }
        ++k;
        if constexpr (kMode != 0) {
          dWc[0] += dW[0];
          dWc[1] += dW[1];
          if (++kc == a.refine) {
            if (!cw.done) {
              mlmc_step<Model, Geom, R>(a, cc, cw, dWc, U, xe);
              if (cw.done) aux_walk(id, 1, cw.s, k / a.refine, xe);
            }
            dWc[0] = dWc[1] = R(0);
            kc = 0;
          }
        }
        fin = fw.done && cw.done;
        if (!fin && k >= a.max_steps) {
          if (!fw.done) {
            mlmc_cap<Model, Geom, R>(a, fw, xe);
            aux_walk(id, 0, fw.s, -k, xe);
            ++my_capped;
          }
          if (!cw.done) {
            mlmc_cap<Model, Geom, R>(a, cw, xe);
            aux_walk(id, 1, cw.s, -(k / a.refine), xe);
            ++my_capped;
          }
          fin = true;
        }
        if (fin) break;
      }
      if (fin) {
        if (a.steps) a.steps[id] = k;
        if constexpr (kMode == 0) {
          const R zero[2] = {R(0), R(0)};
          aux_walk(id, 1, R(0), 0, zero);
        }
        my_steps += static_cast<unsigned long long>(k);
      }
    }
    const unsigned back = __ballot_sync(kFull, has && !fin);
    if (has && !fin) store(st.start, n_start + __popc(back & lt_mask), k, fw, cw);
    n_start += __popc(back);
    finish(has && fin, fw.s, kMode == 0 ? R(0) : cw.s);
    head = (head + cnt) & 63;
    n_check -= cnt;
    fw = f0;
    cw = c0;
    ef = ef0;
    ec = ec0;
    id = id0;
    pp = pp0;
    k = k0;
    __syncwarp();
  };

  // ---- one unit without exit tests; parked as it started if it may hold one
  auto advance = [&]() {
    bool park = false;
    const MlmcWalk<R> f0 = fw, c0 = cw;
    if (active) {
      bool mf = false, mcs = false;
      if constexpr (kMode == 1) {
        R dWc[2] = {R(0), R(0)}, U = R(0);
#pragma unroll 1
        for (int j = 0; j < unit; ++j) {
          R dW[2];
          randoms(k + j, dW, U);
          mf |= mlmc_fast<Model, Geom, R>(a, cf, a.edge[0], fw, dW, unif_log_bits(static_cast<float>(U)), ef);
          dWc[0] += dW[0];
          dWc[1] += dW[1];
        }
        mcs |= mlmc_fast<Model, Geom, R>(a, cc, a.edge[1], cw, dWc, unif_log_bits(static_cast<float>(U)), ec);
      } else {
        R dW[4][2], U[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) randoms(k + j, dW[j], U[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          mf |= mlmc_fast<Model, Geom, R>(a, cf, a.edge[0], fw, dW[j],
                                          unif_log_bits(static_cast<float>(U[j])), ef);
          if constexpr (kMode == 2) {
            if (j & 1) {
              R dWc[2] = {R(0), R(0)};
              dWc[0] += dW[j - 1][0];
              dWc[1] += dW[j - 1][1];
              dWc[0] += dW[j][0];
              dWc[1] += dW[j][1];
              mcs |= mlmc_fast<Model, Geom, R>(a, cc, a.edge[1], cw, dWc,
                                               unif_log_bits(static_cast<float>(U[j])), ec);
            }
          }
        }
      }
      // a walk that is done keeps its state (its score)
      if (f0.done) fw = f0;
      if (c0.done) cw = c0;
      park = (mf && !f0.done) || (mcs && !c0.done) || k > last_fast;
      k += unit;
    }
    const unsigned pm = __ballot_sync(kFull, park);
    if (pm) {
      if (park) {
        store(st.check, (head + n_check + __popc(pm & lt_mask)) & 63, k - unit, f0, c0);
        active = false;
      }
      n_check += __popc(pm);
    }
  };

  auto refill = [&](unsigned need) -> unsigned {
    const int cnt = __popc(need), take = cnt < n_start ? cnt : n_start;
    const int r = __popc(need & lt_mask);
    if (!active && r < take) {
      load(st.start, n_start - 1 - r);
      active = true;
    }
    n_start -= take;
    return __ballot_sync(kFull, !active);
  };

  // One loop (a second copy of its parts for the wave's end, as the path
  // kernel has, cost instruction fetch here): while there are pairs to claim,
  // parked units go 32 together; at the end as soon as they are as many as the
  // busy lanes.
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
  if (n_done > 0) commit(0, n_done);
  __syncwarp();
  for (int p = 0; p < 3; ++p) {
    FixAccum acc;
    acc.v = st.sum[p][lane];
    acc.node = st.sum_node[p];
    acc.flush(a.fix + p * a.n);
  }
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

// fix planes: [3][n] (level 0: the fine score alone), of scores times 2^e; var =
// M2 / (count - 1).  A node outside the closed domain has no scores: NaN mean,
// zero variance and zero walk means.
static __global__ void mlmc_finalize_kernel(const NodeFix *fix, int64_t n, int level, int e, double *mean,
                                            double *var, double *fine_mean, double *coarse_mean) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  double m[3], m2[3];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    fix_moments(fix[(level ? p : 0) * n + i], &m[p], &m2[p]);
    m[p] = scalbn(m[p], -e);
  }
  const long long cnt = fix[i].n;
  mean[i] = m[0];
  var[i] = cnt > 1 ? scalbn(m2[0] / (static_cast<double>(cnt) - 1.0), -2 * e) : 0.0;
  if (fine_mean) fine_mean[i] = cnt > 0 ? m[1] : 0.0;
  if (coarse_mean) coarse_mean[i] = cnt > 0 && level ? m[2] : 0.0;
}

// The exponent e of the power of two that the scores of a level are multiplied
// with before they go to the exact sums (which hold |s| < 2^30 in steps of
// 2^-60), so that the range fits the problem's data: |g| <= e on the square, <=
// sum |theta| for the Fourier data, whose source (1) adds at most the time of
// max_steps steps (twice that in rounded additions); a difference is at most two
// scores; and a factor of two for the rounding of g.  The same sums with e = 0
// made a node with a score of 2^30 NaN and dropped squares below 2^-60.
static int mlmc_scale(const pdd_ctx *ctx, const pdd_mlmc_params *mp, double dtf) {
  double bound = 2.7182818284590452;
  if (ctx->prob.kind == PDD_PROB_POISSON_FOURIER) {
    bound = 2.0 * dtf * static_cast<double>(mp->max_steps);
    for (int i = 0; i < 64; ++i) bound += std::fabs(ctx->params[static_cast<size_t>(i)]);
  }
  if (!std::isfinite(bound)) return 0;
  int e = 0;
  std::frexp(4.0 * bound, &e);  // 4 bound < 2^e
  // (binary32 scores end below 2^128, binary64 ones below 2^1024)
  return std::max(mp->precision == PDD_FP64 ? -1000 : -100, std::min(60, 30 - e));
}

// The most faces within bridge reach of one step of standard deviation s whose
// Brownian increment is at most q s long: a face within reach has d d' < 9 s^2
// and |d - d'| <= q s, so both ends lie within r = (q + sqrt(q^2 + 36)) s / 2
// of it.
template <class Geom>
static int mlmc_reach(double s, double q) {
  const double r = 0.5 * (q + std::sqrt(q * q + 36.0)) * s;
  return r < 0.25 ? 2 : Geom::kFaces;
}

// Scratch of one level: 256 bytes of counters, then the sums.
constexpr size_t kMlmcFixOff = 256;
constexpr size_t kMlmcApart = size_t(1) << 30;  // most scratch for levels side by side
static size_t mlmc_bytes(int64_t n) {
  return align_up(kMlmcFixOff + 3 * static_cast<size_t>(n) * sizeof(NodeFix), 256);
}

// One level's launches on `stream`, with mlmc_bytes(n) bytes at base.
template <class Model, class Geom, typename R>
static pdd_status run_mlmc(pdd_ctx *ctx, cudaStream_t stream, char *base, const double *d_nodes,
                           int64_t n, const pdd_mlmc_params *mp, double *d_mean, double *d_var,
                           double *d_fine, double *d_coarse, pdd_diag *diag) {
  const uint64_t N = static_cast<uint64_t>(mp->n_paths);
  const uint64_t total = static_cast<uint64_t>(n) * N;
  auto *counters = reinterpret_cast<unsigned long long *>(base);
  PDD_CUDA_TRY(ctx, cudaMemsetAsync(base, 0, mlmc_bytes(n), stream));
  MlmcArgs a;
  std::memset(&a, 0, sizeof a);
  a.nodes = d_nodes;
  a.n_paths = N;
  a.total = total;
  a.cursor = counters + 4;
  a.counters = counters;
  a.fix = reinterpret_cast<NodeFix *>(base + kMlmcFixOff);
  a.n = n;
  a.rk = make_round_keys(mp->seed);
  a.dtf = mp->dt0 / std::pow(static_cast<double>(mp->refine), static_cast<double>(mp->level));
  a.sdtf = std::sqrt(a.dtf);
  a.s2 = ctx->prob.sigma * ctx->prob.sigma;
  const int scale_e = mlmc_scale(ctx, mp, a.dtf);
  a.scale = std::ldexp(1.0, scale_e);
  a.level = mp->level;
  a.refine = mp->refine;
  a.max_steps = static_cast<int32_t>(mp->max_steps);
  a.bridge = mp->bridge ? 1 : 0;
  // Box-Muller radii stay below 5.77; a coarse increment is the sum of R fine ones
  const double sf = ctx->prob.sigma * a.sdtf, rr = std::sqrt(static_cast<double>(mp->refine));
  edge_bound(sf, a.bridge != 0, mlmc_reach<Geom>(sf, 5.77), &a.edge[0][0], &a.edge[0][1]);
  edge_bound(sf * rr, a.bridge != 0, mlmc_reach<Geom>(sf * rr, 5.77 * rr), &a.edge[1][0], &a.edge[1][1]);
  branch_divisor(N < (uint64_t(1) << 32) ? static_cast<uint32_t>(N) : 0xffffffffu, &a.nt_m, &a.nt_s1,
                 &a.nt_s2);
  a.mc = ctx->mc;
  if (diag) {
    a.dump_diff = diag->d_path_score;
    a.steps = diag->d_path_steps;
    a.aux = diag->d_path_aux;
  }
  auto kern = mp->level == 0 ? mlmc_kernel<Model, Geom, R, 0>
            : mp->refine == 2 ? mlmc_kernel<Model, Geom, R, 2>
                              : mlmc_kernel<Model, Geom, R, 1>;
  int bps = 0;
  PDD_CUDA_TRY(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, kMlmcBlock<R>, 0));
  if (bps < 1) bps = 1;
  if (ctx->path_blocks_per_sm > 0) bps = std::min(bps, ctx->path_blocks_per_sm);
  uint64_t grid = static_cast<uint64_t>(bps) * ctx->num_sms;
  grid = std::max<uint64_t>(1, std::min<uint64_t>(grid, (total + kMlmcBlock<R> - 1) / kMlmcBlock<R>));
  const auto ev = prof_slot(ctx);
  if (ev.first) PDD_CUDA_TRY(ctx, cudaEventRecord(ev.first, stream));
  kern<<<static_cast<unsigned>(grid), kMlmcBlock<R>, 0, stream>>>(a);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  if (ev.second) PDD_CUDA_TRY(ctx, cudaEventRecord(ev.second, stream));
  mlmc_finalize_kernel<<<static_cast<unsigned>((n + kFinalizeBlock - 1) / kFinalizeBlock), kFinalizeBlock, 0, stream>>>(
      a.fix, n, mp->level, scale_e, d_mean, d_var, d_fine, d_coarse);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  return PDD_OK;
}

// Steps and capped walks of a level from its counters (synchronises).
static pdd_status mlmc_counts(pdd_ctx *ctx, const char *base, pdd_diag *diag) {
  unsigned long long h[4] = {0, 0, 0, 0};
  PDD_CUDA_TRY(ctx, cudaMemcpyAsync(h, base, sizeof h, cudaMemcpyDeviceToHost, ctx->stream));
  PDD_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
  diag->path_steps = static_cast<int64_t>(h[0]);
  diag->capped = static_cast<int64_t>(h[1]);
  if (h[2]) return fail(ctx, PDD_EINVAL, "%llu pairs started outside the closed domain", h[2]);
  if (h[1]) return fail(ctx, PDD_ECAP, "%llu walks hit max_steps", h[1]);
  return PDD_OK;
}

static pdd_status mlmc_check(pdd_ctx *ctx, const double *d_nodes, int64_t n,
                             const pdd_mlmc_params *mp, const double *d_mean, const double *d_var) {
  if (!mp) return fail(ctx, PDD_EINVAL, "params is NULL");
  if (n < 0 || n > (int64_t(1) << 32)) return fail(ctx, PDD_EINVAL, "n out of range");
  if (mp->n_paths < 1 || mp->n_paths > (int64_t(1) << 32))
    return fail(ctx, PDD_EINVAL, "n_paths out of range");
  if (!(mp->dt0 > 0.0) || !std::isfinite(mp->dt0)) return fail(ctx, PDD_EINVAL, "dt0 must be > 0");
  if (mp->level < 0 || mp->level > 12 || mp->refine < 2 || mp->refine > 16)
    return fail(ctx, PDD_EINVAL, "level in [0, 12], refine in [2, 16]");
  if (mp->max_steps < 1 || mp->max_steps > 2147483647LL)
    return fail(ctx, PDD_EINVAL, "max_steps out of range");
  if (mp->precision != PDD_FP32 && mp->precision != PDD_FP64)
    return fail(ctx, PDD_EINVAL, "unknown precision");
  if (ctx->prob.sigma * ctx->prob.sigma * mp->dt0 > 1.0 / 36.0)
    return fail(ctx, PDD_EINVAL, "sigma^2 dt0 must be <= 1/36");
  if (reflect_mask(ctx) != 0) return fail(ctx, PDD_EINVAL, "the multilevel solve covers Dirichlet data");
  if (n > 0 && (!d_nodes || !d_mean || !d_var)) return fail(ctx, PDD_EINVAL, "null buffer");
  if (ctx->prob.kind != PDD_PROB_LAPLACE_EXPCOS && ctx->prob.kind != PDD_PROB_POISSON_FOURIER)
    return fail(ctx, PDD_EINVAL, "the multilevel solve covers the 2-D families");
  return PDD_OK;
}

static pdd_status mlmc_launch(pdd_ctx *ctx, cudaStream_t stream, char *base, const double *d_nodes,
                              int64_t n, const pdd_mlmc_params *mp, double *d_mean, double *d_var,
                              double *d_fine, double *d_coarse, pdd_diag *diag) {
  const bool fp64 = mp->precision == PDD_FP64;
#define PDD_MLMC(M, G)                                                                             \
  (fp64 ? run_mlmc<M, G, double>(ctx, stream, base, d_nodes, n, mp, d_mean, d_var, d_fine, d_coarse, diag) \
        : run_mlmc<M, G, float>(ctx, stream, base, d_nodes, n, mp, d_mean, d_var, d_fine, d_coarse, diag))
  if (ctx->prob.kind == PDD_PROB_POISSON_FOURIER) return PDD_MLMC(PoissonFourier, Box<2>);
  if (ctx->prob.geometry == PDD_GEOM_L_SHAPE) return PDD_MLMC(LaplaceExpCos, LShape);
  return PDD_MLMC(LaplaceExpCos, Box<2>);
#undef PDD_MLMC
}

pdd_status mlmc_level_impl(pdd_ctx *ctx, const double *d_nodes, int64_t n, const pdd_mlmc_params *mp,
                           double *d_mean, double *d_var, double *d_fine, double *d_coarse,
                           pdd_diag *diag) {
  pdd_status st = mlmc_check(ctx, d_nodes, n, mp, d_mean, d_var);
  if (st != PDD_OK) return st;
  if (diag) {
    diag->path_steps = 0;
    diag->capped = 0;
  }
  if (n == 0) return PDD_OK;
  PDD_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  st = ensure_scratch(ctx, mlmc_bytes(n));
  if (st != PDD_OK) return st;
  char *base = static_cast<char *>(ctx->scratch);
  st = mlmc_launch(ctx, ctx->stream, base, d_nodes, n, mp, d_mean, d_var, d_fine, d_coarse, diag);
  if (st != PDD_OK || !diag) return st;
  return mlmc_counts(ctx, base, diag);
}

// The multilevel estimate from its levels, per node, in level order:
// mean = sum_l mean_l, se = sqrt(sum_l var_l / N_l) (independent levels).
struct LevelCounts {
  double n[13];
};
static __global__ void mlmc_combine_kernel(const double *lmean, const double *lvar, int64_t n,
                                           int32_t L, LevelCounts N, double *mean, double *se) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  double m = 0.0, v = 0.0;
  for (int l = 0; l < L; ++l) {
    m += lmean[static_cast<int64_t>(l) * n + i];
    v += lvar[static_cast<int64_t>(l) * n + i] / N.n[l];
  }
  mean[i] = m;
  se[i] = sqrt(v);
}

pdd_status mlmc_solve_impl(pdd_ctx *ctx, const double *d_nodes, int64_t n,
                           const pdd_mlmc_params *mp, int32_t n_levels,
                           const int64_t *h_n_per_level, double *d_mean, double *d_se,
                           double *d_level_mean, double *d_level_var, pdd_diag *diag) {
  if (!mp || !h_n_per_level) return fail(ctx, PDD_EINVAL, "params or path counts NULL");
  if (n_levels < 1 || n_levels > 13) return fail(ctx, PDD_EINVAL, "n_levels must be in [1, 13]");
  for (int l = 0; l < n_levels; ++l)
    if (h_n_per_level[l] < 1) return fail(ctx, PDD_EINVAL, "level %d has no pairs", l);
  if (n < 0 || n > (int64_t(1) << 32)) return fail(ctx, PDD_EINVAL, "n out of range");
  if (diag) {
    diag->path_steps = 0;
    diag->capped = 0;
  }
  if (n == 0) return PDD_OK;
  if (!d_mean || !d_se) return fail(ctx, PDD_EINVAL, "null buffer");
  PDD_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  // level means and variances: the caller's buffers, or the auxiliary buffer
  // (the level calls use the context scratch themselves)
  double *lm = d_level_mean, *lv = d_level_var;
  const size_t plane = static_cast<size_t>(n) * n_levels * sizeof(double);
  if (!lm || !lv) {
    const pdd_status st = ensure_aux(ctx, 2 * plane);
    if (st != PDD_OK) return st;
    if (!lm) lm = static_cast<double *>(ctx->aux);
    if (!lv) lv = reinterpret_cast<double *>(static_cast<char *>(ctx->aux) + plane);
  }
  // every level on its own scratch, the levels over the context's stream and
  // its side streams in turn, so that the end of one level's launch (lanes idle
  // while its last pairs finish) is filled by the next (four levels of 16 nodes:
  // 5.9 ms one after another, 5.45 ms so; a share of the blocks for each level
  // measured 10 ms); the finest, with the longest walks, first (five levels of 4
  // nodes and 20000 pairs: 0.88 -> 0.83 ms)
  pdd_mlmc_params lps[13];
  LevelCounts N{};
  for (int l = 0; l < n_levels; ++l) {
    lps[l] = *mp;
    lps[l].level = l;
    lps[l].n_paths = h_n_per_level[l];
    N.n[l] = static_cast<double>(h_n_per_level[l]);
    const pdd_status st = mlmc_check(ctx, d_nodes, n, &lps[l], lm, lv);
    if (st != PDD_OK) return st;
  }
  // (more than kMlmcApart bytes for all of them: the levels follow one another on
  // one level's scratch, or many nodes times many levels would not fit the device)
  const size_t per = mlmc_bytes(n);
  const bool apart = per <= kMlmcApart / static_cast<size_t>(n_levels);
  pdd_status st = ensure_scratch(ctx, apart ? per * n_levels : per);
  if (st != PDD_OK) return st;
  st = ensure_side_streams(ctx);
  if (st != PDD_OK) return st;
  char *base = static_cast<char *>(ctx->scratch);
  pdd_status worst = PDD_OK;
  int64_t steps = 0, capped = 0;
  auto count = [&](int l) -> pdd_status {
    pdd_diag ld{};
    const pdd_status s = mlmc_counts(ctx, base + (apart ? per * l : 0), &ld);
    if (s == PDD_ECAP) worst = PDD_ECAP;
    steps += ld.path_steps;
    capped += ld.capped;
    return s == PDD_ECAP ? PDD_OK : s;
  };
  // (timed launches follow one another on the context's stream: side by side,
  // each would count the others' time as its own)
  const int side = ctx->profiling || !apart ? 0 : std::min(n_levels - 1, 3);
  PDD_CUDA_TRY(ctx, cudaEventRecord(ctx->batch_fork, ctx->stream));
  for (int k = 0; k < side; ++k)
    PDD_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->batch_side[k], ctx->batch_fork, 0));
  pdd_status launched = PDD_OK;
  for (int q = 0; q < n_levels && launched == PDD_OK; ++q) {
    const int l = n_levels - 1 - q;
    cudaStream_t s = side == 0 || q % 4 == 0 ? ctx->stream : ctx->batch_side[q % 4 - 1];
    launched = mlmc_launch(ctx, s, base + (apart ? per * l : 0), d_nodes, n, &lps[l],
                           lm + static_cast<size_t>(l) * n, lv + static_cast<size_t>(l) * n, nullptr,
                           nullptr, nullptr);
    if (diag && !apart && launched == PDD_OK) launched = count(l);
  }
  // (joined also after a failed launch: nothing of this call runs on past it)
  for (int k = 0; k < side; ++k) {
    PDD_CUDA_TRY(ctx, cudaEventRecord(ctx->batch_join[k], ctx->batch_side[k]));
    PDD_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->stream, ctx->batch_join[k], 0));
  }
  if (launched != PDD_OK) return launched;
  for (int l = 0; diag && apart && l < n_levels; ++l) {
    st = count(l);
    if (st != PDD_OK) return st;
  }
  mlmc_combine_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, ctx->stream>>>(
      lm, lv, n, n_levels, N, d_mean, d_se);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  if (diag) {
    diag->path_steps = steps;
    diag->capped = capped;
    if (worst == PDD_ECAP) return fail(ctx, PDD_ECAP, "%lld walks hit max_steps",
                                       static_cast<long long>(capped));
  }
  return PDD_OK;
}

}  // namespace pdd
