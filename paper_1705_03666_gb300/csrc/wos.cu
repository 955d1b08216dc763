// wos.cu -- Walk on Spheres for the Laplace problem (Eq. 1.1), the scheme
// Sec. 2.1 recommends for stopped Brownian motion when it applies: from x the
// walk jumps to a uniform point on the largest circle inside the domain
// (radius d(x) = distance to the nearest face) and stops when d(x) <= eps,
// scoring g at the projection on that face.  No time step; the bias is
// O(eps) and a path takes O(log 1/eps) jumps.
//
// What bounds it: instruction issue, and the lanes that an instruction finds
// idle (a walk lasts about a dozen jumps).  So a lane runs four jumps, one
// Philox block (block n/4 of stream tag 2), between looks at its warp; starts
// are set up 32 at a time into a per-warp stash, and stopped walks are parked
// and scored 32 at a time straight into the exact per-node sums (nodefix.cuh):
// no score is stored and no reduction follows.  16 nodes x 10^6 walks at
// eps = 10^-4: 1.41 ms with a jump per loop trip (a Philox block for a quarter
// of the lanes at every trip, 17 of 32 lanes busy) and a reduction of 16
// blocks (0.19 ms); 0.63 ms now (28.5 of 32 lanes).
#include <cmath>
#include <cstring>

#include "branch_kernel.cuh"
#include "ctx.hpp"
#include "nodefix.cuh"

namespace pdd {

constexpr int kWosBlock = 128;
constexpr uint64_t kWosClaim = 256;  // most walks claimed per atomic

struct WosArgs {
  const double *nodes;
  uint64_t n_paths, path_offset, total;
  unsigned long long *cursor;
  unsigned long long *counters;  // [0] jumps, [1] capped, [2] bad nodes
  NodeFix *fix;                  // [n] exact per-node sums
  double *dump_score;            // [total] or null
  int32_t *steps;                // [total] or null
  double *exit;                  // [total][2] stopping points (projected), or null
  RoundKeys rk;
  double eps;
  int32_t max_steps;
  uint32_t claim;                // walks claimed per atomic (a multiple of 32)
  // x / n_paths for 32-bit x by one multiply-high and shifts
  uint32_t nt_m;
  int32_t nt_s1, nt_s2;
  ModelConst mc;
};

// A jump of length d in direction 2 pi U.
__device__ __forceinline__ void wos_dir(float U, float &cx, float &sy) {
  const float th = 6.28318530717958648f * (U - 0.5f);  // centred: cos(2pi U) = -cos(th)
  cx = -cos_approx(th);
  sy = -sin_approx(th);
}
__device__ __forceinline__ void wos_dir(double U, double &cx, double &sy) {
  sincospi(2.0 * U, &sy, &cx);
}

// Distance to the nearest face; its index only where a walk stops.
template <class Geom, typename R>
__device__ __forceinline__ R wos_dist(const R *x) {
  R db = Geom::template face_dist<R>(0, x);
#pragma unroll
  for (int j = 1; j < Geom::kFaces; ++j) db = fmin(db, Geom::template face_dist<R>(j, x));
  return db;
}
template <class Geom, typename R>
__device__ __forceinline__ void wos_project(int jb, R *x) {
#pragma unroll
  for (int j = 0; j < Geom::kFaces; ++j)
    if (j == jb) Geom::template project<R>(j, x);
}

template <typename R>
struct WosStage {
  // starts (a stack of at most 32)
  unsigned long long id[32];
  uint32_t w0[32], w1[32];
  R x[2][32];
  // stopped walks (at most 63)
  unsigned long long eid[64];
  int32_t en[64];   // jumps
  R ex[2][64];
};

// Node of global walk index g.
__device__ __forceinline__ uint64_t wos_node(const WosArgs &a, uint64_t g) {
  if (a.total <= 0xffffffffull) {
    const uint32_t x = static_cast<uint32_t>(g), t = __umulhi(a.nt_m, x);
    return (t + ((x - t) >> a.nt_s1)) >> a.nt_s2;
  }
  return g / a.n_paths;
}

// Called by all 32 lanes: score the first cnt stopped walks, one per lane.
template <class Geom, typename R>
__device__ __forceinline__ void wos_flush(const WosArgs &a, WosStage<R> &st, int first, int cnt,
                                          FixAccum &acc, unsigned long long &my_steps,
                                          unsigned long long &my_capped) {
  const int lane = static_cast<int>(threadIdx.x & 31u);
  __syncwarp();
  const bool has = lane < cnt;
  R s = R(0);
  uint64_t node = 0;
  bool capped = false;
  if (has) {
    const int e = first + lane;
    R x[2] = {st.ex[0][e], st.ex[1][e]};
    const unsigned long long id = st.eid[e];
    const int32_t n = st.en[e];
    const int jb = Geom::template nearest_face<R>(x);
    capped = n >= a.max_steps && wos_dist<Geom, R>(x) > static_cast<R>(a.eps);
    my_capped += capped ? 1u : 0u;
    my_steps += static_cast<unsigned long long>(n);
    wos_project<Geom, R>(jb, x);
    s = LaplaceExpCos::g<R>(a.mc, x);
    node = wos_node(a, id);
    if (a.dump_score) a.dump_score[id] = static_cast<double>(s);
    if (a.steps) a.steps[id] = n;
    if (a.exit) {
      a.exit[2 * id] = static_cast<double>(x[0]);
      a.exit[2 * id + 1] = static_cast<double>(x[1]);
    }
  }
  acc.add<R>(a.fix, has, node, s, capped);
  __syncwarp();
}

template <class Geom, typename R>
__global__ void __launch_bounds__(kWosBlock) wos_kernel(const __grid_constant__ WosArgs a) {
  __shared__ WosStage<R> stage_all[kWosBlock / 32];
  WosStage<R> &st = stage_all[threadIdx.x >> 5];
  const unsigned lane = threadIdx.x & 31u, lt_mask = (1u << lane) - 1u;
  const R eps = static_cast<R>(a.eps);
  R X[2] = {R(0), R(0)}, d = R(0);
  PhiloxPath pp{0, 0, 2u};
  unsigned long long id = 0;
  int32_t n = 0;
  bool active = false, exhausted = false;
  int n_start = 0, n_stop = 0;                 // warp-uniform
  unsigned long long next = 0, claimed = 0;    // the warp's claimed range
  FixAccum acc;
  unsigned long long my_steps = 0, my_capped = 0, my_bad = 0;
  for (;;) {
    // ---- idle lanes take starts; the stash is refilled when empty
    unsigned need = __ballot_sync(kFull, !active);
    while (need) {
      if (n_start == 0) {
        if (exhausted) break;
        __syncwarp();
        if (next >= claimed) {
          unsigned long long base = 0;
          if (lane == 0) base = atomicAdd(a.cursor, static_cast<unsigned long long>(a.claim));
          next = __shfl_sync(kFull, base, 0);
          claimed = next + a.claim;
        }
        const unsigned long long q = next + lane;
        next += 32;
        if (next >= a.total) exhausted = true;
        bool in = false;
        R x[2] = {R(0), R(0)};
        uint64_t node = 0;
        PhiloxPath p{0, 0, 0};
        const bool has = q < a.total;
        if (has) {
          node = wos_node(a, q);
          p = philox_path(static_cast<uint32_t>(q - node * a.n_paths + a.path_offset),
                          static_cast<uint32_t>(node), 2u, a.rk);
          x[0] = static_cast<R>(a.nodes[2 * node]);
          x[1] = static_cast<R>(a.nodes[2 * node + 1]);
          in = Geom::inside_closed(x);
          if (!in) {
            ++my_bad;
            if (a.dump_score) a.dump_score[q] = static_cast<double>(NAN);
            if (a.steps) a.steps[q] = 0;
            if (a.exit) {
              a.exit[2 * q] = static_cast<double>(x[0]);
              a.exit[2 * q + 1] = static_cast<double>(x[1]);
            }
          }
        }
        if (__any_sync(kFull, has && !in)) fix_commit<R>(a.fix, has && !in, node, R(NAN), false, false);
        const unsigned im = __ballot_sync(kFull, in);
        if (in) {
          const int e = __popc(im & lt_mask);
          st.id[e] = q;
          st.w0[e] = p.r0_w0;
          st.w1[e] = p.r0_w1;
          st.x[0][e] = x[0];
          st.x[1][e] = x[1];
        }
        __syncwarp();
        n_start = __popc(im);
        continue;
      }
      const int cnt = __popc(need), take = cnt < n_start ? cnt : n_start;
      const int r = __popc(need & lt_mask);
      if (!active && r < take) {
        const int e = n_start - 1 - r;
        id = st.id[e];
        pp.r0_w0 = st.w0[e];
        pp.r0_w1 = st.w1[e];
        X[0] = st.x[0][e];
        X[1] = st.x[1][e];
        d = wos_dist<Geom, R>(X);
        n = 0;
        active = true;
      }
      n_start -= take;
      need = __ballot_sync(kFull, !active);
    }
    if (need == kFull) break;
    // ---- up to four jumps
    bool go = active && !(d <= eps) && n < a.max_steps;
    {
      const uint4 w = philox10_path(static_cast<uint32_t>(n >> 2), pp, a.rk);
      const uint32_t wj[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (go) {
          R cx, sy;
          wos_dir(unif<R>(wj[j]), cx, sy);
          X[0] += d * cx;
          X[1] += d * sy;
          ++n;
          d = wos_dist<Geom, R>(X);
          go = !(d <= eps) && n < a.max_steps;
        }
      }
    }
    // ---- stopped walks
    const bool stop = active && !go;
    const unsigned sm = __ballot_sync(kFull, stop);
    if (sm) {
      if (stop) {
        const int e = n_stop + __popc(sm & lt_mask);
        st.eid[e] = id;
        st.en[e] = n;
        st.ex[0][e] = X[0];
        st.ex[1][e] = X[1];
        active = false;
      }
      n_stop += __popc(sm);
      if (n_stop >= 32) {
        n_stop -= 32;
        wos_flush<Geom, R>(a, st, n_stop, 32, acc, my_steps, my_capped);
      }
    }
  }
  if (n_stop > 0) wos_flush<Geom, R>(a, st, 0, n_stop, acc, my_steps, my_capped);
  acc.flush(a.fix);
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

// Mean and standard error from the exact sums; the count is of all walks, also
// of a node outside the closed domain (whose mean and error are NaN).
__global__ void wos_finalize_kernel(const NodeFix *fix, int64_t n, double *mean, double *se,
                                    int64_t *cnt) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const NodeFix F = fix[i];
  double m, M2;
  fix_moments(F, &m, &M2);
  const double nn = static_cast<double>(F.n);
  mean[i] = m;
  se[i] = F.n > 1 ? sqrt(M2 / ((nn - 1.0) * nn)) : M2;
  if (cnt) cnt[i] = F.n + F.bad;
}

template <class Geom, typename R>
static pdd_status run_wos(pdd_ctx *ctx, const double *d_nodes, int64_t n, const pdd_wos_params *wp,
                          double *d_mean, double *d_se, int64_t *d_npaths, pdd_diag *diag) {
  const uint64_t N = static_cast<uint64_t>(wp->n_paths);
  const uint64_t total = static_cast<uint64_t>(n) * N;
  const size_t fix_off = 256;
  const size_t bytes = align_up(fix_off + static_cast<size_t>(n) * sizeof(NodeFix), 256);
  pdd_status st = ensure_scratch(ctx, bytes);
  if (st != PDD_OK) return st;
  char *base = static_cast<char *>(ctx->scratch);
  auto *counters = reinterpret_cast<unsigned long long *>(base);
  PDD_CUDA_TRY(ctx, cudaMemsetAsync(base, 0, bytes, ctx->stream));
  WosArgs a;
  std::memset(&a, 0, sizeof a);
  a.nodes = d_nodes;
  a.n_paths = N;
  a.path_offset = static_cast<uint64_t>(wp->path_offset);
  a.total = total;
  a.cursor = counters + 4;
  a.counters = counters;
  a.fix = reinterpret_cast<NodeFix *>(base + fix_off);
  a.rk = make_round_keys(wp->seed);
  a.eps = wp->eps;
  a.max_steps = static_cast<int32_t>(wp->max_steps);
  branch_divisor(N < (uint64_t(1) << 32) ? static_cast<uint32_t>(N) : 0xffffffffu, &a.nt_m, &a.nt_s1,
                 &a.nt_s2);
  a.mc = ctx->mc;
  if (diag) {
    a.dump_score = diag->d_path_score;
    a.steps = diag->d_path_steps;
    a.exit = diag->d_path_exit;
  }
  auto kern = wos_kernel<Geom, R>;
  int bps = 0;
  PDD_CUDA_TRY(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, kWosBlock, 0));
  if (bps < 1) bps = 1;
  if (ctx->path_blocks_per_sm > 0) bps = std::min(bps, ctx->path_blocks_per_sm);
  uint64_t grid = static_cast<uint64_t>(bps) * ctx->num_sms;
  grid = std::max<uint64_t>(1, std::min<uint64_t>(grid, (total + kWosBlock - 1) / kWosBlock));
  // a quarter of a warp's share at a time, so that a small call reaches every warp
  const uint64_t share = total / (grid * (kWosBlock / 32) * 4) / 32 * 32;
  a.claim = static_cast<uint32_t>(std::max<uint64_t>(32, std::min<uint64_t>(kWosClaim, share)));
  const auto ev = prof_slot(ctx);
  if (ev.first) PDD_CUDA_TRY(ctx, cudaEventRecord(ev.first, ctx->stream));
  kern<<<static_cast<unsigned>(grid), kWosBlock, 0, ctx->stream>>>(a);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  if (ev.second) PDD_CUDA_TRY(ctx, cudaEventRecord(ev.second, ctx->stream));
  wos_finalize_kernel<<<static_cast<unsigned>((n + kFinalizeBlock - 1) / kFinalizeBlock), kFinalizeBlock, 0, ctx->stream>>>(
      a.fix, n, d_mean, d_se, d_npaths);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  if (diag) {
    unsigned long long h[4] = {0, 0, 0, 0};
    PDD_CUDA_TRY(ctx, cudaMemcpyAsync(h, counters, sizeof h, cudaMemcpyDeviceToHost, ctx->stream));
    PDD_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    diag->path_steps = static_cast<int64_t>(h[0]);
    diag->capped = static_cast<int64_t>(h[1]);
    if (h[2]) return fail(ctx, PDD_EINVAL, "%llu paths started outside the closed domain", h[2]);
    if (h[1]) return fail(ctx, PDD_ECAP, "%llu walks hit max_steps", h[1]);
  }
  return PDD_OK;
}

pdd_status wos_solve_impl(pdd_ctx *ctx, const double *d_nodes, int64_t n, const pdd_wos_params *wp,
                          double *d_mean, double *d_se, int64_t *d_npaths, pdd_diag *diag) {
  if (!wp) return fail(ctx, PDD_EINVAL, "params is NULL");
  if (ctx->prob.kind != PDD_PROB_LAPLACE_EXPCOS)
    return fail(ctx, PDD_EINVAL, "Walk on Spheres needs the Laplace problem (Eq. 1.1)");
  if (reflect_mask(ctx) != 0)
    return fail(ctx, PDD_EINVAL, "Walk on Spheres needs Dirichlet data on every face");
  if (n < 0 || n > (int64_t(1) << 32) || wp->n_paths < 1 || wp->path_offset < 0 ||
      wp->path_offset + wp->n_paths > (int64_t(1) << 32))
    return fail(ctx, PDD_EINVAL, "sizes out of range");
  if (!(wp->eps > 0.0) || !(wp->eps < 0.5)) return fail(ctx, PDD_EINVAL, "eps must be in (0, 1/2)");
  if (wp->max_steps < 1 || wp->max_steps > 2147483647LL)
    return fail(ctx, PDD_EINVAL, "max_steps out of range");
  if (wp->precision != PDD_FP32 && wp->precision != PDD_FP64)
    return fail(ctx, PDD_EINVAL, "unknown precision");
  if (wp->precision == PDD_FP32 && wp->eps < 1e-6)
    return fail(ctx, PDD_EINVAL, "FP32 walks need eps >= 1e-6");
  if (diag) {
    diag->path_steps = 0;
    diag->capped = 0;
  }
  if (n == 0) return PDD_OK;
  if (!d_nodes || !d_mean || !d_se) return fail(ctx, PDD_EINVAL, "null buffer");
  PDD_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  const bool l = ctx->prob.geometry == PDD_GEOM_L_SHAPE;
  if (wp->precision == PDD_FP64)
    return l ? run_wos<LShape, double>(ctx, d_nodes, n, wp, d_mean, d_se, d_npaths, diag)
             : run_wos<Box<2>, double>(ctx, d_nodes, n, wp, d_mean, d_se, d_npaths, diag);
  return l ? run_wos<LShape, float>(ctx, d_nodes, n, wp, d_mean, d_se, d_npaths, diag)
           : run_wos<Box<2>, float>(ctx, d_nodes, n, wp, d_mean, d_se, d_npaths, diag);
}

}  // namespace pdd
