// grad_kernel.cuh -- the gradient mode of the path kernel: the same paths
// (bit for bit, recomputed from their Philox keys), carrying the 16
// likelihood-ratio sums of the drift weights and writing one record per path
// for the Jacobian reduction (grad.cu).
//
// The units test every step where it occurs (em_step through path_unit_code):
// a parked unit would have to keep the 16 sums as well.
#pragma once

#include "path_kernel.cuh"

namespace pdd {

// Per-path record of the gradient mode: score, exit point, and the
// likelihood-ratio sums L_j (already scaled by sqrt(dt)/sigma).
struct GradRec {
  float s, x, y, z;
  float L[kMaxLR];
};

// The record's first four words (score and exit point) with
// the step count, and the likelihood-ratio sums.
template <int D, typename R>
__device__ __forceinline__ void write_score(const PathArgs &a, uint64_t slot, R s, int32_t st,
                                            const R *xe) {
  float4 *o = reinterpret_cast<float4 *>(static_cast<GradRec *>(a.score) + slot);
  o[0] = make_float4(static_cast<float>(s), static_cast<float>(xe[0]),
                     D > 1 ? static_cast<float>(xe[D > 1 ? 1 : 0]) : 0.f,
                     D > 2 ? static_cast<float>(xe[D > 2 ? 2 : 0]) : 0.f);
  if (a.steps) a.steps[slot] = st;
}
template <typename R>
__device__ __forceinline__ void write_lr_sums(const PathArgs &a, uint64_t slot, const R *L) {
  float4 *o = reinterpret_cast<float4 *>(static_cast<GradRec *>(a.score) + slot);
  const float c = a.lr_scale;
#pragma unroll
  for (int q = 0; q < kMaxLR / 4; ++q)
    o[1 + q] = make_float4(c * static_cast<float>(L[4 * q]), c * static_cast<float>(L[4 * q + 1]),
                           c * static_cast<float>(L[4 * q + 2]), c * static_cast<float>(L[4 * q + 3]));
}

// Per-warp staging in shared memory (one column per lane).  Claiming and
// setting up a path (atomic, node division, Philox key, FP64 node load) and
// scoring an ended path (exit point, accurate g) happen once per path, at
// times that differ from lane to lane: done where they occur, each would run
// with one lane of the warp active.  Instead a warp claims 32 consecutive
// paths at once and sets them all up with every lane busy (StartStash), and
// ended paths are parked (ExitQueue) and scored 32 at a time.  Every path
// writes its own slot, so the results do not depend on this order.
template <int D, typename R>
struct StartStash {
  unsigned long long slot[32];  // index in the wave
  uint32_t w0[32], w1[32];      // PhiloxPath words (tag 0)
  R x[D][32];                   // start point
};
template <int D, typename R>
struct ExitQueue {
  unsigned long long slot[32];
  int32_t st[32], code[32];     // step count (or -max_steps) and exit code
  R x[D][32], xn[D][32], y[32], z[32];
};
template <int D, typename R>
struct PathStage {
  StartStash<D, R> start;
  ExitQueue<D, R> exit;
};

// Called by all 32 lanes: claim the next 32 indices of the wave, set each up,
// score at once the ones that start on the boundary (tau = 0, u = g, Eq. 2.1)
// or outside the closed domain (invalid input: NaN, counted), and stage the
// interior ones.  Returns how many were staged (warp-uniform).
template <class Model, class Geom, typename R>
__device__ __forceinline__ int stage_starts(const PathArgs &a, StartStash<Model::D, R> &st,
                                            unsigned long long span, bool &exhausted,
                                            unsigned long long &my_bad) {
  constexpr int D = Model::D;
  const unsigned lane = threadIdx.x & 31u;
  __syncwarp();  // earlier reads of the stash are done
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(a.cursor, 32ull);
  base = __shfl_sync(kFull, base, 0);
  if (base + 32 >= span) exhausted = true;
  const unsigned long long q = base + lane;
  bool interior = false;
  R x[D];
  PhiloxPath pp{0, 0, 0};
  if (q < span) {
    const unsigned long long g = a.begin + q;
    const uint64_t node = path_node(a, g);
    const uint64_t path = g - node * a.n_paths + a.path_offset;
    pp = philox_path(static_cast<uint32_t>(path), static_cast<uint32_t>(node) + a.node_offset, 0u,
                     a.rk);
#pragma unroll
    for (int d = 0; d < D; ++d) x[d] = static_cast<R>(a.nodes[node * D + d]);
    interior = Geom::inside_open(x);
    if (!interior) {
      R s0 = Model::g(a.mc, x);
      if (!Geom::inside_closed(x)) {
        s0 = R(NAN);
        ++my_bad;
      }
      R L0[kMaxLR];
#pragma unroll
      for (int j = 0; j < kMaxLR; ++j) L0[j] = R(0);
      write_score<D, R>(a, q, s0, 0, x);
      write_lr_sums<R>(a, q, L0);
    }
  }
  const unsigned im = __ballot_sync(kFull, interior);
  if (interior) {
    const int e = __popc(im & ((1u << lane) - 1u));
    st.slot[e] = q;
    st.w0[e] = pp.r0_w0;
    st.w1[e] = pp.r0_w1;
#pragma unroll
    for (int d = 0; d < D; ++d) st.x[d][e] = x[d];
  }
  __syncwarp();
  return __popc(im);
}

// Called by all 32 lanes: score the first cnt parked paths, one per lane, and
// write the record's score and exit point (the likelihood-ratio sums were
// written when the path ended).
template <class Model, class Geom, typename R>
__device__ __forceinline__ void flush_exits(const PathArgs &a, ExitQueue<Model::D, R> &q, int cnt) {
  constexpr int D = Model::D;
  const int lane = static_cast<int>(threadIdx.x & 31u);
  __syncwarp();
  if (lane < cnt) {
    R s, X[D], Xn[D], xe[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      X[d] = q.x[d][lane];
      Xn[d] = q.xn[d][lane];
    }
    const int code = q.code[lane];
    if (code == kStepCapped) {
#pragma unroll
      for (int d = 0; d < D; ++d) xe[d] = X[d];
      Geom::project(Geom::nearest_face(X), xe);
      s = Model::g(a.mc, xe) * q.y[lane] + q.z[lane];
    } else {
      s = exit_score<Model, Geom, R>(a.mc, code, X, Xn, q.y[lane], q.z[lane], xe);
    }
    write_score<D, R>(a, q.slot[lane], s, q.st[lane], xe);
  }
  __syncwarp();
}

constexpr int kGradBlock = 128;
template <class Model, class Geom, typename R>
__global__ void __launch_bounds__(kGradBlock)
path_lr_kernel(const __grid_constant__ PathArgs a) {
  constexpr int D = Model::D;
  constexpr int NL = kMaxLR;
  __shared__ PathStage<D, R> stage_all[kGradBlock / 32];
  PathStage<D, R> &stage = stage_all[threadIdx.x >> 5];
  R L[NL];
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt_mask = (1u << lane) - 1u;
  const StepConst<R> k(a);
  const unsigned long long span = a.end - a.begin;
  R X[D], Xn[D];
  R Y = R(1), Z = R(0);
  PhiloxPath pp{0, 0, 0};
  unsigned long long slot = 0;
  int32_t n = 0;
  bool active = false;
  int n_start = 0, n_exit = 0;  // stash / queue fill (warp-uniform)
  bool exhausted = false;       // the wave's indices are all claimed (warp-uniform)
  unsigned long long my_steps = 0, my_capped = 0, my_bad = 0;

  for (;;) {
    // ---- idle lanes take staged paths; the stash is refilled when empty
    unsigned needmask = __ballot_sync(kFull, !active);
    if (needmask) {
    while (needmask) {
      if (n_start == 0) {
        if (exhausted) break;
        n_start = stage_starts<Model, Geom, R>(a, stage.start, span, exhausted, my_bad);
        continue;
      }
      const int cnt = __popc(needmask);
      const int take = cnt < n_start ? cnt : n_start;
      if (!active) {
        const int r = __popc(needmask & lt_mask);
        if (r < take) {
          const int e = n_start - 1 - r;
          slot = stage.start.slot[e];
          pp.r0_w0 = stage.start.w0[e];
          pp.r0_w1 = stage.start.w1[e];
          pp.tag = 0u;
#pragma unroll
          for (int d = 0; d < D; ++d) X[d] = stage.start.x[d][e];
          Y = R(1);
          Z = R(0);
          n = 0;
#pragma unroll
          for (int j = 0; j < NL; ++j) L[j] = R(0);
          active = true;
        }
      }
      n_start -= take;
      needmask = __ballot_sync(kFull, !active);
    }
    if (!__any_sync(kFull, active)) break;
    }

    // ---- advance the lane's path by one unit
    int code = kStepContinue;
    bool done = false;
    if (active) {
      code = path_unit_code<Model, Geom, R, true, true>(a, k, pp, a.rk, a.max_steps, X, Y, Z, n, Xn, L);
      done = code != kStepContinue || n >= a.max_steps;
      if (done) {
        my_steps += static_cast<unsigned long long>(n);
        if (code == kStepContinue) {
          code = kStepCapped;
          ++my_capped;
        }
      }
    }

    // ---- ended paths: parked, and scored 32 at a time (the likelihood-ratio
    // sums are written at once)
    const unsigned dm = __ballot_sync(kFull, done);
    if (dm) {
      const int nd = __popc(dm);
      if (n_exit + nd > 32) {
        flush_exits<Model, Geom, R>(a, stage.exit, n_exit);
        n_exit = 0;
      }
      if (done) {
        write_lr_sums<R>(a, slot, L);
        const int e = n_exit + __popc(dm & lt_mask);
        ExitQueue<D, R> &q = stage.exit;
        q.slot[e] = slot;
        q.st[e] = code == kStepCapped ? -a.max_steps : n;
        q.code[e] = code;
#pragma unroll
        for (int d = 0; d < D; ++d) {
          q.x[d][e] = X[d];
          q.xn[d][e] = Xn[d];
        }
        q.y[e] = Y;
        q.z[e] = Z;
        active = false;
      }
      n_exit += nd;
    }
  }
  if (n_exit > 0) flush_exits<Model, Geom, R>(a, stage.exit, n_exit);

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

}  // namespace pdd
