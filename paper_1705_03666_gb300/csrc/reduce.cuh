// reduce.cuh -- per-node sample mean / standard error of per-path scores
// (the Monte Carlo estimator of Sec. 2: the mean over independent
// realisations, with its statistical error).
//
// Each wave of the path index space is reduced by `parts` blocks per node: a
// block sums the shifted scores (s - K, with K the node's first score in the
// wave) and their squares, combines the threads in a fixed tree (warp shuffles,
// then shared memory), and the node's last block to finish adds the parts in a
// fixed tree and merges the wave's (count, mean, M2) into the node's running
// triple with Chan's formula.  Waves are processed in order, so the result is
// deterministic.
#pragma once

#include "common.cuh"
#include "ctx.hpp"
#include "nodefix.cuh"

namespace pdd {

constexpr int kReduceBlock = 256;

struct NodeAcc {  // running (count, mean, M2) per node, FP64
  double n, mean, m2;
};

// Per-thread accumulation.  Binary32 scores are summed on the FP32 pipe as
// two-float values (Knuth's TwoSum: a ~48-bit significand, far below the
// scores' own rounding), the shift s - K split exactly into two floats and
// the square's rounding error recovered with an FMA; binary64 scores are
// summed plainly in FP64 (a few thousand terms per thread).  FP64 is a
// 1/64-rate pipe on this part, so a compensated FP64 sum per score would
// make the reduction, not the paths, the cost of short-path workloads.
// Threads are then combined in fixed trees in FP64, a warp's (warp_total) and the
// warps' compensated.  Compensated additions throughout, 170 FP64 instructions per
// warp, took 76 of 125 us for 1024 nodes of 10^5 binary32 scores; 93 us in all with
// the warp's exact ones.
struct F2Sum {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float s = hi + v;
    const float bb = s - hi;
    lo += (hi - (s - bb)) + (v - bb);
    hi = s;
  }
};

// Whether 32 binary32 numbers add up exactly in FP64 in any order: the last bit of
// the smallest and the top of the sum within 53 bits (finite, exponents within 24).
__device__ __forceinline__ bool warp_adds_exactly(float v) {
  const uint32_t b = __float_as_uint(v) & 0x7fffffffu, e = max(b >> 23, 1u);
  const uint32_t top = __reduce_max_sync(kFull, b ? e : 0u);
  const uint32_t low = __reduce_max_sync(kFull, b ? 256u - e : 0u);  // 256 less the smallest
  return top == 0u || (top < 255u && top + low <= 256u + 24u);
}
// The total of n unevaluated sums s + c (n a power of two up to 32), one per lane
// below n: compensated, the larger of two found by their bits (an FP64 comparison
// occupies its scheduler's pipe for 64 clocks as the additions do, five of them a
// step of the tree).
__device__ __forceinline__ CSum lanes_total(CSum t, int n) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    if (m >= n) continue;
    const CSum o = shfl_xor(t, m);
    constexpr unsigned long long kAbs = 0x7fffffffffffffffull;
    const bool own = (static_cast<unsigned long long>(__double_as_longlong(t.s)) & kAbs) >=
                     (static_cast<unsigned long long>(__double_as_longlong(o.s)) & kAbs);
    const double big = own ? t.s : o.s, small = own ? o.s : t.s, sum = t.s + o.s;
    t.c = t.c + o.c + ((big - sum) + small);
    t.s = sum;
  }
  return t;
}
// The warp's total, in every lane.  Two-float sums: the high and the low parts by
// themselves where the high ones add up exactly, as they do but for sums of very
// different size (the low ones, below 2^-24 of them, then lose 2^-77, a two-float sum
// itself 2^-48); compensated otherwise, and for binary64 sums.
__device__ __forceinline__ CSum warp_total(const CSum &t) { return lanes_total(t, 32); }
__device__ __forceinline__ CSum warp_total(const F2Sum &v) {
  CSum t;
  t.s = static_cast<double>(v.hi);
  t.c = static_cast<double>(v.lo);
  if (!warp_adds_exactly(v.hi)) return lanes_total(t, 32);
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    t.s += __shfl_xor_sync(kFull, t.s, m);
    t.c += __shfl_xor_sync(kFull, t.c, m);
  }
  return t;
}

template <typename R, bool kSkipNaN>
struct ThreadSums;
template <bool kSkipNaN>
struct ThreadSums<float, kSkipNaN> {
  F2Sum s1, s2;
  unsigned kept = 0;  // below 2^32: a wave holds at most 2^31 scores
  __device__ __forceinline__ void add(float v, float K) {
    if constexpr (kSkipNaN) {
      // K = 0 here: a NaN score is replaced by 0, which adds exactly zero,
      // and the shift needs no split
      const bool ok = !isnan(v);
      kept += ok ? 1u : 0u;
      v = ok ? v : 0.0f;
      s1.add(v);
      const float q = v * v;
      const float e = fmaf(v, v, -q);
      s2.add(q);
      s2.lo += e;
      return;
    }
    ++kept;
    const float d = v - K;  // d + dl = v - K exactly
    const float bb = d - v;
    const float dl = (v - (d - bb)) + (-K - bb);
    s1.add(d);
    s1.lo += dl;
    const float q = d * d;
    const float e = fmaf(d, d, -q);
    s2.add(q);
    s2.lo += e + 2.0f * d * dl;
  }
  __device__ __forceinline__ CSum total1() const { return warp_total(s1); }
  __device__ __forceinline__ CSum total2() const { return warp_total(s2); }
};
template <bool kSkipNaN>
struct ThreadSums<double, kSkipNaN> {
  double s1 = 0.0, s2 = 0.0;
  unsigned long long kept = 0;
  __device__ __forceinline__ void add(double v, double K) {
    if (kSkipNaN && isnan(v)) return;
    ++kept;
    const double d = v - K;
    s1 += d;
    s2 = fma(d, d, s2);
  }
  __device__ __forceinline__ CSum total1() const { return warp_total(CSum{s1, 0.0}); }
  __device__ __forceinline__ CSum total2() const { return warp_total(CSum{s2, 0.0}); }
};

// The parts of a wave's nodes (rec [planes][nodes][parts], done [planes][nodes]
// counts the finished ones, zero before and after).
struct ReducePart {
  CSum s1, s2;
  unsigned long long kept;
};
struct ReduceParts {
  int parts;
  ReducePart *rec;
  unsigned *done;
};
// Blocks per node: one while the nodes fill the GPU (512 blocks), else up to 32
// of at least 4096 scores (4 nodes x 10^5 scores: 36 us with one, 14 us
// with 16; 16 x 10^6: 186 -> 30 us).  A function of the sizes alone, so the order of
// the additions does not depend on the device.
inline int reduce_parts(uint64_t n_paths, uint64_t blocks) {
  int p = 1;
  while (p < 32 && blocks * p < 512 && n_paths / (2 * p) >= 4096) p *= 2;
  return p;
}
inline size_t reduce_parts_bytes(uint64_t blocks, int parts) {
  return parts > 1 ? align_up(blocks * parts * sizeof(ReducePart), 256) +
                         align_up(blocks * sizeof(unsigned), 256)
                   : 0;
}
// The layout at `base` (its counters zeroed by the caller).
inline ReduceParts reduce_parts_at(char *base, uint64_t blocks, int parts) {
  return {parts, reinterpret_cast<ReducePart *>(base),
          reinterpret_cast<unsigned *>(base + align_up(blocks * parts * sizeof(ReducePart), 256))};
}

// kSkipNaN: NaN scores mark discarded samples (pruned trees) and are left
// out of the count; the shift K is then 0 (scores are bounded weights).
template <typename R, bool kSkipNaN = false>
__global__ void __launch_bounds__(kReduceBlock)
reduce_wave_kernel(const R *__restrict__ score, uint64_t begin, uint64_t end,
                   uint64_t n_paths, uint64_t node_lo, NodeAcc *acc, ReduceParts rp,
                   uint64_t score_plane = 0, uint64_t acc_plane = 0) {
  // blockIdx.y selects a plane (score + y score_plane, acc + y acc_plane):
  // several score planes of one wave reduced by one launch
  score += blockIdx.y * score_plane;
  acc += blockIdx.y * acc_plane;
  const uint64_t node = node_lo + blockIdx.x / rp.parts;
  const unsigned part = blockIdx.x % rp.parts;
  const uint64_t nlo = max(begin, node * n_paths);
  const uint64_t nhi = min(end, (node + 1) * n_paths);
  if (nlo >= nhi) return;
  const uint64_t lo = nlo + (nhi - nlo) * part / rp.parts;
  const uint64_t hi = nlo + (nhi - nlo) * (part + 1) / rp.parts;
  const R *s = score + (lo - begin);
  const uint64_t cnt = hi - lo;
  const R Kr = kSkipNaN ? R(0) : score[nlo - begin];
  const double K = static_cast<double>(Kr);
  ThreadSums<R, kSkipNaN> ts;
  if constexpr (sizeof(R) == 4) {
    // binary32 scores: scalar up to a 16-byte boundary, then four per load
    // with several loads in flight per thread (the reduction is bound by
    // memory latency otherwise), then the scalar tail
    uint64_t head = ((16u - (reinterpret_cast<uintptr_t>(s) & 15u)) & 15u) / 4u;
    if (head > cnt) head = cnt;
    if (threadIdx.x < head) ts.add(s[threadIdx.x], Kr);
    const float4 *v = reinterpret_cast<const float4 *>(s + head);
    const uint64_t n4 = (cnt - head) / 4;
#pragma unroll 4
    for (uint64_t j = threadIdx.x; j < n4; j += kReduceBlock) {
      const float4 q = __ldcs(v + j);
      ts.add(q.x, Kr);
      ts.add(q.y, Kr);
      ts.add(q.z, Kr);
      ts.add(q.w, Kr);
    }
    for (uint64_t i = head + 4 * n4 + threadIdx.x; i < cnt; i += kReduceBlock) ts.add(s[i], Kr);
  } else {
    for (uint64_t i = threadIdx.x; i < cnt; i += kReduceBlock) ts.add(s[i], Kr);
  }
  const CSum s1 = ts.total1(), s2 = ts.total2();
  unsigned long long kept = ts.kept;
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) kept += __shfl_xor_sync(kFull, kept, m);
  constexpr int kWarps = kReduceBlock / 32;
  __shared__ CSum sh1[kWarps], sh2[kWarps];
  __shared__ unsigned long long shk[kWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    sh1[warp] = s1;
    sh2[warp] = s2;
    shk[warp] = kept;
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  CSum t1 = lanes_total(sh1[lane % kWarps], kWarps), t2 = lanes_total(sh2[lane % kWarps], kWarps);
  unsigned long long tk = 0;
  for (int w = 0; w < kWarps; ++w) tk += shk[w];
  if (rp.parts > 1) {
    const uint64_t q = blockIdx.y * (gridDim.x / rp.parts) + blockIdx.x / rp.parts;
    ReducePart *const rec = rp.rec + q * rp.parts;
    unsigned before = 0;
    if (lane == 0) {
      rec[part] = {t1, t2, tk};
      __threadfence();
      before = atomicAdd(rp.done + q, 1u);
    }
    if (__shfl_sync(kFull, before, 0) != static_cast<unsigned>(rp.parts - 1)) return;
    __threadfence();
    t1 = t2 = CSum{};
    tk = 0;
    if (lane < rp.parts) {
      const volatile ReducePart *const v = rec + lane;
      t1.s = v->s1.s;
      t1.c = v->s1.c;
      t2.s = v->s2.s;
      t2.c = v->s2.c;
      tk = v->kept;
    }
    t1 = lanes_total(t1, rp.parts);
    t2 = lanes_total(t2, rp.parts);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) tk += __shfl_xor_sync(kFull, tk, m);
    if (lane == 0) rp.done[q] = 0;
  }
  if (threadIdx.x == 0) {
    if (tk == 0) return;
    const double nb = static_cast<double>(tk);
    const double S1 = t1.value(), S2 = t2.value();
    const double mean_b = K + S1 / nb;
    const double m2_b = fmax(0.0, S2 - S1 * S1 / nb);
    NodeAcc A = acc[node];
    const double nt = A.n + nb;
    const double d = mean_b - A.mean;
    A.mean = A.mean + d * (nb / nt);
    A.m2 = A.m2 + m2_b + d * d * (A.n * nb / nt);
    A.n = nt;
    acc[node] = A;
  }
}

// Mean, standard error and count per node; with `flags`, PDD_NODE_EMPTY is
// OR-ed into the node's flags when no sample was kept (the kernels OR in the
// rarer events themselves).
static __global__ void finalize_kernel(const NodeAcc *acc, int64_t n_nodes, double *mean,
                                       double *se, int64_t *npaths, int32_t *flags = nullptr) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n_nodes) return;
  const NodeAcc A = acc[i];
  mean[i] = A.n > 0.0 ? A.mean : static_cast<double>(NAN);  // no sample kept
  se[i] = A.n > 1.0 ? sqrt(A.m2 / (A.n - 1.0) / A.n) : (A.n > 0.0 ? 0.0 : static_cast<double>(NAN));
  if (npaths) npaths[i] = static_cast<int64_t>(A.n);
  if (flags && !(A.n > 0.0)) flags[i] |= kNodeEmpty;
}

template <typename R>
__global__ void widen_scores_kernel(const R *__restrict__ src, double *dst, uint64_t count) {
  for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < count;
       i += static_cast<uint64_t>(gridDim.x) * blockDim.x)
    dst[i] = static_cast<double>(src[i]);
}

}  // namespace pdd
