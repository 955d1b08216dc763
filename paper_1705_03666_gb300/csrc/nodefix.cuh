// nodefix.cuh -- exact, order-independent per-node sums of path scores (the
// Monte Carlo estimator of Sec. 2: the mean over independent realisations and
// its statistical error), formed inside the path kernel.
//
// Each score s is truncated once to the fixed-point grid 2^-60 and written
// as five base-2^24 digits (weights 2^-60, 2^-36, 2^-12, 2^12, 2^36), and so
// is s^2, formed exactly from the significand in integers.  A warp sums the
// digits of its lanes' paths of one node with one 32-bit reduction
// instruction per digit (32 digits below 2^24 in magnitude cannot overflow),
// and the node's first lane adds the totals to the node's 64-bit words with
// atomics, without carries between digits (at most 2^32 paths per node keep
// every word within 2^56).  Integer addition is associative: the totals are
// the same whichever lane, warp or launch added which path, so the estimate is
// bitwise reproducible while no per-path score is ever stored.
//
// Range: |s| < 2^30 (so that s^2 < 2^60).  A score outside it, or NaN (a node
// outside the closed domain), is counted in `bad` and makes the node's
// estimate NaN.  Truncation at 2^-60 changes a score by less than 2^-60 in
// absolute value, far below the rounding of the score itself.
#pragma once

#include <cstring>

#include "common.cuh"

namespace pdd {

constexpr int kFixDigits = 5;
struct NodeFix {
  long long n;                 // paths scored (boundary starts included)
  long long s1[kFixDigits];    // digit sums of s
  long long s2[kFixDigits];    // digit sums of s^2
  long long capped;            // paths stopped by the step cap
  long long bad;               // NaN or out-of-range scores
  long long boundary;          // paths that started on the boundary (tau = 0)
};
constexpr int kFixWords = 2 + 2 * kFixDigits + 2;
static_assert(sizeof(NodeFix) == kFixWords * sizeof(long long), "NodeFix layout");
constexpr int kFixCapped = 1 + 2 * kFixDigits, kFixBad = kFixCapped + 1,
              kFixBoundary = kFixCapped + 2;

// Per-node flags (include/pdd.h, pdd_diag.d_node_flags).
constexpr int32_t kNodeOnBoundary = 1;
constexpr int32_t kNodeOutside = 2;
constexpr int32_t kNodeCapped = 4;
constexpr int32_t kNodeDiscarded = 8;
constexpr int32_t kNodeEmpty = 16;
constexpr int32_t kNodeSeUnmet = 32;

constexpr uint32_t kDigitMask = (1u << 24) - 1;

// Digit k of floor(M 2^sh) for M < 2^24: floor(M 2^(sh - 24k)) mod 2^24
// (the 32-bit shift keeps the low 24 bits of M 2^t for 0 <= t < 24).
__device__ __forceinline__ int32_t fix_digit24(uint32_t M, int t) {
  if (t >= 24 || t <= -24) return 0;
  return static_cast<int32_t>(t >= 0 ? (M << t) & kDigitMask : M >> (-t));
}
// The same for M < 2^48 (a product of two 24-bit significands).
__device__ __forceinline__ int32_t fix_digit48(unsigned long long M, int t) {
  if (t >= 24 || t <= -48) return 0;
  return static_cast<int32_t>((t >= 0 ? M << t : M >> (-t)) & kDigitMask);
}
// The same for M < 2^106 (a product of two 53-bit significands).
__device__ __forceinline__ int32_t fix_digit106(unsigned __int128 M, int t) {
  if (t >= 24 || t <= -106) return 0;
  return static_cast<int32_t>(static_cast<unsigned long long>(t >= 0 ? M << t : M >> (-t)) &
                              kDigitMask);
}

// Digits of s 2^60 (d1, with the sign of s) and of s^2 2^60 (d2), each
// truncated toward zero, from the bits of s: s = +-m 2^e, so s 2^60 =
// m 2^(e + 60) and s^2 2^60 = m^2 2^(2e + 60) with m^2 formed exactly in
// integers.  Integer arithmetic only (the FP64 pipe is a 1/64-rate unit on
// this part).  Requires |s| < 2^30.
__device__ __forceinline__ void fix_limbs(float s, int32_t *d1, int32_t *d2) {
  const uint32_t b = __float_as_uint(s);
  const int E = static_cast<int>((b >> 23) & 0xffu);
  const uint32_t m = (b & 0x7fffffu) | (E ? 0x800000u : 0u);
  const int e = (E ? E : 1) - 150;  // s = m 2^e
  const unsigned long long m2 = static_cast<unsigned long long>(m) * m;
  const bool neg = (b >> 31) != 0;
#pragma unroll
  for (int k = 0; k < kFixDigits; ++k) {
    const int32_t v = fix_digit24(m, e + 60 - 24 * k);
    d1[k] = neg ? -v : v;
    d2[k] = fix_digit48(m2, 2 * e + 60 - 24 * k);
  }
}
__device__ __forceinline__ void fix_limbs(double s, int32_t *d1, int32_t *d2) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(s));
  const int E = static_cast<int>((b >> 52) & 0x7ffu);
  const unsigned long long m = (b & 0xfffffffffffffull) | (E ? (1ull << 52) : 0ull);
  const int e = (E ? E : 1) - 1075;  // s = m 2^e
  const unsigned __int128 m2 = static_cast<unsigned __int128>(m) * m;
  const bool neg = (b >> 63) != 0;
#pragma unroll
  for (int k = 0; k < kFixDigits; ++k) {
    const int32_t v = fix_digit106(m, e + 60 - 24 * k);
    d1[k] = neg ? -v : v;
    d2[k] = fix_digit106(m2, 2 * e + 60 - 24 * k);
  }
}

// Called by all 32 lanes of a warp.  A lane with `has` set adds one path of
// node `node` with score s (capped: stopped by the step cap; boundary: started
// on the boundary; NaN s: invalid start).  Every lane forms its digits first
// (no divergence); then, one node at a time, each digit is summed over the
// node's lanes with one warp reduction and the node's first lane issues the
// atomics.  The rare events (capped, boundary, invalid) are counted with
// per-lane atomics.
template <typename R>
__device__ __forceinline__ void fix_commit(NodeFix *fix, bool has, uint64_t node, R s,
                                           bool capped, bool boundary) {
  const bool valid = has && fabs(s) < R(0x1p30);  // false for NaN
  if (has) {
    unsigned long long *w = reinterpret_cast<unsigned long long *>(fix + node);
    if (!valid) atomicAdd(w + kFixBad, 1ull);
    if (valid && capped) atomicAdd(w + kFixCapped, 1ull);
    if (valid && boundary) atomicAdd(w + kFixBoundary, 1ull);
  }
  int32_t d[2 * kFixDigits];
#pragma unroll
  for (int k = 0; k < 2 * kFixDigits; ++k) d[k] = 0;
  if (valid) fix_limbs(s, d, d + kFixDigits);
  const unsigned lane = threadIdx.x & 31u;
  unsigned pending = __ballot_sync(kFull, valid);
  while (pending) {
    const int leader = __ffs(pending) - 1;
    const uint64_t ln = __shfl_sync(kFull, node, leader);
    const bool mem = valid && node == ln;
    const unsigned members = __ballot_sync(kFull, mem);
    unsigned long long *w = reinterpret_cast<unsigned long long *>(fix + ln);
    int32_t r[2 * kFixDigits];
#pragma unroll
    for (int k = 0; k < 2 * kFixDigits; ++k) r[k] = __reduce_add_sync(kFull, mem ? d[k] : 0);
    if (lane == static_cast<unsigned>(leader)) {
      atomicAdd(w, static_cast<unsigned long long>(__popc(members)));
#pragma unroll
      for (int k = 0; k < 2 * kFixDigits; ++k)
        if (r[k] != 0)
          atomicAdd(w + 1 + k, static_cast<unsigned long long>(static_cast<long long>(r[k])));
    }
    pending &= ~members;
  }
}

// Per-warp running sums of one node, for work units so short that an atomic per
// digit and flush would contend (10^6 walks of a dozen jumps per node): lane l
// holds word l of the node's sums (the count, then the digits), added to the
// node with one atomic per word when the warp moves to another node.
struct FixAccum {
  long long v = 0;
  uint64_t node = ~0ull;
  __device__ __forceinline__ void flush(NodeFix *fix) {
    const unsigned lane = threadIdx.x & 31u;
    if (node != ~0ull && lane <= 2u * kFixDigits && v != 0)
      atomicAdd(reinterpret_cast<unsigned long long *>(fix + node) + lane,
                static_cast<unsigned long long>(v));
    v = 0;
  }
  // As fix_commit (no boundary starts).
  template <typename R>
  __device__ __forceinline__ void add(NodeFix *fix, bool has, uint64_t nd, R s, bool capped) {
    const unsigned lane = threadIdx.x & 31u;
    const bool valid = has && fabs(s) < R(0x1p30);  // false for NaN
    if (has && (!valid || capped))
      atomicAdd(reinterpret_cast<unsigned long long *>(fix + nd) + (valid ? kFixCapped : kFixBad), 1ull);
    int32_t d[2 * kFixDigits];
#pragma unroll
    for (int k = 0; k < 2 * kFixDigits; ++k) d[k] = 0;
    if (valid) fix_limbs(s, d, d + kFixDigits);
    unsigned pending = __ballot_sync(kFull, valid);
    while (pending) {
      const uint64_t ln = __shfl_sync(kFull, nd, __ffs(pending) - 1);
      const bool mem = valid && nd == ln;
      const unsigned members = __ballot_sync(kFull, mem);
      if (ln != node) {
        flush(fix);
        node = ln;
      }
      if (lane == 0) v += __popc(members);
#pragma unroll
      for (int k = 0; k < 2 * kFixDigits; ++k) {
        const int32_t r = __reduce_add_sync(kFull, mem ? d[k] : 0);
        if (lane == static_cast<unsigned>(k + 1)) v += r;
      }
      pending &= ~members;
    }
  }
};

// 2^e, a normal number.
__host__ __device__ __forceinline__ double fix_pow2(int e) {
  const long long b = static_cast<long long>(e + 1023) << 52;
  double d;
  memcpy(&d, &b, sizeof d);
  return d;
}
// The 63 leading bits m of a (256 bits, w[3] the highest word, not zero) and
// their weight: a = m 2^e but for what is below m.
__host__ __device__ __forceinline__ unsigned long long fix_top(const unsigned long long *w, int *e) {
  int h = 3;
  while (h > 0 && w[h] == 0) --h;
  int lz = 0;
  for (int s = 32; s > 0; s >>= 1)
    if ((w[h] << lz) >> (64 - s) == 0) lz += s;
  const unsigned long long below = h > 0 ? w[h - 1] : 0;
  const unsigned long long top = lz ? (w[h] << lz) | (below >> (64 - lz)) : w[h];
  *e = 64 * h - lz + 1;
  return top >> 1;
}

// m / nn for m < 2^63 and an integer nn below 2^53 with rn = 1 / nn: the quotient
// of m's leading part corrected by its exact remainder and the rest of m, and one
// rounding.
__host__ __device__ __forceinline__ double fix_quotient(unsigned long long m, double nn, double rn) {
  const double hi = static_cast<double>(m);
  const double lo = static_cast<double>(static_cast<long long>(m - static_cast<unsigned long long>(hi)));
  const double q = hi * rn;
  return q + (fma(-q, nn, hi) + lo) * rn;
}

// Mean and the sum of squared deviations M2 of a node's scores from its exact
// sums: mean = S1 / n and M2 = (n S2 - S1^2) / n, the numerator in exact integers
// (256 bits, cut to 63) and the quotient rounded once, so that FP64, a 1/64-rate
// pipe on this part, only has to divide: one warp took 10.4 us for both in
// double-doubles (some 350 dependent instructions) after every small solve.  M2 =
// 0 when every path started on the boundary, or with one path; both NaN when a
// path was invalid or nothing was scored.
__host__ __device__ __forceinline__ void fix_moments(const NodeFix &F, double *mean, double *m2) {
  using u64 = unsigned long long;
  using u128 = unsigned __int128;
  *mean = static_cast<double>(NAN);
  *m2 = static_cast<double>(NAN);
  if (F.bad != 0 || F.n <= 0) return;
  const u64 n = static_cast<u64>(F.n);
  const double nn = static_cast<double>(F.n), rn = 1.0 / nn;
  // S1 2^60: below n 2^90 <= 2^122 in magnitude, so sums mod 2^128 hold it
  u128 t = 0;
#pragma unroll
  for (int k = 0; k < kFixDigits; ++k)
    t += static_cast<u128>(static_cast<__int128>(F.s1[k])) << (24 * k);
  const bool neg = (t >> 127) != 0;
  if (neg) t = 0 - t;
  const u64 a0 = static_cast<u64>(t), a1 = static_cast<u64>(t >> 64);
  if (t == 0) {
    *mean = 0.0;
  } else {
    const u64 w[4] = {a0, a1, 0, 0};
    int e;
    const u64 m = fix_top(w, &e);
    const double q = fix_quotient(m, nn, rn);
    *mean = (neg ? -q : q) * fix_pow2(e - 60);
  }
  *m2 = 0.0;
  if (F.boundary == F.n || F.n <= 1) return;
  // n S2 2^120 (S2's digits are not negative)
  const u128 lo = static_cast<u128>(static_cast<u64>(F.s2[0])) +
                  (static_cast<u128>(static_cast<u64>(F.s2[1])) << 24) +
                  (static_cast<u128>(static_cast<u64>(F.s2[2])) << 48);
  const u128 hi = static_cast<u128>(static_cast<u64>(F.s2[3])) +
                  (static_cast<u128>(static_cast<u64>(F.s2[4])) << 24);  // weight 2^72
  const u128 mid = (lo >> 64) + (hi << 8);
  const u128 p0 = static_cast<u128>(static_cast<u64>(lo)) * n;
  const u128 p1 = static_cast<u128>(static_cast<u64>(mid)) * n + (p0 >> 64);
  const u64 n0 = static_cast<u64>(p0), n1 = static_cast<u64>(p1);
  const u64 n2 = static_cast<u64>(mid >> 64) * n + static_cast<u64>(p1 >> 64);
  u64 d[4] = {n0 << 60, (n0 >> 4) | (n1 << 60), (n1 >> 4) | (n2 << 60), n2 >> 4};
  // minus (S1 2^60)^2
  const u128 q00 = static_cast<u128>(a0) * a0, q01 = static_cast<u128>(a0) * a1 << 1,
             q11 = static_cast<u128>(a1) * a1;
  const u128 c1 = (q00 >> 64) + static_cast<u64>(q01);
  const u128 c2 = (c1 >> 64) + (q01 >> 64) + static_cast<u64>(q11);
  const u64 sq[4] = {static_cast<u64>(q00), static_cast<u64>(c1), static_cast<u64>(c2),
                     static_cast<u64>(c2 >> 64) + static_cast<u64>(q11 >> 64)};
  u64 borrow = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const u128 v = static_cast<u128>(d[k]) - sq[k] - borrow;
    d[k] = static_cast<u64>(v);
    borrow = (v >> 127) != 0 ? 1 : 0;
  }
  // (the truncation of the scores can leave it negative where they are all alike)
  if (borrow || (d[0] | d[1] | d[2] | d[3]) == 0) return;
  int e;
  const u64 m = fix_top(d, &e);
  *m2 = fix_quotient(m, nn, rn) * fix_pow2(e - 120);
}

// Mean, standard error of the mean, path count and flags per node from the
// exact sums: se = sqrt(M2 / (n - 1) / n), 0 when every path started on the
// boundary (tau = 0, the estimate is exact) or with one path; NaN when a
// path was invalid or nothing was scored.  32 threads to a block: the warps'
// FP64 divisions and square roots run on an SM each.
constexpr int kFinalizeBlock = 32;
static __global__ void fix_finalize_kernel(const NodeFix *fix, int64_t n_nodes, double *mean,
                                           double *se, int64_t *npaths, int32_t *flags) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n_nodes) return;
  const NodeFix F = fix[i];
  const double nn = static_cast<double>(F.n);
  double m, M2;
  fix_moments(F, &m, &M2);
  const double e = F.n > 1 ? sqrt(M2 / ((nn - 1.0) * nn)) : M2;  // M2 is 0 or NaN for n <= 1
  mean[i] = m;
  se[i] = e;
  if (npaths) npaths[i] = F.n;
  if (flags) {
    int32_t f = 0;
    if (F.boundary > 0) f |= kNodeOnBoundary;
    if (F.bad > 0) f |= kNodeOutside;
    if (F.capped > 0) f |= kNodeCapped;
    if (F.n == 0) f |= kNodeEmpty;
    flags[i] = f;
  }
}

}  // namespace pdd
