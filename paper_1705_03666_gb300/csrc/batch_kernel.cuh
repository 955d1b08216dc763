// batch_kernel.cuh -- one persistent work-queue launch over a heterogeneous,
// ragged batch of interface nodes (several domains and PDE families, per-node
// time steps, per-node path counts).
//
// The launch runs the forward path kernel's scheme (forward_paths) on another
// source of paths: the nodes' path counts are prefix-summed (in device memory,
// so a launch sized on the host can consume a work list produced on the
// device, the adaptive pass, and the whole pipeline can be captured in a CUDA
// graph), a warp claims 32 consecutive paths of that list at a time, and a lane
// finds its path's node by bisection.  Node constants (the step constants, the
// start point in binary32) come from a per-node table formed once per call;
// a lane reads its path's when it takes it.  Scores go to the nodes' exact
// integer sums, so the result does not depend on which lane ran what.
//
// (Until the paths were claimed one by one, a lane ran runs of 256 paths of one
// node: on a list of 2000 nodes a third of the time was lanes without a run.
// 2000 nodes, 9.8e7 paths: 351 -> 118 ms, with the unit scheme.)
//
// The nodes are grouped by domain/family (a stable partition built on the
// device, `perm`), the list follows that order, and each family runs its own
// instantiation of the kernel over its own range: a kernel compiled for one
// family has the registers and the code of that family's path unit only.
#pragma once

#include "path_kernel.cuh"

namespace pdd {

constexpr int kMaxBatchProblems = 4;

// Domain/family combinations the batch kernel dispatches on.
enum : int32_t {
  kComboSquareLaplace = 0,   // LaplaceExpCos on Box<2>
  kComboLShapeLaplace = 1,   // LaplaceExpCos on LShape
  kComboCubeElliptic = 2,    // EllipticManufactured on Box<3>
  kComboSquarePoisson = 3    // PoissonFourier on Box<2>
};

template <int C> struct ComboTraits;
template <> struct ComboTraits<kComboSquareLaplace> { using M = LaplaceExpCos; using G = Box<2>; };
template <> struct ComboTraits<kComboLShapeLaplace> { using M = LaplaceExpCos; using G = LShape; };
template <> struct ComboTraits<kComboCubeElliptic> { using M = EllipticManufactured; using G = Box<3>; };
template <> struct ComboTraits<kComboSquarePoisson> { using M = PoissonFourier; using G = Box<2>; };

struct BatchProblem {
  ModelConst mc;
  int32_t combo;
  int32_t bridge;
  double sigma;
  double c_kill;  // constant killing rate (paper's c)
};

struct BatchNode {        // per node, formed once per call
  StepConst<float> k;
  float x[3];
  int32_t prob;
};

struct BatchArgs {
  int64_t n;
  // node order grouped by family: perm[j] is the node at position j; family c
  // holds positions [cstart[c], cstart[c+1])
  const int32_t *perm;
  const int64_t *cstart;
  // work list, in that order: the node at position j owns the list's paths
  // [off[j], off[j+1]), its paths first, first + 1, ...
  const int64_t *off;
  int64_t first;
  const BatchNode *table;      // [n]
  int32_t claim;               // paths a warp claims at a time (a multiple of 32)
  unsigned long long *cursor;  // [4]: one per family
  unsigned long long *counters;  // [0] path steps, [1] capped, [2] bad nodes
  NodeFix *fix;                // [n] exact per-node sums (both passes add to them)
  RoundKeys rk;
  int32_t max_steps;
  int32_t n_probs;
  BatchProblem probs[kMaxBatchProblems];
};

// The batch as a source of paths (see PathWork).  The path id is the node,
// with bit 32 set for the node's path 0.
template <int C>
struct BatchWork {
  using Env = PathEnv;
  using G = typename ComboTraits<C>::G;
  static constexpr int D = ComboTraits<C>::M::D;
  static constexpr bool kOwnConsts = true;
  const BatchArgs &a;
  const RoundKeys &rk;
  const double2 *normal_tables;
  NodeFix *fix;
  unsigned long long *counters;
  int32_t max_steps;
  int64_t jlo, jhi;              // the family's positions
  unsigned long long lo, hi;     // its paths of the list
  // the warp's claimed range of the list (warp-uniform)
  mutable unsigned long long next = 0, end = 0;
  __device__ __forceinline__ explicit BatchWork(const BatchArgs &b)
      : a(b), rk(b.rk), normal_tables(nullptr), fix(b.fix), counters(b.counters),
        max_steps(b.max_steps), jlo(b.cstart[C]), jhi(b.cstart[C + 1]) {
    lo = static_cast<unsigned long long>(b.off[jlo]);
    hi = static_cast<unsigned long long>(b.off[jhi]);
  }
  __device__ __forceinline__ Env env(unsigned long long id) const {
    const BatchProblem &p = a.probs[a.table[static_cast<uint32_t>(id)].prob];
    return Env{p.mc, p.bridge};
  }
  __device__ __forceinline__ StepConst<float> consts(unsigned long long id) const {
    return a.table[static_cast<uint32_t>(id)].k;
  }
  __device__ __forceinline__ uint64_t node(unsigned long long id) const {
    return static_cast<uint32_t>(id);
  }
  __device__ __forceinline__ bool first(unsigned long long id) const { return (id >> 32) != 0; }
  __device__ __forceinline__ bool claim(bool &exhausted, unsigned long long &id, uint64_t &node,
                                        PhiloxPath &pp, float *x) const {
    const unsigned lane = threadIdx.x & 31u;
    if (next >= end) {
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(a.cursor + C, static_cast<unsigned long long>(a.claim));
      next = lo + __shfl_sync(kFull, base, 0);
      end = next + a.claim < hi ? next + a.claim : hi;
    }
    const unsigned long long q = next + lane;
    next += 32;
    if (end == hi && next >= hi) exhausted = true;
    if (q >= end) return false;
    // position owning path q of the list: last j in [jlo, jhi) with off[j] <= q
    int64_t jl = jlo, jh = jhi;
    while (jh - jl > 1) {
      const int64_t mid = (jl + jh) >> 1;
      if (static_cast<unsigned long long>(a.off[mid]) <= q) jl = mid; else jh = mid;
    }
    const uint32_t i = static_cast<uint32_t>(a.perm[jl]);
    const uint32_t path = static_cast<uint32_t>(a.first + static_cast<int64_t>(q) - a.off[jl]);
    node = i;
    id = i | (path == 0u ? 1ull << 32 : 0ull);
    pp = philox_path(path, i, 0u, rk);
#pragma unroll
    for (int d = 0; d < D; ++d) x[d] = a.table[i].x[d];
    return true;
  }
  __device__ __forceinline__ void dump(unsigned long long, float, int32_t, const float *) const {}
};

template <int C>
__global__ void __launch_bounds__(kForwardBlock, 7) batch_kernel(const __grid_constant__ BatchArgs a) {
  if (a.cstart[C] >= a.cstart[C + 1]) return;
  forward_paths<typename ComboTraits<C>::M, typename ComboTraits<C>::G, float>(BatchWork<C>(a));
}

}  // namespace pdd
