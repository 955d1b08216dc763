// stage2_3d.cu -- stage two of PDD in three dimensions (Sec. 2.1, Fig. 2.2):
// the independent subdomain solves of the elliptic problem
//   (1/2) sigma^2 Lap u + b . grad u + c u + f = 0   (Eq. 2.3 without time)
// by 7-point second differences and central first differences (the interface
// interpolation that feeds them is in rbf.cu).
//
// Subdomain solve (pdd_subdomain_solve with a 3-D grid): defect correction
//   u <- u + P^{-1} (rhs - A u)
// with A the full operator (FP64 residual) and P its constant-coefficient part
// (1/2) sigma^2 Lap_h + c, which the three-dimensional discrete sine
// transform diagonalises on a box with Dirichlet data.  P^{-1} is applied in
// binary32 (three dense passes of the sine matrices, a division by the
// eigenvalues, three passes back); the drift is a small perturbation of P on
// a subdomain (|b| / |grad| against the Laplacian's scale), so the error
// contracts by roughly ten per iteration, down to the FP64 residual
// tolerance.  A plain Jacobi sweep is kept as the reference method.
//
// A correction is four launches: the residual (its last block per box forms
// the norm and decides whether the box goes on, so the host only looks one
// correction behind), the forward y and x passes of each z plane, the z pass
// with the eigenvalues and its inverse for 32 columns at a time, and the
// inverse y and x passes with the update.  What bounds it is the FP64 pipe
// (1/64 rate: the residual takes 14 FP64 instructions per point), then launch
// gaps; the transforms run out of shared memory.  FP64 work that does not
// change between corrections (drift over 2h, the eigenvalue factors) is formed
// once per call.  Measured on the 64 boxes of 33^3 points of the 4 x 4 x 4 split
// (eight residuals, seven corrections; device time): residuals 2.27 -> 0.56 ms
// (64-bit index divisions, three FP64 divisions per thread and three arrays of
// drift before), transforms 3.70 -> 0.55 ms (one output per thread with two
// shared loads per FMA, and the residual rescaled in FP64 for each of a row's
// 31 products, before), eigenvalues 1.45 -> 0.01 ms, set-up 0.46 -> 0.08 ms, and
// no host round trip per correction; the call 8.3 -> 1.6 ms.
#include <cmath>
#include <cstring>
#include <vector>

#include "ctx.hpp"
#include "models.cuh"

namespace pdd {

// ---------------------------------------------------------------------------
// Subdomain solves on 3-D boxes.  The subdomains of stage two are independent
// problems (Sec. 2), so one call solves a batch of boxes of the same grid
// size together: every kernel below takes the box from blockIdx.y, and a box
// whose correction loop has stopped is skipped (live[b] == 0).  A batch of
// one box is the single solve; each box's arithmetic does not depend on the
// others, so a box gets the same bits alone or in a batch.
// ---------------------------------------------------------------------------
constexpr int kBox3MaxInterior = 126;  // interior points per axis (sine matrix in shared memory)
constexpr int kBox3Block = 256;
constexpr int kBox3Axis = kBox3MaxInterior + 2;  // grid points per axis

struct Box3 {
  double lo[3], h[3];
  int n[3];           // grid points per axis, boundary included
  int P[3];           // interior points per axis
  double w[3], diag;  // (sigma^2 / 2) / h_a^2 and the operator's diagonal
  int mask;           // bit 2a + side: that face carries interface data
  int next;           // bit 2a + 1: that face's points are written by the next box along a
  int face_ld[6];       // row length of each face's data (its slow axis)
  int64_t face_off[6];  // offset of each face's data in the caller's array
  // the box's grid in the caller's array: point (i, j, k) is at u_off + k u_sz
  // + j u_sy + i (a box of its own, or a block of one global grid: of the boxes
  // that share a point the last along every axis writes it, as its first: g on
  // a shared edge of the cube's boundary depends on the last bit of the
  // coordinate, and lo + h (n - 1) is not always the next box's lo)
  int64_t u_off, u_sz;
  int u_sy;
};

__device__ __forceinline__ int64_t box3_index(const Box3 &B, int i, int j, int k) {
  return B.u_off + k * B.u_sz + static_cast<int64_t>(j) * B.u_sy + i;
}
__device__ __forceinline__ int64_t box3_np(const Box3 &B) {
  return static_cast<int64_t>(B.P[0]) * B.P[1] * B.P[2];
}

// Dirichlet data and coefficients, one block per z plane and box: boundary
// layer of u from the faces (a point on a face without interface data -- the
// physical boundary -- takes g; otherwise the interface face of lowest index),
// interior u = 0, and per interior point b and f of the family.  The family's
// functions of one coordinate are tabulated per block (a few dozen FP64
// sines and exponentials in place of three per point).  kTables: in place of
// the arrays of b, the blocks of the first plane write b_a / (2 h_a) at the grid
// points of the coordinate it depends on, drift[box][a][index].
template <class Model, bool kTables>
__global__ void __launch_bounds__(kBox3Block)
box3_setup_kernel(const Box3 *boxes, ModelConst mc, const double *face, double *u, double *coef,
                  double *drift) {
  const Box3 B = boxes[blockIdx.y];
  const int k = blockIdx.x;
  const int64_t np = box3_np(B);
  u += B.u_off + k * B.u_sz;
  coef += blockIdx.y * (kTables ? 1 : 4) * np;
  __shared__ typename Model::AxisTable tab[3][kBox3Axis];
  for (int e = threadIdx.x; e < B.n[0] + B.n[1] + 1; e += blockDim.x) {
    const int a = e < B.n[0] ? 0 : (e < B.n[0] + B.n[1] ? 1 : 2);
    const int i = a == 0 ? e : (a == 1 ? e - B.n[0] : k);
    tab[a][a == 2 ? 0 : i] = Model::axis_table(a, B.lo[a] + B.h[a] * i);
  }
  __syncthreads();
  if constexpr (kTables) {
    if (k == 0)
      for (int e = threadIdx.x; e < 2 * kBox3Axis; e += blockDim.x) {
        const int a = e / kBox3Axis, i = e % kBox3Axis, on = Model::drift_axis(a);
        if (!((Model::kDriftAxes >> a) & 1u) || i >= B.n[on]) continue;
        double b[3], f;
        Model::coeffs_tab(tab[0][on == 0 ? i : 0], tab[1][on == 1 ? i : 0], tab[2][0], b, f);
        drift[(blockIdx.y * 2 + a) * kBox3Axis + i] = b[a] * (0.5 / B.h[a]);
      }
  }
  for (int e = threadIdx.x; e < B.n[0] * B.n[1]; e += blockDim.x) {
    const int j = e / B.n[0], i = e - j * B.n[0];
    const int idx[3] = {i, j, k};
    double *ue = u + static_cast<int64_t>(j) * B.u_sy + i;
    const bool interior = i > 0 && j > 0 && k > 0 && i < B.n[0] - 1 && j < B.n[1] - 1 &&
                          k < B.n[2] - 1;
    if (interior) {
      *ue = 0.0;
      double b[3], f = 0.0;
      Model::coeffs_tab(tab[0][i], tab[1][j], tab[2][0], b, f);
      const int64_t q = (static_cast<int64_t>(k - 1) * B.P[1] + (j - 1)) * B.P[0] + (i - 1);
      if constexpr (!kTables) {
#pragma unroll
        for (int a = 0; a < 3; ++a) coef[a * np + q] = b[a];
      }
      coef[(kTables ? 0 : 3) * np + q] = f;
      continue;
    }
    bool physical = false, next = false;
    int fbest = -1;
    for (int fc = 0; fc < 6; ++fc) {
      const int a = fc >> 1, side = fc & 1;
      const bool on = side ? idx[a] == B.n[a] - 1 : idx[a] == 0;
      if (!on) continue;
      next |= ((B.next >> fc) & 1) != 0;
      if ((B.mask >> fc) & 1) {
        if (fbest < 0) fbest = fc;
      } else {
        physical = true;
      }
    }
    if (next) continue;
    double v;
    if (physical || fbest < 0) {
      v = Model::g_tab(tab[0][i], tab[1][j], tab[2][0]);
    } else {
      // face grid of face fbest: the two other axes, the higher one slow
      const int a = fbest >> 1;
      const int a1 = a == 0 ? 1 : 0, a2 = a == 2 ? 1 : 2;
      v = face[B.face_off[fbest] + static_cast<int64_t>(idx[a2]) * B.face_ld[fbest] + idx[a1]];
    }
    *ue = v;
  }
}

// Correction state of the boxes (device arrays, one entry per box, but
// n_live): norm of the residual, its inverse, the first norm, their ratio, the
// corrections done, whether the box goes on, and the ticket of its blocks.
struct Box3State {
  double *rn, *inv, *r0, *res;
  int64_t *iters;
  int32_t *live, *ticket;
  int32_t *n_live;
};

// r = -f - A u at the interior points (FP64), one block per z plane and box,
// and the block's sum of r^2; the box's last block adds the planes' sums in a
// fixed order, forms the norm and decides whether the box goes on (stopping
// rule of correction `it`).
template <class Model>
__global__ void __launch_bounds__(kBox3Block)
box3_residual_kernel(const Box3 *boxes, const __grid_constant__ Box3State st, const double *u,
                     const double *f, const double *drift, double *r, double *part,
                     int64_t it, int64_t max_iter, double tol) {
  static_assert(Model::kDriftAxes == 3u && Model::drift_axis(0) == 1 && Model::drift_axis(1) == 0,
                "b_0(y), b_1(x), no drift along z");
  const int box = blockIdx.y;
  if (!st.live[box]) return;
  const Box3 B = boxes[box];
  const int64_t np = box3_np(B);
  const int plane = B.P[0] * B.P[1];
  const int64_t q0 = static_cast<int64_t>(blockIdx.x) * plane;
  const int64_t sy = B.u_sy, sz = B.u_sz;
  u += box3_index(B, 1, 1, static_cast<int>(blockIdx.x) + 1);
  f += box * np + q0;
  r += box * np + q0;
  const double *b0 = drift + (box * 2) * kBox3Axis + 1, *b1 = b0 + kBox3Axis;
  const double w0 = B.w[0], w1 = B.w[1], w2 = B.w[2], diag = B.diag;
  double acc = 0.0;
#pragma unroll 2
  for (int q = threadIdx.x; q < plane; q += kBox3Block) {
    const int j = q / B.P[0], i = q - j * B.P[0];
    const double *v = u + j * sy + i;
    const double ux0 = v[-1], ux1 = v[1], uy0 = v[-sy], uy1 = v[sy], uz0 = v[-sz], uz1 = v[sz];
    double Au = diag * v[0] + w0 * (ux0 + ux1) + w1 * (uy0 + uy1) + w2 * (uz0 + uz1);
    Au += fma(b1[i], uy1 - uy0, b0[j] * (ux1 - ux0));
    const double rv = -f[q] - Au;
    r[q] = rv;
    acc = fma(rv, rv, acc);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
  __shared__ double sh[kBox3Block / 32];
  __shared__ bool last;
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kBox3Block / 32; ++w) t += sh[w];
    part[static_cast<int64_t>(box) * gridDim.x + blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(st.ticket + box, 1) == static_cast<int>(gridDim.x) - 1;
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return;
  __threadfence();
  double t = 0.0;
  for (unsigned k = threadIdx.x; k < gridDim.x; k += 32)
    t += __ldcg(part + static_cast<int64_t>(box) * gridDim.x + k);
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
  if (threadIdx.x == 0) {
    const double rn = sqrt(t);
    if (it == 0) st.r0[box] = rn;
    const double r0 = it == 0 ? rn : st.r0[box];
    st.rn[box] = rn;
    st.inv[box] = 1.0 / rn;
    st.iters[box] = it;
    st.res[box] = r0 > 0.0 ? rn / r0 : 0.0;
    st.ticket[box] = 0;
    if (rn <= tol * r0 || rn == 0.0 || it >= max_iter) {
      st.live[box] = 0;
      atomicSub(st.n_live, 1);
    }
  }
}

// Jacobi: per box the largest of its block partials; one thread per box.
__global__ void box3_combine_kernel(const double *part, int nblk, int nb, const int32_t *live,
                                    double *out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb || !live[b]) return;
  double t = 0.0;
  for (int k = 0; k < nblk; ++k) {
    t = fmax(t, part[static_cast<int64_t>(b) * nblk + k]);
  }
  out[b] = t;
}

// Rows of the sine matrices and of the staged planes are padded to a multiple
// of four floats, so that four consecutive entries are one 16-byte load.
__host__ __device__ constexpr int box3_pad(int P) { return (P + 3) & ~3; }

// The sine matrices S_a[k][j] = sin(pi (k+1)(j+1) / (P_a + 1)), binary32,
// rows padded with zeros, the argument reduced exactly in integers; blockIdx.y
// is the axis.  Also the eigenvalue factors of the 1-D second differences,
// cos(pi (k+1) / (P_a + 1)) - 1.
struct Box3Sines {
  float *S[3];
  double *cm1[3];
};
__global__ void box3_sine_kernel(int P0, int P1, int P2, const __grid_constant__ Box3Sines T) {
  const int a = blockIdx.y;
  const int P = a == 0 ? P0 : (a == 1 ? P1 : P2), ld = box3_pad(P);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < P * ld; e += gridDim.x * blockDim.x) {
    const int k = e / ld + 1, j = e % ld + 1;
    const int m = (k * j) % (2 * (P + 1));
    T.S[a][e] = j <= P ? static_cast<float>(sinpi(static_cast<double>(m) / (P + 1))) : 0.0f;
    if (e < P) T.cm1[a][e] = cospi(static_cast<double>(e + 1) / (P + 1)) - 1.0;
  }
}

// Factors of the division by the eigenvalues of (1/2) sigma^2 Lap_h + c in the
// sine basis, lambda = sum_a (sigma^2 / h_a^2) (cos(pi k_a / (P_a + 1)) - 1) +
// c, with the normalisation of the two transforms: (8 / prod_a (P_a + 1)) /
// lambda (FP64, formed once per call; one table for boxes of one mesh size).
__global__ void box3_eig_kernel(const Box3 *boxes, const __grid_constant__ Box3Sines T, double s2,
                                double c, double *fac) {
  const Box3 B = boxes[blockIdx.y];
  const int plane = B.P[0] * B.P[1];
  fac += blockIdx.y * box3_np(B) + static_cast<int64_t>(blockIdx.x) * plane;
  const double norm = 8.0 / ((B.P[0] + 1.0) * (B.P[1] + 1.0) * (B.P[2] + 1.0));
  const double e0 = s2 / (B.h[0] * B.h[0]), e1 = s2 / (B.h[1] * B.h[1]),
               e2 = s2 / (B.h[2] * B.h[2]);
  for (int q = threadIdx.x; q < plane; q += blockDim.x) {
    const int k1 = q / B.P[0], k0 = q - k1 * B.P[0];
    fac[q] = norm / (e0 * T.cm1[0][k0] + e1 * T.cm1[1][k1] + e2 * T.cm1[2][blockIdx.x] + c);
  }
}

// out[a][k] = sum_i Bc[i][a] V[i][k] (a < A, k < N, i < K ascending), the
// block's warps sharing the output: a lane forms four consecutive a of one k
// per turn (one 16-byte broadcast load, one load and four FMAs per i), and
// passes them to put(a, k, v[4]) (entries at a + q >= A are padding).
template <class Put>
__device__ __forceinline__ void box3_apply(const float *Bc, int ldb, const float *V, int ldv, int K,
                                           int A, int N, Put put) {
  const int lane = threadIdx.x & 31, nag = (A + 3) / 4, nkc = (N + 31) / 32;
  for (int t = threadIdx.x >> 5; t < nag * nkc; t += kBox3Block / 32) {
    const int kc = t / nag, a = 4 * (t - kc * nag), k = kc * 32 + lane;
    const float *b = Bc + a, *v = V + min(k, N - 1);
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 4
    for (int i = 0; i < K; ++i) {
      const float4 w = *reinterpret_cast<const float4 *>(b + i * ldb);
      const float x = v[i * ldv];
      s0 = fmaf(w.x, x, s0);
      s1 = fmaf(w.y, x, s1);
      s2 = fmaf(w.z, x, s2);
      s3 = fmaf(w.w, x, s3);
    }
    if (k < N) {
      const float s[4] = {s0, s1, s2, s3};
      put(a, k, s);
    }
  }
}

// Row length of the transposed plane: four more than the padded row, so that
// the 16-byte stores of neighbouring lanes fall on different banks.
__host__ __device__ constexpr int box3_pad_t(int P) { return box3_pad(P) + 4; }
static size_t box3_plane_smem(int P0, int P1) {
  const size_t l = static_cast<size_t>(P0) * box3_pad(P0) + static_cast<size_t>(P0) * box3_pad_t(P1) +
                   static_cast<size_t>(P1) * P0;
  return l * sizeof(float);
}

// The y and x passes of one z plane (blockIdx.x) of box blockIdx.y.  kInverse
// = false: in is the FP64 residual, scaled by 1 / |r|_2 (scale) and rounded, and
// the result goes to v.  kInverse = true: in place of the residual v, and the
// result times |r|_2 (scale) is added to u.  The sine matrix along x sits in shared
// memory; along y it is the same one when the box is as long, else read
// through L1.
template <bool kInverse>
__global__ void __launch_bounds__(kBox3Block)
box3_plane_kernel(const Box3 *boxes, const int32_t *live, const double *scale,
                  const __grid_constant__ Box3Sines T, const double *r, float *v, double *u) {
  const int box = blockIdx.y;
  if (!live[box]) return;
  extern __shared__ __align__(16) float bsm[];
  const Box3 B = boxes[box];
  const int P0 = B.P[0], P1 = B.P[1], plane = P0 * P1;
  const int ld0 = box3_pad(P0), ldt = box3_pad_t(P1);
  float *Sx = bsm;               // [P0][ld0]
  float *Tt = Sx + P0 * ld0;     // [x][y]: after the y pass
  float *Tn = Tt + P0 * ldt;     // [y][x]: the plane
  const int64_t off = box * box3_np(B) + static_cast<int64_t>(blockIdx.x) * plane;
  const double sc = scale[box];
  for (int e = threadIdx.x; e < P0 * ld0; e += kBox3Block) Sx[e] = T.S[0][e];
  for (int e = threadIdx.x; e < plane; e += kBox3Block)
    Tn[e] = kInverse ? v[off + e] : static_cast<float>(r[off + e] * sc);
  __syncthreads();
  const float *Sy = P1 == P0 ? Sx : T.S[1];
  box3_apply(Sy, box3_pad(P1), Tn, P0, P1, P1, P0, [&](int a, int k, const float *s) {
    *reinterpret_cast<float4 *>(Tt + k * ldt + a) = make_float4(s[0], s[1], s[2], s[3]);
  });
  __syncthreads();
  if constexpr (kInverse) {
    double *up = u + box3_index(B, 1, 1, static_cast<int>(blockIdx.x) + 1);
    box3_apply(Tt, ldt, Sx, ld0, P0, P1, P0, [&](int a, int k, const float *s) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (a + q < P1) {
          double *p = up + static_cast<int64_t>(a + q) * B.u_sy + k;
          *p = fma(static_cast<double>(s[q]), sc, *p);
        }
    });
  } else {
    float *vp = v + off;
    box3_apply(Tt, ldt, Sx, ld0, P0, P1, P0, [&](int a, int k, const float *s) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (a + q < P1) vp[(a + q) * P0 + k] = s[q];
    });
  }
}

// The z pass of 32 columns (blockIdx.x), the division by the eigenvalues and
// the inverse z pass, in place.
constexpr int kBox3Cols = 32;
static size_t box3_z_smem(int P2) {
  return (static_cast<size_t>(P2) * box3_pad(P2) + 2 * static_cast<size_t>(P2) * kBox3Cols) * sizeof(float);
}
__global__ void __launch_bounds__(kBox3Block)
box3_z_kernel(int P0, int P1, int P2, const int32_t *live, const __grid_constant__ Box3Sines T,
              const double *fac, int64_t fac_stride, float *v) {
  const int box = blockIdx.y;
  if (!live[box]) return;
  extern __shared__ __align__(16) float bsm[];
  const int ld = box3_pad(P2), plane = P0 * P1;
  float *S = bsm;                    // [P2][ld]
  float *V = S + P2 * ld;            // [P2][32]
  float *H = V + P2 * kBox3Cols;     // [P2][32]
  const int c0 = blockIdx.x * kBox3Cols, nc = min(kBox3Cols, plane - c0);
  v += box * static_cast<int64_t>(plane) * P2 + c0;
  fac += box * fac_stride + c0;
  for (int e = threadIdx.x; e < P2 * ld; e += kBox3Block) S[e] = T.S[2][e];
  for (int e = threadIdx.x; e < P2 * kBox3Cols; e += kBox3Block) {
    const int z = e / kBox3Cols, c = e % kBox3Cols;
    if (c < nc) V[e] = v[static_cast<int64_t>(z) * plane + c];
  }
  __syncthreads();
  box3_apply(S, ld, V, kBox3Cols, P2, P2, nc, [&](int a, int k, const float *s) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (a + q < P2)
        H[(a + q) * kBox3Cols + k] = static_cast<float>(
            static_cast<double>(s[q]) * fac[static_cast<int64_t>(a + q) * plane + k]);
  });
  __syncthreads();
  box3_apply(S, ld, H, kBox3Cols, P2, P2, nc, [&](int a, int k, const float *s) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (a + q < P2) v[static_cast<int64_t>(a + q) * plane + k] = s[q];
  });
}

// One Jacobi sweep (the plain reference method): u' = (-f - offdiag(A) u) / diag,
// the block's largest change in part[box][block].
__global__ void __launch_bounds__(kBox3Block)
box3_jacobi_kernel(const Box3 *boxes, const int32_t *live, double s2, double c, const double *u,
                   double *un, const double *coef, double *part) {
  if (!live[blockIdx.y]) return;
  const Box3 B = boxes[blockIdx.y];
  const int64_t np = box3_np(B);
  coef += blockIdx.y * 4 * np;
  const double w0 = 0.5 * s2 / (B.h[0] * B.h[0]), w1 = 0.5 * s2 / (B.h[1] * B.h[1]),
               w2 = 0.5 * s2 / (B.h[2] * B.h[2]);
  const double d0 = 0.5 / B.h[0], d1 = 0.5 / B.h[1], d2 = 0.5 / B.h[2];
  const double diag = c - 2.0 * (w0 + w1 + w2);
  double mx = 0.0;
  for (int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < np;
       q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int i = static_cast<int>(q % B.P[0]) + 1;
    const int j = static_cast<int>((q / B.P[0]) % B.P[1]) + 1;
    const int k = static_cast<int>(q / (static_cast<int64_t>(B.P[0]) * B.P[1])) + 1;
    const int64_t e = box3_index(B, i, j, k);
    const int64_t sy = B.u_sy, sz = B.u_sz;
    const double ux0 = u[e - 1], ux1 = u[e + 1], uy0 = u[e - sy], uy1 = u[e + sy],
                 uz0 = u[e - sz], uz1 = u[e + sz];
    const double off = (w0 - coef[q] * d0) * ux0 + (w0 + coef[q] * d0) * ux1 +
                       (w1 - coef[np + q] * d1) * uy0 + (w1 + coef[np + q] * d1) * uy1 +
                       (w2 - coef[2 * np + q] * d2) * uz0 + (w2 + coef[2 * np + q] * d2) * uz1;
    const double v = (-coef[3 * np + q] - off) / diag;
    mx = fmax(mx, fabs(v - u[e]));
    un[e] = v;
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(kFull, mx, o));
  __shared__ double sh[kBox3Block / 32];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kBox3Block / 32; ++w) t = fmax(t, sh[w]);
    part[static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x] = t;
  }
}

// Blocks of a Jacobi sweep over np interior points.
static int box3_blocks(int64_t np) {
  return static_cast<int>(std::min<int64_t>((np + kBox3Block - 1) / kBox3Block, 1024));
}
// Scratch of a batch of boxes (offsets).
struct Box3Layout {
  size_t it, res, state_bytes, rn, inv, r0, live, ticket, nlive, box, coef, drift, part, un, r, fac, v,
      S[3], cm1[3], total;
  bool one_h;  // boxes of one mesh size share one table of eigenvalue factors
};
static Box3Layout box3_layout(const std::vector<Box3> &boxes, bool jacobi, int64_t u_span) {
  const Box3 &B0 = boxes[0];
  const size_t NB = boxes.size();
  const int64_t np = static_cast<int64_t>(B0.P[0]) * B0.P[1] * B0.P[2];
  Box3Layout L;
  L.one_h = true;
  for (const Box3 &B : boxes)
    for (int a = 0; a < 3; ++a) L.one_h = L.one_h && B.h[a] == B0.h[a];
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align_up(o + bytes, 256);
    return at;
  };
  // the boxes' state first: one copy back at the end
  L.it = take(NB * sizeof(int64_t));
  L.res = take(NB * sizeof(double));
  L.state_bytes = o;
  L.rn = take(NB * sizeof(double));
  L.inv = take(NB * sizeof(double));
  L.r0 = take(NB * sizeof(double));
  L.live = take(NB * sizeof(int32_t));
  L.ticket = take(NB * sizeof(int32_t));
  L.nlive = take(sizeof(int32_t));
  L.box = take(NB * sizeof(Box3));
  L.coef = take(NB * (jacobi ? 4 : 1) * np * sizeof(double));
  L.drift = take(NB * 2 * kBox3Axis * sizeof(double));
  L.part = take(NB * std::max(box3_blocks(np), B0.P[2]) * sizeof(double));
  L.un = take(jacobi ? u_span * sizeof(double) : 0);
  L.r = take(jacobi ? 0 : NB * np * sizeof(double));
  L.fac = take(jacobi ? 0 : (L.one_h ? 1 : NB) * np * sizeof(double));
  L.v = take(jacobi ? 0 : NB * np * sizeof(float));
  for (int a = 0; a < 3; ++a) {
    L.S[a] = take(static_cast<size_t>(B0.P[a]) * box3_pad(B0.P[a]) * sizeof(float));
    L.cm1[a] = take(static_cast<size_t>(B0.P[a]) * sizeof(double));
  }
  L.total = o;
  return L;
}

// The boxes' solves (one grid size and method; faces and grids where the boxes
// say, u_span values of d_u in all).  *iters and *resid (if non-null) get the
// largest count and relative residual over the boxes; iters_each / resid_each
// (host, one entry per box, may be null) get each box's own.
static pdd_status solve_boxes(pdd_ctx *ctx, std::vector<Box3> &boxes, int32_t method,
                              int64_t max_iter, double tol, const double *d_face, double *d_u,
                              int64_t u_span, int64_t *iters, double *resid, int64_t *iters_each,
                              double *resid_each) {
  const double s2 = ctx->prob.sigma * ctx->prob.sigma;
  const double c = constant_kill(ctx->prob.kind);
  for (Box3 &B : boxes) {
    for (int a = 0; a < 3; ++a) B.w[a] = 0.5 * s2 / (B.h[a] * B.h[a]);
    B.diag = c - 2.0 * (B.w[0] + B.w[1] + B.w[2]);
  }
  const int32_t nb = static_cast<int32_t>(boxes.size());
  const Box3 &B0 = boxes[0];
  const bool jacobi = method == PDD_STENCIL_JACOBI;
  const int64_t np = static_cast<int64_t>(B0.P[0]) * B0.P[1] * B0.P[2];
  const size_t NB = static_cast<size_t>(nb);
  const int nblk = box3_blocks(np);
  const Box3Layout L = box3_layout(boxes, jacobi, u_span);
  const bool one_h = L.one_h;
  pdd_status st = ensure_scratch(ctx, L.total);
  if (st != PDD_OK) return st;
  char *base = static_cast<char *>(ctx->scratch);
  double *rn = reinterpret_cast<double *>(base + L.rn);  // per box: |r|_2 (Jacobi: largest change)
  int32_t *live = reinterpret_cast<int32_t *>(base + L.live);
  Box3 *d_boxes = reinterpret_cast<Box3 *>(base + L.box);
  double *coef = reinterpret_cast<double *>(base + L.coef);
  double *drift = reinterpret_cast<double *>(base + L.drift);
  double *part = reinterpret_cast<double *>(base + L.part);
  double *un = reinterpret_cast<double *>(base + L.un);

  // host state of the correction loop (copied to and from the device
  // synchronously, so these buffers outlive every copy)
  std::vector<int32_t> h_live(NB, 1);
  std::vector<double> h_rn(NB, 0.0), h_res(NB, 0.0);
  std::vector<int64_t> h_it(NB, 0);
  PDD_CUDA_TRY(ctx, cudaMemcpyAsync(d_boxes, boxes.data(), NB * sizeof(Box3),
                                    cudaMemcpyHostToDevice, ctx->stream));
  PDD_CUDA_TRY(ctx, cudaMemcpyAsync(live, h_live.data(), NB * sizeof(int32_t),
                                    cudaMemcpyHostToDevice, ctx->stream));
  const dim3 gset(static_cast<unsigned>(B0.n[2]), nb);
  if (jacobi)
    box3_setup_kernel<EllipticManufactured, false><<<gset, kBox3Block, 0, ctx->stream>>>(
        d_boxes, ctx->mc, d_face, d_u, coef, drift);
  else
    box3_setup_kernel<EllipticManufactured, true><<<gset, kBox3Block, 0, ctx->stream>>>(
        d_boxes, ctx->mc, d_face, d_u, coef, drift);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  const unsigned gcomb = static_cast<unsigned>((nb + 127) / 128);
  const auto ev = prof_slot(ctx);
  if (ev.first) PDD_CUDA_TRY(ctx, cudaEventRecord(ev.first, ctx->stream));
  // read the per-box measures, then decide per box whether it goes on
  auto read_measures = [&]() -> pdd_status {
    PDD_CUDA_TRY(ctx, cudaMemcpyAsync(h_rn.data(), rn, NB * sizeof(double), cudaMemcpyDeviceToHost,
                                      ctx->stream));
    PDD_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return PDD_OK;
  };
  auto push_live = [&]() -> pdd_status {
    PDD_CUDA_TRY(ctx, cudaMemcpyAsync(live, h_live.data(), NB * sizeof(int32_t),
                                      cudaMemcpyHostToDevice, ctx->stream));
    return PDD_OK;
  };
  if (jacobi) {
    // each box sweeps between its own two buffers; a box that stops keeps its
    // latest iterate where its own step count left it
    PDD_CUDA_TRY(ctx, cudaMemcpyAsync(un, d_u, u_span * sizeof(double),
                                      cudaMemcpyDeviceToDevice, ctx->stream));
    const unsigned gj = static_cast<unsigned>(nblk);
    int n_live = nb;
    for (int64_t it = 1; it <= max_iter && n_live > 0; ++it) {
      const bool odd = (it & 1) != 0;
      box3_jacobi_kernel<<<dim3(gj, nb), kBox3Block, 0, ctx->stream>>>(
          d_boxes, live, s2, c, odd ? d_u : un, odd ? un : d_u, coef, part);
      PDD_CUDA_TRY(ctx, cudaGetLastError());
      for (size_t b = 0; b < NB; ++b)
        if (h_live[b]) h_it[b] = it;
      if (it % 16 == 0 || it == max_iter) {
        box3_combine_kernel<<<gcomb, 128, 0, ctx->stream>>>(part, nblk, nb, live, rn);
        PDD_CUDA_TRY(ctx, cudaGetLastError());
        st = read_measures();
        if (st != PDD_OK) return st;
        for (size_t b = 0; b < NB; ++b) {
          if (!h_live[b]) continue;
          h_res[b] = h_rn[b];
          if (h_rn[b] < tol || it == max_iter) {
            h_live[b] = 0;
            --n_live;
          }
        }
        st = push_live();
        if (st != PDD_OK) return st;
      }
    }
    // a box whose last sweep was odd holds its iterate in un
    for (size_t b = 0; b < NB; ++b) {
      if (!(h_it[b] & 1)) continue;
      const Box3 &B = boxes[b];
      for (int k = 0; k < B.n[2]; ++k)
        PDD_CUDA_TRY(ctx, cudaMemcpy2DAsync(d_u + B.u_off + k * B.u_sz, B.u_sy * sizeof(double),
                                            un + B.u_off + k * B.u_sz, B.u_sy * sizeof(double),
                                            B.n[0] * sizeof(double), static_cast<size_t>(B.n[1]),
                                            cudaMemcpyDeviceToDevice, ctx->stream));
    }
  } else {
    st = ensure_watch(ctx);
    if (st != PDD_OK) return st;
    Box3Sines T;
    for (int a = 0; a < 3; ++a) {
      T.S[a] = reinterpret_cast<float *>(base + L.S[a]);
      T.cm1[a] = reinterpret_cast<double *>(base + L.cm1[a]);
    }
    Box3State S;
    S.rn = rn;
    S.inv = reinterpret_cast<double *>(base + L.inv);
    S.r0 = reinterpret_cast<double *>(base + L.r0);
    S.res = reinterpret_cast<double *>(base + L.res);
    S.iters = reinterpret_cast<int64_t *>(base + L.it);
    S.live = live;
    S.ticket = reinterpret_cast<int32_t *>(base + L.ticket);
    S.n_live = reinterpret_cast<int32_t *>(base + L.nlive);
    double *r = reinterpret_cast<double *>(base + L.r);
    double *fac = reinterpret_cast<double *>(base + L.fac);
    float *v = reinterpret_cast<float *>(base + L.v);
    PDD_CUDA_TRY(ctx, cudaMemsetAsync(S.ticket, 0, NB * sizeof(int32_t), ctx->stream));
    const int32_t h_nlive = nb;
    PDD_CUDA_TRY(ctx, cudaMemcpyAsync(S.n_live, &h_nlive, sizeof h_nlive, cudaMemcpyHostToDevice,
                                      ctx->stream));
    const int P0 = B0.P[0], P1 = B0.P[1], P2 = B0.P[2];
    const int Pm = std::max(P0, std::max(P1, P2));
    box3_sine_kernel<<<dim3(static_cast<unsigned>((Pm * box3_pad(Pm) + 255) / 256), 3), 256, 0, ctx->stream>>>(
        P0, P1, P2, T);
    PDD_CUDA_TRY(ctx, cudaGetLastError());
    const dim3 gp(static_cast<unsigned>(P2), nb);
    box3_eig_kernel<<<dim3(static_cast<unsigned>(P2), one_h ? 1u : static_cast<unsigned>(nb)),
                      kBox3Block, 0, ctx->stream>>>(d_boxes, T, s2, c, fac);
    PDD_CUDA_TRY(ctx, cudaGetLastError());
    const size_t smem_p = box3_plane_smem(P0, P1);
    const size_t smem_z = box3_z_smem(P2);
    // (the limits belong to the kernels on the device, not to this call: constants,
    // so that a call with small boxes lowers nothing under another thread's solve)
    const int lim_p = static_cast<int>(box3_plane_smem(kBox3MaxInterior, kBox3MaxInterior));
    const int lim_z = static_cast<int>(box3_z_smem(kBox3MaxInterior));
    PDD_CUDA_TRY(ctx, cudaFuncSetAttribute(box3_plane_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim_p));
    PDD_CUDA_TRY(ctx, cudaFuncSetAttribute(box3_plane_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim_p));
    PDD_CUDA_TRY(ctx, cudaFuncSetAttribute(box3_z_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim_z));
    const dim3 gz(static_cast<unsigned>((P0 * P1 + kBox3Cols - 1) / kBox3Cols), nb);
    const int64_t fac_stride = one_h ? 0 : np;
    // The boxes stop themselves.  The host looks at their number one
    // correction behind (a copy into pinned memory and an event), so the
    // device never waits for it; what it enqueues after the last box has
    // stopped returns at once.
    for (int64_t it = 0;; ++it) {
      box3_residual_kernel<EllipticManufactured><<<gp, kBox3Block, 0, ctx->stream>>>(
          d_boxes, S, d_u, coef, drift, r, part, it, max_iter, tol);
      PDD_CUDA_TRY(ctx, cudaMemcpyAsync(ctx->watch + (it & 1), S.n_live, sizeof(int32_t),
                                        cudaMemcpyDeviceToHost, ctx->stream));
      PDD_CUDA_TRY(ctx, cudaEventRecord(ctx->watch_ev[it & 1], ctx->stream));
      if (it > 0) {
        PDD_CUDA_TRY(ctx, cudaEventSynchronize(ctx->watch_ev[(it - 1) & 1]));
        if (ctx->watch[(it - 1) & 1] == 0) break;
      }
      box3_plane_kernel<false><<<gp, kBox3Block, smem_p, ctx->stream>>>(d_boxes, live, S.inv, T, r, v, nullptr);
      box3_z_kernel<<<gz, kBox3Block, smem_z, ctx->stream>>>(P0, P1, P2, live, T, fac, fac_stride, v);
      box3_plane_kernel<true><<<gp, kBox3Block, smem_p, ctx->stream>>>(d_boxes, live, rn, T, nullptr, v, d_u);
      PDD_CUDA_TRY(ctx, cudaGetLastError());
    }
    std::vector<char> h_state(L.state_bytes);
    PDD_CUDA_TRY(ctx, cudaMemcpyAsync(h_state.data(), base, L.state_bytes, cudaMemcpyDeviceToHost, ctx->stream));
    PDD_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    std::memcpy(h_it.data(), h_state.data() + L.it, NB * sizeof(int64_t));
    std::memcpy(h_res.data(), h_state.data() + L.res, NB * sizeof(double));
  }
  if (ev.second) PDD_CUDA_TRY(ctx, cudaEventRecord(ev.second, ctx->stream));
  PDD_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
  int64_t it_max = 0;
  double res_max = 0.0;
  bool unmet = false;
  for (size_t b = 0; b < NB; ++b) {
    it_max = std::max(it_max, h_it[b]);
    res_max = std::max(res_max, h_res[b]);
    unmet |= jacobi ? h_res[b] >= tol : h_res[b] > tol;
    if (iters_each) iters_each[b] = h_it[b];
    if (resid_each) resid_each[b] = h_res[b];
  }
  if (iters) *iters = it_max;
  if (resid) *resid = res_max;
  if (unmet) return fail(ctx, PDD_ETIMEOUT, "max_iter reached before the tolerance");
  return PDD_OK;
}

// A batch of nb boxes with the same grid size and method: the faces of box b
// follow those of box b - 1 in d_face, and d_u is [nb][n2][n1][n0].  *iters
// and *resid (if non-null) get the largest count and relative residual over
// the boxes; iters_each / resid_each (host, nb entries, may be null) get each
// box's own.
pdd_status subdomain_solve3d_batch_impl(pdd_ctx *ctx, const pdd_subdomain *sds, int32_t nb,
                                        const double *d_face, int64_t m, double *d_u,
                                        int64_t *iters, double *resid, int64_t *iters_each,
                                        double *resid_each) {
  if (!sds || nb < 1 || nb > 65535) return fail(ctx, PDD_EINVAL, "batch of 1 .. 65535 boxes");
  if (ctx->prob.kind != PDD_PROB_ELLIPTIC_MANUFACTURED || ctx->prob.dim != 3)
    return fail(ctx, PDD_EINVAL, "the 3-D subdomain solver covers the 3-D family");
  if (reflect_mask(ctx) != 0)
    return fail(ctx, PDD_EINVAL, "the 3-D subdomain solver takes Dirichlet data only");
  const pdd_subdomain &S0 = sds[0];
  std::vector<Box3> boxes(static_cast<size_t>(nb));
  int64_t off = 0;
  for (int32_t b = 0; b < nb; ++b) {
    const pdd_subdomain *sd = sds + b;
    Box3 &B = boxes[static_cast<size_t>(b)];
    for (int a = 0; a < 3; ++a) {
      if (sd->n[a] < 3 || sd->n[a] - 2 > kBox3MaxInterior)
        return fail(ctx, PDD_EINVAL, "3-D grids take 3 .. %d points per axis", kBox3MaxInterior + 2);
      if (sd->n[a] != S0.n[a])
        return fail(ctx, PDD_EINVAL, "the boxes of a batch share one grid size");
      if (!(sd->hi[a] > sd->lo[a]) || sd->lo[a] < 0.0 || sd->hi[a] > 1.0)
        return fail(ctx, PDD_EINVAL, "box must be non-empty and inside the unit cube");
      B.lo[a] = sd->lo[a];
      B.n[a] = sd->n[a];
      B.P[a] = sd->n[a] - 2;
      B.h[a] = (sd->hi[a] - sd->lo[a]) / (sd->n[a] - 1);
    }
    if (sd->iface_axis < 0 || sd->iface_axis > 63 || sd->iface_side != 0)
      return fail(ctx, PDD_EINVAL, "3-D: iface_axis is a mask of interface faces (0..63), "
                                   "iface_side must be 0");
    if (sd->method != PDD_STENCIL_DST && sd->method != PDD_STENCIL_JACOBI)
      return fail(ctx, PDD_EINVAL, "3-D methods: PDD_STENCIL_DST or PDD_STENCIL_JACOBI");
    if (sd->method != S0.method || sd->max_iter != S0.max_iter || !(sd->tol == S0.tol))
      return fail(ctx, PDD_EINVAL, "the boxes of a batch share one method and stopping rule");
    if (sd->max_iter < 1 || !(sd->tol >= 0.0)) return fail(ctx, PDD_EINVAL, "bad stopping rule");
    B.mask = sd->iface_axis;
    for (int fc = 0; fc < 6; ++fc) {
      B.face_off[fc] = off;
      if ((B.mask >> fc) & 1) {
        const int a = fc >> 1;
        B.face_ld[fc] = B.n[a == 0 ? 1 : 0];
        off += static_cast<int64_t>(B.face_ld[fc]) * B.n[a == 2 ? 1 : 2];
      }
    }
    B.u_sy = B.n[0];
    B.u_sz = static_cast<int64_t>(B.n[0]) * B.n[1];
    B.u_off = b * B.u_sz * B.n[2];
  }
  if (m != off) return fail(ctx, PDD_EINVAL, "expected %lld face values, got %lld",
                            static_cast<long long>(off), static_cast<long long>(m));
  if (off > 0 && !d_face) return fail(ctx, PDD_EINVAL, "null face data");
  if (!d_u) return fail(ctx, PDD_EINVAL, "null output");
  PDD_CUDA_TRY(ctx, cudaSetDevice(ctx->device));

  return solve_boxes(ctx, boxes, S0.method, S0.max_iter, S0.tol, d_face, d_u,
                     nb * boxes[0].u_sz * boxes[0].n[2], iters, resid, iters_each, resid_each);
}

pdd_status subdomain_solve3d_impl(pdd_ctx *ctx, const pdd_subdomain *sd, const double *d_face,
                                  int64_t m, double *d_u, int64_t *iters, double *resid) {
  return subdomain_solve3d_batch_impl(ctx, sd, 1, d_face, m, d_u, iters, resid, nullptr, nullptr);
}

// ---------------------------------------------------------------------------
// Stage two on the split cube (pdd_elliptic3d_stage2): nodes sorted to their
// planes, the planes' interpolants on their grids, and the boxes solved in
// place in the global grid, their faces read from the plane grids (no packing
// and no scatter of the solution).
// ---------------------------------------------------------------------------
constexpr int kPickBlock = 1024;

// Nodes of plane blockIdx.x (axis a = p / (split - 1), x_a = (p mod (split -
// 1) + 1) / split; with axis, only the nodes that name a) and their values,
// in node order, at most cap of them; count[p] is how many there are.
__global__ void __launch_bounds__(kPickBlock)
stage2_pick_kernel(const double *nodes, const double *values, const int32_t *axis, int64_t n,
                   int split, int64_t cap, double *pn, double *pv, int64_t *count) {
  const int a = blockIdx.x / (split - 1);
  const double pos = static_cast<double>(blockIdx.x % (split - 1) + 1) / split;
  pn += blockIdx.x * cap * 3;
  pv += blockIdx.x * cap;
  __shared__ int warp_sum[kPickBlock / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t base = 0;
  for (int64_t i0 = 0; i0 < n; i0 += kPickBlock) {
    const int64_t i = i0 + threadIdx.x;
    const bool on = i < n && nodes[3 * i + a] == pos && (!axis || axis[i] == a);
    const unsigned m = __ballot_sync(kFull, on);
    if (lane == 0) warp_sum[warp] = __popc(m);
    __syncthreads();
    int before = 0, all = 0;
    for (int w = 0; w < kPickBlock / 32; ++w) {
      before += w < warp ? warp_sum[w] : 0;
      all += warp_sum[w];
    }
    const int64_t e = base + before + __popc(m & ((1u << lane) - 1u));
    if (on && e < cap) {
      for (int d = 0; d < 3; ++d) pn[3 * e + d] = nodes[3 * i + d];
      pv[e] = values[i];
    }
    base += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) count[blockIdx.x] = base;
}

// The grid points of every plane ([slow = higher axis][fast = lower axis]).
__global__ void stage2_grid_kernel(int split, int grid, double *q) {
  const int p = blockIdx.y, a = p / (split - 1);
  const int a1 = a == 0 ? 1 : 0, a2 = a == 2 ? 1 : 2;
  q += 3 * static_cast<int64_t>(p) * grid * grid;
  const double step = 1.0 / (grid - 1);
  // (from both ends, so that the last point is 1 exactly)
  auto t = [&](int i) { return i < grid / 2 ? i * step : 1.0 - (grid - 1 - i) * step; };
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < grid * grid; e += gridDim.x * blockDim.x) {
    const int j = e / grid, i = e - j * grid;
    q[3 * static_cast<int64_t>(e) + a] = static_cast<double>(p % (split - 1) + 1) / split;
    q[3 * static_cast<int64_t>(e) + a1] = t(i);
    q[3 * static_cast<int64_t>(e) + a2] = t(j);
  }
}

pdd_status elliptic3d_stage2_impl(pdd_ctx *ctx, const double *d_nodes, const double *d_values,
                                  const int32_t *d_axis, int64_t n, const pdd_stage2_params *sp,
                                  double *d_planes, double *d_u, int64_t *iters, double *resid) {
  if (!sp || !d_planes || !d_u) return fail(ctx, PDD_EINVAL, "null argument");
  if (ctx->prob.kind != PDD_PROB_ELLIPTIC_MANUFACTURED || ctx->prob.dim != 3)
    return fail(ctx, PDD_EINVAL, "the 3-D stage two covers the 3-D family");
  if (reflect_mask(ctx) != 0)
    return fail(ctx, PDD_EINVAL, "the 3-D subdomain solver takes Dirichlet data only");
  const int split = sp->split, grid = sp->grid;
  if (split < 2 || split > 22) return fail(ctx, PDD_EINVAL, "split must be in [2, 22]");
  if (grid < 3 || (grid - 1) % split) return fail(ctx, PDD_EINVAL, "grid - 1 must be a multiple of split");
  const int m = (grid - 1) / split + 1;
  if (m < 3 || m - 2 > kBox3MaxInterior)
    return fail(ctx, PDD_EINVAL, "3-D grids take 3 .. %d points per axis", kBox3MaxInterior + 2);
  if (sp->method != PDD_STENCIL_DST && sp->method != PDD_STENCIL_JACOBI)
    return fail(ctx, PDD_EINVAL, "3-D methods: PDD_STENCIL_DST or PDD_STENCIL_JACOBI");
  if (sp->max_iter < 1 || !(sp->tol >= 0.0)) return fail(ctx, PDD_EINVAL, "bad stopping rule");
  if (n < 0 || (n > 0 && (!d_nodes || !d_values))) return fail(ctx, PDD_EINVAL, "null buffer");
  PDD_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  const int np = 3 * (split - 1);
  const int64_t g2 = static_cast<int64_t>(grid) * grid;
  // (a plane with more nodes than any system may hold is refused below)
  const int64_t cap = std::min<int64_t>(n, 8192);
  const size_t off_cnt = 0, off_n = 512;
  const size_t off_v = align_up(off_n + static_cast<size_t>(np) * cap * 3 * sizeof(double), 256);
  const size_t off_q = align_up(off_v + static_cast<size_t>(np) * cap * sizeof(double), 256);
  // the auxiliary buffer: the interpolation and the boxes use the scratch
  pdd_status st = ensure_aux(ctx, off_q + static_cast<size_t>(np) * g2 * 3 * sizeof(double));
  if (st != PDD_OK) return st;
  char *base = static_cast<char *>(ctx->aux);
  auto *cnt = reinterpret_cast<int64_t *>(base + off_cnt);
  auto *pn = reinterpret_cast<double *>(base + off_n);
  auto *pv = reinterpret_cast<double *>(base + off_v);
  auto *q = reinterpret_cast<double *>(base + off_q);
  stage2_pick_kernel<<<np, kPickBlock, 0, ctx->stream>>>(d_nodes, d_values, d_axis, n, split, cap,
                                                         pn, pv, cnt);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  stage2_grid_kernel<<<dim3(static_cast<unsigned>(std::min<int64_t>((g2 + 255) / 256, 1024)),
                            static_cast<unsigned>(np)), 256, 0, ctx->stream>>>(split, grid, q);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  int64_t h_cnt[64], h_off[64], h_q[64];
  int32_t h_axis[64];
  double h_pos[64];
  PDD_CUDA_TRY(ctx, cudaMemcpyAsync(h_cnt, cnt, np * sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
  PDD_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
  for (int p = 0; p < np; ++p) {
    h_axis[p] = p / (split - 1);
    h_pos[p] = static_cast<double>(p % (split - 1) + 1) / split;
    h_off[p] = p * cap;
    h_q[p] = g2;
  }
  std::vector<Box3> boxes;
  for (int kz = 0; kz < split; ++kz)
    for (int ky = 0; ky < split; ++ky)
      for (int kx = 0; kx < split; ++kx) {
        const int kk[3] = {kx, ky, kz};
        Box3 B;
        std::memset(&B, 0, sizeof B);
        for (int a = 0; a < 3; ++a) {
          B.lo[a] = static_cast<double>(kk[a]) / split;
          B.n[a] = m;
          B.P[a] = m - 2;
          B.h[a] = (static_cast<double>(kk[a] + 1) / split - B.lo[a]) / (m - 1);
        }
        for (int fc = 0; fc < 6; ++fc) {
          const int a = fc >> 1, plane = kk[a] + (fc & 1);
          if (plane == 0 || plane == split) continue;
          const int a1 = a == 0 ? 1 : 0, a2 = a == 2 ? 1 : 2;
          B.mask |= 1 << fc;
          if (fc & 1) B.next |= 1 << fc;
          B.face_ld[fc] = grid;
          B.face_off[fc] = (a * (split - 1) + plane - 1) * g2 +
                           static_cast<int64_t>(kk[a2] * (m - 1)) * grid + kk[a1] * (m - 1);
        }
        B.u_sy = grid;
        B.u_sz = g2;
        B.u_off = (kz * g2 + static_cast<int64_t>(ky) * grid + kx) * (m - 1);
        boxes.push_back(B);
      }
  // (scratch for the larger of the two parts at once)
  st = ensure_scratch(ctx, box3_layout(boxes, sp->method == PDD_STENCIL_JACOBI, g2 * grid).total);
  if (st != PDD_OK) return st;
  st = interface_interp_impl(ctx, np, h_axis, h_pos, h_cnt, pn, pv, sp->n_bnd, h_q, q, d_planes, h_off);
  if (st != PDD_OK) return st;
  return solve_boxes(ctx, boxes, sp->method, sp->max_iter, sp->tol, d_planes, d_u, g2 * grid, iters,
                     resid, nullptr, nullptr);
}

}  // namespace pdd
