// dst.cu -- direct subdomain solve of stage two (Sec. 2.1) by discrete sine
// transforms.  On a rectangle with Dirichlet data the 5-point operator
//   A U = (2/hx^2 + 2/hy^2) U - (U_W + U_E)/hx^2 - (U_S + U_N)/hy^2
// over the P x Q interior points (P = nx - 2, Q = ny - 2) is diagonal in the
// DST-I basis: with S_P[i][k] = sin(pi (i+1)(k+1) / (P+1)) (symmetric,
// S_P^2 = (P+1)/2 I) and the eigenvalues
//   lambda_k = 4/hx^2 sin^2(pi (k+1) / (2 (P+1))),
//   nu_l     = 4/hy^2 sin^2(pi (l+1) / (2 (Q+1))),
// the solution of A U = F (F: the boundary values moved to the right) is
//   U = 4 / ((P+1)(Q+1)) S_Q [(S_Q F S_P) ./ (nu_l + lambda_k)] S_P,
// the same discrete solution the iterative methods converge to, here to
// rounding.  Four dense FP64 products of the sine matrices (O(PQ(P+Q))
// flops) replace the iterations.
#include <algorithm>
#include <cmath>

#include "ctx.hpp"

namespace pdd {

constexpr int kDstTile = 8, kDstK = 32;
constexpr int kDstResBlocks = 64;

// The Dirichlet values next to interior point (i+1, j+1), weighted by 1/h^2.
__device__ __forceinline__ double dst_rhs(const double *u, int nx, int ny, int i, int j, double ihx2,
                                          double ihy2) {
  const int64_t row = static_cast<int64_t>(j + 1) * nx;
  double f = 0.0;
  if (i == 0) f += u[row] * ihx2;
  if (i == nx - 3) f += u[row + nx - 1] * ihx2;
  if (j == 0) f += u[i + 1] * ihy2;
  if (j == ny - 3) f += u[static_cast<int64_t>(ny - 1) * nx + i + 1] * ihy2;
  return f;
}

// S[i][k] = sin(pi (i+1)(k+1) / (n+1)), i, k < n: the product is reduced
// modulo 2(n+1) in integers, so sinpi sees an exact argument in [0, 2).
__device__ __forceinline__ double dst_sine(int64_t t, int n) {
  const uint32_t i = static_cast<uint32_t>(t) / n, k = static_cast<uint32_t>(t) - i * n;  // n <= 8192
  const uint32_t r = ((i + 1) * (k + 1)) % (2u * (n + 1));
  return sinpi(static_cast<double>(r) / static_cast<double>(n + 1));
}
// What a solve starts from, in one launch: the sine matrices SP and SQ (one
// when they are the same), the eigenvalues lam (P along x, then Q along y), the
// right-hand side F[j][i] (j < Q rows along y, i < P columns along x) and a zero
// counter of the residual's blocks.
__global__ void dst_setup_kernel(const double *u, int nx, int ny, double ihx2, double ihy2, double *SP,
                                 double *SQ, double *lam, double *F, unsigned *done) {
  const int P = nx - 2, Q = ny - 2;
  const int64_t pp = static_cast<int64_t>(P) * P, qq = SQ == SP ? 0 : static_cast<int64_t>(Q) * Q,
                pq = static_cast<int64_t>(P) * Q, total = pp + qq + P + Q + pq;
  if (blockIdx.x == 0 && threadIdx.x == 0) *done = 0;
  for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < total;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    int64_t q = t;
    if (q < pp) {
      SP[q] = dst_sine(q, P);
    } else if ((q -= pp) < qq) {
      SQ[q] = dst_sine(q, Q);
    } else if ((q -= qq) < P + Q) {
      const int n = q < P ? P : Q, k = static_cast<int>(q < P ? q : q - P);
      const double sn = sinpi(static_cast<double>(k + 1) / (2.0 * (n + 1)));
      lam[q] = 4.0 * (q < P ? ihx2 : ihy2) * sn * sn;
    } else {
      q -= P + Q;
      const int j = static_cast<int>(q / P), i = static_cast<int>(q - static_cast<int64_t>(j) * P);
      F[q] = dst_rhs(u, nx, ny, i, j, ihx2, ihy2);
    }
  }
}

// C[M][N] = A[M][K] B[K][N], FP64, row-major, one output per thread, and with
// it what follows the product: kDivide: C[l][k] *= scale / (lam_k + nu_l) (lam:
// N along x, then M along y); kScatter: into the interior of the grid u of rows
// of N + 2 instead of C.  Bound by the FP64 rate, which is per SM: 8 x 8 outputs
// a block spread a 127 x 127 product over the chip (256 blocks; 16 x 16 on 64 SMs
// took 15.8 us, 8.7 us now), the next 32 of K loaded while these are multiplied.
enum DstEpilogue { kPlain, kDivide, kScatter };
template <DstEpilogue kEp>
__global__ void __launch_bounds__(kDstTile * kDstTile)
dst_gemm_kernel(const double *A, const double *B, double *C, int M, int N, int K, const double *lam,
                double scale) {
  __shared__ double As[kDstTile][kDstK + 1];
  __shared__ double Bs[kDstK][kDstTile + 1];
  constexpr int kLoads = kDstK / kDstTile, kT = kDstTile * kDstTile;
  const int t = threadIdx.x, tx = t % kDstTile, ty = t / kDstTile;
  const int row0 = blockIdx.y * kDstTile, col0 = blockIdx.x * kDstTile;
  double a[kLoads], b[kLoads];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      const int ia = t + kT * q, ra = row0 + ia / kDstK, ka = k0 + ia % kDstK;
      a[q] = ra < M && ka < K ? A[static_cast<int64_t>(ra) * K + ka] : 0.0;
      const int kb = k0 + ia / kDstTile, cb = col0 + ia % kDstTile;
      b[q] = kb < K && cb < N ? B[static_cast<int64_t>(kb) * N + cb] : 0.0;
    }
  };
  double acc = 0.0;
  load(0);
  for (int k0 = 0; k0 < K; k0 += kDstK) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      const int ia = t + kT * q;
      As[ia / kDstK][ia % kDstK] = a[q];
      Bs[ia / kDstTile][ia % kDstTile] = b[q];
    }
    __syncthreads();
    if (k0 + kDstK < K) load(k0 + kDstK);
#pragma unroll 8
    for (int kk = 0; kk < kDstK; ++kk) acc = fma(As[ty][kk], Bs[kk][tx], acc);
  }
  const int row = row0 + ty, col = col0 + tx;
  if (row >= M || col >= N) return;
  if constexpr (kEp == kDivide) acc *= scale / (lam[col] + lam[N + row]);
  if constexpr (kEp == kScatter) C[static_cast<int64_t>(row + 1) * (N + 2) + col + 1] = acc;
  else C[static_cast<int64_t>(row) * N + col] = acc;
}

// ||F - A U||_2 / ||F||_2 over the interior (0 when F = 0; F from the boundary),
// in a fixed order: each block sums a fixed slice of points (part[2 b], part[2 b
// + 1]), and the last block to finish adds the partials in a fixed tree;
// *it = 0 (a direct solve).
__global__ void __launch_bounds__(256)
dst_residual_kernel(const double *u, int nx, int ny, double ihx2, double ihy2, double *part,
                    unsigned *done, int64_t *it, double *res) {
  __shared__ double sr[256], sb[256];
  __shared__ bool last;
  const int P = nx - 2, Q = ny - 2;
  const int64_t total = static_cast<int64_t>(P) * Q;
  const double diag = 2.0 * ihx2 + 2.0 * ihy2;
  double r2 = 0.0, b2 = 0.0;
  for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < total;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int j = static_cast<int>(t / P), i = static_cast<int>(t - static_cast<int64_t>(j) * P);
    const int64_t c = static_cast<int64_t>(j + 1) * nx + i + 1;
    // interior neighbours only: the boundary ones are in F
    const double w = i > 0 ? u[c - 1] : 0.0, e = i < P - 1 ? u[c + 1] : 0.0;
    const double s = j > 0 ? u[c - nx] : 0.0, n = j < Q - 1 ? u[c + nx] : 0.0;
    const double Au = diag * u[c] - ihx2 * (w + e) - ihy2 * (s + n);
    const double f = dst_rhs(u, nx, ny, i, j, ihx2, ihy2), r = f - Au;
    r2 += r * r;
    b2 += f * f;
  }
  auto block_totals = [&]() {
    sr[threadIdx.x] = r2;
    sb[threadIdx.x] = b2;
    __syncthreads();
    for (int m = 128; m > 0; m >>= 1) {
      if (static_cast<int>(threadIdx.x) < m) {
        sr[threadIdx.x] += sr[threadIdx.x + m];
        sb[threadIdx.x] += sb[threadIdx.x + m];
      }
      __syncthreads();
    }
  };
  block_totals();
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = sr[0];
    part[2 * blockIdx.x + 1] = sb[0];
    __threadfence();
    last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const volatile double *const v = part;
  const bool has = threadIdx.x < gridDim.x;
  r2 = has ? v[2 * threadIdx.x] : 0.0;
  b2 = has ? v[2 * threadIdx.x + 1] : 0.0;
  __syncthreads();
  block_totals();
  if (threadIdx.x == 0) {
    *it = 0;
    *res = sb[0] > 0.0 ? sqrt(sr[0] / sb[0]) : sqrt(sr[0]);
  }
}

static unsigned dst_grid(int64_t work) {
  return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, 4096)));
}

template <DstEpilogue kEp>
static void dst_gemm(cudaStream_t st, const double *A, const double *B, double *C, int M, int N, int K,
                     const double *lam = nullptr, double scale = 0.0) {
  const dim3 grid((N + kDstTile - 1) / kDstTile, (M + kDstTile - 1) / kDstTile);
  dst_gemm_kernel<kEp><<<grid, kDstTile * kDstTile, 0, st>>>(A, B, C, M, N, K, lam, scale);
}

size_t dst_scratch_bytes(int nx, int ny) {
  const size_t P = static_cast<size_t>(nx - 2), Q = static_cast<size_t>(ny - 2);
  return align_up(P * P * sizeof(double), 256) + align_up(Q * Q * sizeof(double), 256) +
         2 * align_up(P * Q * sizeof(double), 256) + 2 * kDstResBlocks * sizeof(double) + 256 +
         (P + Q) * sizeof(double);
}

// d_u holds the Dirichlet data on the boundary (interior ignored); on return
// the interior holds the solution.  work: dst_scratch_bytes(nx, ny) bytes.
pdd_status dst_solve(pdd_ctx *ctx, double *d_u, int nx, int ny, double hx, double hy, char *work,
                     int64_t *it_d, double *res_d) {
  const int P = nx - 2, Q = ny - 2;
  const double ihx2 = 1.0 / (hx * hx), ihy2 = 1.0 / (hy * hy);
  double *SP = reinterpret_cast<double *>(work);
  double *SQ = reinterpret_cast<double *>(work + align_up(static_cast<size_t>(P) * P * sizeof(double), 256));
  double *F = reinterpret_cast<double *>(reinterpret_cast<char *>(SQ) +
                                         align_up(static_cast<size_t>(Q) * Q * sizeof(double), 256));
  double *T = reinterpret_cast<double *>(reinterpret_cast<char *>(F) +
                                         align_up(static_cast<size_t>(P) * Q * sizeof(double), 256));
  double *part = reinterpret_cast<double *>(reinterpret_cast<char *>(T) +
                                            align_up(static_cast<size_t>(P) * Q * sizeof(double), 256));
  auto *done = reinterpret_cast<unsigned *>(part + 2 * kDstResBlocks);
  double *lam = reinterpret_cast<double *>(reinterpret_cast<char *>(done) + 256);
  if (P == Q) SQ = SP;
  cudaStream_t st = ctx->stream;
  const int64_t work_items = static_cast<int64_t>(P) * P + static_cast<int64_t>(Q) * (P + Q);
  dst_setup_kernel<<<dst_grid(work_items), 256, 0, st>>>(d_u, nx, ny, ihx2, ihy2, SP, SQ, lam, F, done);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  dst_gemm<kPlain>(st, F, SP, T, Q, P, P);    // T  = F S_P
  dst_gemm<kDivide>(st, SQ, T, F, Q, P, Q, lam,
                    4.0 / (static_cast<double>(P + 1) * static_cast<double>(Q + 1)));  // Uh
  dst_gemm<kPlain>(st, F, SP, T, Q, P, P);    // T  = Uh S_P
  dst_gemm<kScatter>(st, SQ, T, d_u, Q, P, Q);  // U  = S_Q T
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  dst_residual_kernel<<<kDstResBlocks, 256, 0, st>>>(d_u, nx, ny, ihx2, ihy2, part, done, it_d, res_d);
  PDD_CUDA_TRY(ctx, cudaGetLastError());
  return PDD_OK;
}

}  // namespace pdd
