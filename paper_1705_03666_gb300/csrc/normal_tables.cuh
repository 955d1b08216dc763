// normal_tables.cuh -- binary64 Box-Muller normals of 23-bit uniforms from
// tables, for the FP64 path kernel.
//
// FP64 is a 1/64-rate pipe here (64 clocks per warp instruction and
// scheduler), and the library's log, sqrt and sincospi took about 90 of the
// 130 FP64 instructions of a 2-D step.  The uniforms are odd multiples of
// 2^-24, so both maps split exactly into a table's part and a small remainder:
//
// * angle 2 pi U, k = 23 bits of the word: k = 2048 h + l with -1024 <= l < 1024,
//   and (cos, sin) of 2 pi h / 4096 rotated by (cos - 1, sin) of 2 pi (2 l + 1) /
//   2^24, the small correction added last (6 FP64 instructions).  h is the
//   nearest, so that beside a zero of the cosine or sine the table's value is an
//   exact zero and the correction is the result: a difference of two entries
//   (l from 0 to 2047) was off by up to 700 units in the last place there;
// * -2 ln U: U = 2^e m with m in [3/4, 3/2), c the nearest multiple of
//   2^-10 (2^-11 below 1), d = m - c exact, x = d / c (|x| <= 2^-11), ln U =
//   e ln 2 + ln c + x - x^2/2 + x^3/3 - x^4/4 + x^5/5 (the next term is below
//   2^-57 x).  Near U = 1, c = 1 and e = 0, so the relative accuracy holds
//   there (9 instructions);
// * the square root by two Heron corrections of a 20-bit binary32 seed (4).
//
// Over all 2^23 codes of either uniform a normal is within 2.7 units in the last
// place.  The tables (115 KB, read through L1) are formed by a small kernel in the
// call's own scratch.
#pragma once

#include "common.cuh"

namespace pdd {

constexpr int kAngleHi = 4096, kAngleLo = 2048, kLogIdx = 1025, kLogExp = 32;
constexpr int kNormalEntries = kAngleHi + kAngleLo + kLogIdx + kLogExp;
constexpr size_t kNormalBytes = kNormalEntries * sizeof(double2);

struct NormalTables {
  const double2 *hi, *lo;  // (cos, sin) by h; (cos - 1, sin) by l + 1024
  const double2 *lg;       // (1 / c, ln c)
  const double2 *ex;       // (-i ln 2, 0)
  __device__ __forceinline__ explicit NormalTables(const double2 *t)
      : hi(t), lo(t + kAngleHi), lg(lo + kAngleLo), ex(lg + kLogIdx) {}
};

static __global__ void normal_tables_kernel(double2 *t) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kNormalEntries) return;
  double2 *o = t + i;
  if (i < kAngleHi) {
    double s, c;
    sincospi(2.0 * i / kAngleHi, &s, &c);
    *o = make_double2(c, s);
    return;
  }
  i -= kAngleHi;
  if (i < kAngleLo) {
    const double half = (2 * (i - kAngleLo / 2) + 1) * 0x1p-24;  // angle / (2 pi)
    const double h = sinpi(half);
    *o = make_double2(-2.0 * h * h, sinpi(2.0 * half));
    return;
  }
  i -= kAngleLo;
  if (i < kLogIdx) {
    const double c = (1.0 + i * 0x1p-10) * (i >= 512 ? 0.5 : 1.0);
    *o = make_double2(1.0 / c, log(c));
    return;
  }
  i -= kLogIdx;
  *o = make_double2(-i * 0.6931471805599453094, 0.0);
}
inline void launch_normal_tables(double2 *t, cudaStream_t s) {
  normal_tables_kernel<<<(kNormalEntries + 63) / 64, 64, 0, s>>>(t);
}

__device__ __forceinline__ void box_muller_tables(const NormalTables &t, uint32_t a, uint32_t b,
                                                  double &z0, double &z1) {
  // -2 ln U
  const uint32_t bits = __float_as_uint(unif_f(a));
  const uint32_t mant = bits & 0x7fffffu;
  const uint32_t idx = (mant + 4096u) >> 13;
  const uint32_t up = idx >= 512u ? 1u : 0u;        // m = mantissa / 2
  const uint32_t e = 127u - (bits >> 23) - up;      // U = 2^-e m
  const uint32_t one = 0x3ff00000u - (up << 20);
  const double m = __hiloint2double(one | (mant >> 3), mant << 29);
  const double c = __hiloint2double(one + (idx << 10), 0);
  const double2 lc = __ldg(t.lg + idx);
  const double base = __ldg(&t.ex[e].x) + lc.y;
  const double x = (m - c) * lc.x;
  double p = fma(x, 0.2, -0.25);
  p = fma(p, x, 1.0 / 3.0);
  p = fma(p, x, -0.5);
  const double w = -2.0 * (base + fma(x * x, p, x));
  // its square root (w in [1e-7, 34])
  const float f = __int_as_float((__double2hiint(w) - (896 << 20)) << 3);
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const double s0 = __hiloint2double((__float_as_int(f * y) >> 3) + (896 << 20), 0);
  const double h = __hiloint2double((__float_as_int(0.5f * y) >> 3) + (896 << 20), 0);
  const double s1 = fma(fma(-s0, s0, w), h, s0);
  const double r = fma(fma(-s1, s1, w), h, s1);
  // cos and sin of 2 pi U_b
  const uint32_t k = (b >> 9) + kAngleLo / 2;
  const double2 A = __ldg(t.hi + ((k >> 11) & (kAngleHi - 1))), B = __ldg(t.lo + (k & (kAngleLo - 1)));
  const double cs = A.x + fma(A.x, B.x, -(A.y * B.y));
  const double sn = A.y + fma(A.y, B.x, A.x * B.y);
  z0 = r * cs;
  z1 = r * sn;
}

}  // namespace pdd
