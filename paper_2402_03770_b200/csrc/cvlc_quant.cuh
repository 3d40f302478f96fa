// The two stochastic quantizers of the encoder (device code shared by the packet and the unframed writers).
#pragma once

#include "cvlc_common.cuh"

namespace cvlc {

#ifdef __CUDACC__

// Stochastic rounding of t = num * scale onto the integers 0 .. L in fp32, word = the coordinate's random word: false where fp32
// cannot tell floor(t) or [u < frac(t)], u = word / 2^32.  t is good to 3 * 2^-24 of itself (num, scale and the product each
// rounded once), u to 2^-23 (its low bits dropped), so both decisions are certain when the fraction is farther than
// 2^-22 (t + 1) from 0, 1 and u.  Meant for L < 2^12: one warp in sixteen then has a lane that needs the binary64 form below,
// whose conversions run at an eighth of the fp32 rate.  Packing kernel, 100 ResNet-18-sized clients: 528 -> 442 us together
// with its loop freed of branches.
constexpr uint32_t kFastRoundBits = 12;
__device__ __forceinline__ bool fast_round(float num, float scale, float L, uint32_t word, uint32_t& code) {
  const float t = __fmul_rn(num, scale);
  const float s = __fadd_rn(t, 12582912.0f);  // 1.5 * 2^23: the nearest integer in the low mantissa bits
  float f = __fsub_rn(t, __fsub_rn(s, 12582912.0f));
  int j = __float_as_int(s) - 0x4B400000;
  if (f < 0.0f) {
    f = __fadd_rn(f, 1.0f);
    j -= 1;
  }
  const float u = __fsub_rn(__uint_as_float(0x3F800000u | (word >> 9)), 1.0f);
  const float eps = fmaf(t, 0x1p-22f, 0x1p-22f);
  code = (uint32_t)j + (u < f ? 1u : 0u);
  return f > eps && f < 1.0f - eps && fabsf(f - u) > eps && t < L;
}
// the scale in fp32, or 0 (never certain) for long codes and where it is no normal number
__device__ __forceinline__ float fast_scale(double scale, uint32_t bits) {
  return (bits <= kFastRoundBits && scale > 0x1p-100 && scale < 0x1p100) ? (float)scale : 0.0f;
}
__device__ __forceinline__ double unit_of(uint32_t word) { return __dmul_rn((double)word, 1.0 / 4294967296.0); }

// PQ: stochastic rounding of num = x - lo onto the 2^y uniform centroids of [lo, hi]; den = hi - lo > 0, Lc = 2^y - 1,
// scale = Lc / den, u = the coordinate's random word / 2^32.  t = (num / den) * Lc decides floor(t) and [u < frac(t)].
// num * scale is within a few ulp of it; unless its fraction sits that close to 0, 1 or u, both decisions are the same
// and the division is not needed.
__device__ __forceinline__ uint32_t pq_quantize(double num, double den, double Lc, double scale, double u) {
  const double tf = __dmul_rn(num, scale);
  const double jf = floor(tf);
  const double ff = __dsub_rn(tf, jf);
  const double eps = __dmul_rn(tf, 0x1p-48) + 0x1p-1000;
  if (ff > eps && ff < 1.0 - eps && fabs(ff - u) > eps && jf < Lc) return __double2uint_rz(jf) + ((u < ff) ? 1u : 0u);
  const double t = __dmul_rn(__ddiv_rn(num, den), Lc);
  double j0 = floor(t);
  if (j0 > Lc) j0 = Lc;
  const double frac = __dsub_rn(t, j0);
  return __double2uint_rz(j0) + ((u < frac) ? 1u : 0u);
}

// QSGD: level of a = |x| against the packet's norm dn > 0 on a grid of sq = sqd steps; scale = sqd / dn
__device__ __forceinline__ uint32_t qsgd_quantize_level(double a, double dn, double sqd, uint32_t sq, double scale, double u) {
  const double tf = __dmul_rn(a, scale);
  const double jf = floor(tf);
  const double ff = __dsub_rn(tf, jf);
  const double eps = __dmul_rn(tf, 0x1p-48) + 0x1p-1000;
  if (ff > eps && ff < 1.0 - eps && fabs(ff - u) > eps && jf < sqd) return __double2uint_rz(jf) + ((u < ff) ? 1u : 0u);
  const double t = __dmul_rn(__ddiv_rn(a, dn), sqd);
  double j0 = floor(t);
  if (j0 > sqd) j0 = sqd;
  const double frac = __dsub_rn(t, j0);
  uint32_t level = __double2uint_rz(j0) + ((u < frac) ? 1u : 0u);
  if (level > sq) level = sq;
  return level;
}

// the binary64 forms out of line, for the few records that need them
static __device__ __noinline__ uint32_t pq_quantize_slow(float v, float lo, float hi, uint32_t y, uint32_t word) {
  const double Lc = (double)((1ull << y) - 1ull), den = __dsub_rn((double)hi, (double)lo);
  const double x = v == 0.0f ? 0.0 : (double)v;  // -0 is stored as +0
  return pq_quantize(__dsub_rn(x, (double)lo), den, Lc, __ddiv_rn(Lc, den), unit_of(word));
}
static __device__ __noinline__ uint32_t qsgd_quantize_slow(float a, float norm, uint32_t sq, uint32_t word) {
  return qsgd_quantize_level((double)a, (double)norm, (double)sq, sq, __ddiv_rn((double)sq, (double)norm), unit_of(word));
}

// the l2-norm of P values whose exact squares sit in sqv, added in the given order in double, rounded to fp32
// (FLT_MAX beyond the fp32 range); one thread walks the chain: the order is part of the stream's definition
__device__ __forceinline__ float qsgd_norm_of_squares(const double* sqv, uint32_t P) {
  double sum = 0.0;
  uint32_t j = 0;
  for (; j + 8 <= P; j += 8) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = sqv[j + u];
#pragma unroll
    for (int u = 0; u < 8; ++u) sum = __dadd_rn(sum, v[u]);
  }
  for (; j < P; ++j) sum = __dadd_rn(sum, sqv[j]);
  const double rt = __dsqrt_rn(sum);
  return (rt > 3.4028234663852886e38) ? 3.4028234663852886e38f : __double2float_rn(rt);
}

#endif  // __CUDACC__

}  // namespace cvlc
