// inv_fx.cuh -- 1/|d| in FP64 accuracy from integer coordinate differences.
//
// The FP64 pipe of this GPU issues 2 FMAs per clock and SM, the integer and
// FP32 pipes 64 to 128: the 20 FP64 operations of a distance and its
// reciprocal square root cost as much as about 1000 integer ones.  Here
// coordinates are 64-bit fixed-point numbers (differences are exact), |d|^2 is
// formed in 126 bits, its leading 64 bits m 2^62, 1 <= m < 4, feed one third-order
// step from the FP32 reciprocal square root,
//   y = y0 (1 + e/2 + 3 e^2 / 8),  e = 1 - m y0^2,  |e| < 2^-20,
// in integers (error below 2^-60), and y is rounded once to FP64: 0.501 ulp
// against about 1.5 for the FP64 sequence.  About 70 instructions, 20 of them
// multiplications.
#pragma once
#include <stdint.h>

namespace eifmm {

// |d| below 2^54 units is refused: 64 leading bits would reach below the
// coordinates' last place.
constexpr unsigned kFxMinHi = 1u << 12;

// 1 / (|d| 2^-K) for |dx|, |dy|, |dz| <= 2^62; kb = K + 958.  False (and no
// value) when |d| < 2^54 or so.
__device__ __forceinline__ bool inv_fx(long long dx, long long dy, long long dz, int kb, double* out) {
  // d = h 2^32 + l with l signed
  const int lx = (int)dx, ly = (int)dy, lz = (int)dz;
  const int hx = (int)(dx >> 32) + (int)((unsigned)lx >> 31);
  const int hy = (int)(dy >> 32) + (int)((unsigned)ly >> 31);
  const int hz = (int)(dz >> 32) + (int)((unsigned)lz >> 31);
  long long A = (long long)hx * hx, B = (long long)hx * lx;
  unsigned long long C = (unsigned long long)((long long)lx * lx);
  A += (long long)hy * hy;
  B += (long long)hy * ly;
  C += (unsigned long long)((long long)ly * ly);
  A += (long long)hz * hz;
  B += (long long)hz * lz;
  C += (unsigned long long)((long long)lz * lz);
  // |d|^2 = A 2^64 + 2 B 2^32 + C = a 2^64 + rem 2^32
  const long long T = B + (long long)(C >> 33);
  const long long a = A + (T >> 31);
  const unsigned rem = (unsigned)T << 1, ah = (unsigned)(a >> 32), al = (unsigned)a;
  if (ah < kFxMinHi) return false;
  const int sh = __clz(ah) & ~1;  // even: m 2^(126 - sh) has an integer root exponent
  const unsigned r1 = __funnelshift_l(al, ah, sh), r0 = __funnelshift_l(rem, al, sh);
  // y0 = Y0 2^-23; 2^23 + y0 2^23 has Y0 as its mantissa
  const float t = fmaf(rsqrtf((float)r1), 274877906944.0f /* 2^38 */, 8388608.0f);
  const unsigned Y0 = __float_as_uint(t) - 0x4B000000u;
  // D = 2^76 (1 - m y0^2), |D| < 2^56: modulo 2^64 the leading term drops
  const unsigned long long P = (unsigned long long)Y0 * Y0;
  const unsigned p0 = (unsigned)P, p1 = (unsigned)(P >> 32);
  unsigned long long S = (unsigned long long)r1 * p0 + __umulhi(r0, p0);
  S += (unsigned long long)r0 * p1;
  S += (unsigned long long)(r1 * p1) << 32;
  const long long D = -(long long)S;
  const int dh = (int)(D >> 32);
  const unsigned dl = (unsigned)D;
  const long long c = (long long)(int)Y0 * dh + __umulhi(Y0, dl);     // Y0 D 2^-32
  const unsigned long long q = (unsigned long long)((long long)dh * dh);
  const unsigned s2 = __umulhi(3u * (unsigned)(q >> 18), Y0) >> 1;     // 3/8 e^2 Y0 2^40
  // y 2^63 = Y0 2^40 (1 + ...), rounded to 53 bits; bit 52 of Y >> 10 adds
  // the implicit one to the exponent field
  const unsigned long long Y = ((unsigned long long)Y0 << 40) + (unsigned long long)(c >> 5) + s2 + 512;
  *out = __longlong_as_double((long long)((Y >> 10) + ((unsigned long long)(unsigned)((sh >> 1) + kb) << 52)));
  return true;
}

// p 2^K modulo 2^64, rounded to the nearest unit (exact when the last bit of p
// is worth a unit or more).
__device__ __forceinline__ long long to_fx(double p, int K) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(p);
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned long long m = (b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
  const int s = (e ? e : 1) - 1075 + K;  // p = m 2^(e - 1075)
  unsigned long long q;
  if (s >= 0) q = s < 64 ? m << s : 0;
  else q = s > -64 ? (m >> (-s)) + ((m >> (-s - 1)) & 1) : 0;
  return (long long)(b >> 63 ? 0 - q : q);
}

}  // namespace eifmm
