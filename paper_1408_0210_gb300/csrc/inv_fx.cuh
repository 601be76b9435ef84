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

// A sum of squares a 2^64 + rem 2^32 normalised to R = m 2^62, 1 <= m < 4: the
// sum is m 2^(126 - sh), sh even.  False when a is below 2^44.
__device__ __forceinline__ bool fx_normalise(long long a, unsigned rem, unsigned long long* R, int* sh) {
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  if (ah < kFxMinHi) return false;
  *sh = __clz(ah) & ~1;
  const unsigned r1 = __funnelshift_l(al, ah, *sh), r0 = __funnelshift_l(rem, al, *sh);
  *R = (unsigned long long)r1 << 32 | r0;
  return true;
}

// 2^63 / sqrt(m) from R = m 2^62, error a few units.
__device__ __forceinline__ unsigned long long fx_rsqrt(unsigned long long R) {
  const unsigned r1 = (unsigned)(R >> 32), r0 = (unsigned)R;
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
  return ((unsigned long long)Y0 << 40) + (unsigned long long)(c >> 5) + s2;
}

// 2^K / sqrt(m 2^(126 - sh)) as a double from Y = 2^63 / sqrt(m), rounded; bit 52
// of Y >> 10 adds the implicit one to the exponent field.  kb = K + 958.
__device__ __forceinline__ double fx_double(unsigned long long Y, int sh, int kb) {
  return __longlong_as_double(
      (long long)(((Y + 512) >> 10) + ((unsigned long long)(unsigned)((sh >> 1) + kb) << 52)));
}

// d = h 2^32 + l with l signed; the squares as A 2^64 + 2 B 2^32 + C
struct FxSquare {
  long long A = 0, B = 0;
  unsigned long long C = 0;
  __device__ __forceinline__ void add(long long d) {
    const int l = (int)d, h = (int)(d >> 32) + (int)((unsigned)l >> 31);
    A += (long long)h * h;
    B += (long long)h * l;
    C += (unsigned long long)((long long)l * l);
  }
  // = a 2^64 + rem 2^32 (the rest below is dropped)
  __device__ __forceinline__ void value(long long* a, unsigned* rem) const {
    const long long T = B + (long long)(C >> 33);
    *a = A + (T >> 31);
    *rem = (unsigned)T << 1;
  }
};

// 1 / (|d| 2^-K) for |dx|, |dy|, |dz| <= 2^62; kb = K + 958.  False (and no
// value) when |d| < 2^54 or so.
__device__ __forceinline__ bool inv_fx(long long dx, long long dy, long long dz, int kb, double* out) {
  FxSquare s;
  s.add(dx);
  s.add(dy);
  s.add(dz);
  long long a;
  unsigned rem;
  s.value(&a, &rem);
  unsigned long long R;
  int sh;
  if (!fx_normalise(a, rem, &R, &sh)) return false;
  *out = fx_double(fx_rsqrt(R), sh, kb);
  return true;
}

// exp(-r) for 0 <= r < 700, about 1 ulp: the table-driven scheme of P. T. P. Tang
// (ACM TOMS 15, 1989) with 64 entries 2^(j/64), -r = k ln2/64 + f, and the Taylor
// polynomial of e^f - 1 of degree 5 (|f| < 0.0055: the next term is below 4e-17).
__device__ const double kExp2Tab[64] = {
    0x1.0000000000000p+0, 0x1.02c9a3e778061p+0, 0x1.059b0d3158574p+0, 0x1.0874518759bc8p+0,
    0x1.0b5586cf9890fp+0, 0x1.0e3ec32d3d1a2p+0, 0x1.11301d0125b51p+0, 0x1.1429aaea92de0p+0,
    0x1.172b83c7d517bp+0, 0x1.1a35beb6fcb75p+0, 0x1.1d4873168b9aap+0, 0x1.2063b88628cd6p+0,
    0x1.2387a6e756238p+0, 0x1.26b4565e27cddp+0, 0x1.29e9df51fdee1p+0, 0x1.2d285a6e4030bp+0,
    0x1.306fe0a31b715p+0, 0x1.33c08b26416ffp+0, 0x1.371a7373aa9cbp+0, 0x1.3a7db34e59ff7p+0,
    0x1.3dea64c123422p+0, 0x1.4160a21f72e2ap+0, 0x1.44e086061892dp+0, 0x1.486a2b5c13cd0p+0,
    0x1.4bfdad5362a27p+0, 0x1.4f9b2769d2ca7p+0, 0x1.5342b569d4f82p+0, 0x1.56f4736b527dap+0,
    0x1.5ab07dd485429p+0, 0x1.5e76f15ad2148p+0, 0x1.6247eb03a5585p+0, 0x1.6623882552225p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6dfb23c651a2fp+0, 0x1.71f75e8ec5f74p+0, 0x1.75feb564267c9p+0,
    0x1.7a11473eb0187p+0, 0x1.7e2f336cf4e62p+0, 0x1.82589994cce13p+0, 0x1.868d99b4492edp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8f1ae99157736p+0, 0x1.93737b0cdc5e5p+0, 0x1.97d829fde4e50p+0,
    0x1.9c49182a3f090p+0, 0x1.a0c667b5de565p+0, 0x1.a5503b23e255dp+0, 0x1.a9e6b5579fdbfp+0,
    0x1.ae89f995ad3adp+0, 0x1.b33a2b84f15fbp+0, 0x1.b7f76f2fb5e47p+0, 0x1.bcc1e904bc1d2p+0,
    0x1.c199bdd85529cp+0, 0x1.c67f12e57d14bp+0, 0x1.cb720dcef9069p+0, 0x1.d072d4a07897cp+0,
    0x1.d5818dcfba487p+0, 0x1.da9e603db3285p+0, 0x1.dfc97337b9b5fp+0, 0x1.e502ee78b3ff6p+0,
    0x1.ea4afa2a490dap+0, 0x1.efa1bee615a27p+0, 0x1.f50765b6e4540p+0, 0x1.fa7c1819e90d8p+0};
__device__ __forceinline__ double exp_neg(double r) {
  const double magic = 6755399441055744.0;  // 1.5 2^52: k lands in the low word
  const double t = fma(r, -0x1.71547652b82fep+6, magic);
  const int k = (int)__double_as_longlong(t);
  const double kd = t - magic;
  // ln2/64 in two parts, the first with 21 trailing zero bits (k below 2^17)
  const double f = fma(-kd, 0x1.a39ef35793c76p-39, fma(-kd, 0x1.62e42fee00000p-7, -r));
  double q = fma(f, 1.0 / 120.0, 1.0 / 24.0);
  q = fma(q, f, 1.0 / 6.0);
  q = fma(q, f, 0.5);
  const double p = fma(f * f, q, f);
  const double T = __ldg(kExp2Tab + (k & 63));
  const double e = fma(T, p, T);
  return __longlong_as_double(__double_as_longlong(e) + ((long long)(k >> 6) << 52));
}

// The config-3 kernel e^-r / r + 1 / sqrt(d_x^2 + 0.01 d_y^2 + d_z^2 + 1e-3) on the
// same integers; e128: 1e-3 2^(2 K) as hi and lo words.
struct FxConfig3 {
  unsigned long long e_hi, e_lo;
};
__device__ __forceinline__ bool config3_fx(long long dx, long long dy, long long dz, int kb, const FxConfig3& c,
                                           double* out) {
  FxSquare s02, s1;
  s02.add(dx);
  s02.add(dz);
  s1.add(dy);
  long long a02, a1, ar;
  unsigned q02, q1, qr;
  s02.value(&a02, &q02);
  s1.value(&a1, &q1);
  unsigned long long lo = ((unsigned long long)q02 << 32) + ((unsigned long long)q1 << 32);
  ar = a02 + a1 + (long long)(lo < ((unsigned long long)q02 << 32));
  qr = (unsigned)(lo >> 32);
  unsigned long long R;
  int sh;
  if (!fx_normalise(ar, qr, &R, &sh)) return false;
  const unsigned long long Y = fx_rsqrt(R);
  // r = |d|^2 / |d|: sqrt(m) 2^61 from the product of R and Y
  const unsigned long long rr = __umul64hi(R, Y);
  const double r = __longlong_as_double(
      (long long)(((rr + 256) >> 9) + ((unsigned long long)(unsigned)(2043 - kb - (sh >> 1)) << 52)));
  // 0.01 d_y^2: times 0.01 2^64, of the 96 bits a1:q1
  const unsigned long long k = 184467440737095516ull;
  unsigned long long hl = (unsigned long long)a1 * k, hh = __umul64hi((unsigned long long)a1, k);
  auto add = [&](unsigned long long h, unsigned long long l) {
    hl += l;
    hh += h + (hl < l ? 1 : 0);
  };
  add(0, (unsigned long long)q1 * (unsigned)(k >> 32));
  add((unsigned long long)a02, (unsigned long long)q02 << 32);
  add(c.e_hi, c.e_lo);
  unsigned long long R2;
  int sh2;
  if (!fx_normalise((long long)hh, (unsigned)(hl >> 32), &R2, &sh2)) return false;
  *out = fma(exp_neg(r), fx_double(Y, sh, kb), fx_double(fx_rsqrt(R2), sh2, kb));
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
