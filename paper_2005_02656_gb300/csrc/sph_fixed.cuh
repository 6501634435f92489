// The FP64 kernel series in 64-bit fixed point.
//
// FP64 instructions run at 2 per clock and SM on this part (1/64 of FP32);
// measured: 1.9 DFMA against 7.3 64x64-bit high products, 29 32-bit high
// products and 58 32-bit multiply-adds per clock and SM.  S(v) of Eq. 6 has a
// fixed range (argument in [0, 4), value in [0, 1]), so its series needs no
// floating point: evaluated on the integer pipes it costs about a third of
// the 15 FP64 multiply-adds of the same series, beside an FP64 pipe that is
// free for the sums.  The rounding is smaller, too: the absolute error of S is
// below 2^-59 over [0, 4), against about 2^-52 for the FP64 Horner form.
#pragma once

#include <stdint.h>

namespace sph {
namespace fx {

#ifdef __CUDA_ARCH__
#define SPH_FX __device__ __forceinline__
SPH_FX float rsqrt32(float a) { return rsqrtf(a); }
SPH_FX uint32_t bits_of(float v) { return __float_as_uint(v); }
SPH_FX float from_bits(uint32_t b) { return __uint_as_float(b); }
SPH_FX uint32_t mulhi32(uint32_t a, uint32_t b) { return __umulhi(a, b); }
SPH_FX int clz64(uint64_t a) { return __clzll((long long)a); }
// a >> s, 0 for s outside 0..63 (PTX shr clamps its amount, taken as unsigned).  With
// it a pair's conversions cost what they did before zero had a shift of its own (1.07M
// particles 13.51 ms per step; 13.64 with the amount clamped by an instruction more).
SPH_FX uint64_t shr64(uint64_t a, int s) {
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
}
SPH_FX uint64_t bits_of(double v) { return (uint64_t)__double_as_longlong(v); }
SPH_FX double from_bits(uint64_t b) { return __longlong_as_double((long long)b); }
#else
#define SPH_FX inline
SPH_FX float rsqrt32(float a) { return (float)(1.0 / __builtin_sqrt((double)a)); }
SPH_FX uint32_t bits_of(float v) { uint32_t b; __builtin_memcpy(&b, &v, 4); return b; }
SPH_FX float from_bits(uint32_t b) { float v; __builtin_memcpy(&v, &b, 4); return v; }
SPH_FX uint32_t mulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
SPH_FX int clz64(uint64_t a) { return a ? __builtin_clzll(a) : 64; }
SPH_FX uint64_t shr64(uint64_t a, int s) { return (unsigned)s < 64u ? a >> s : 0; }
SPH_FX uint64_t bits_of(double v) { uint64_t b; __builtin_memcpy(&b, &v, 8); return b; }
SPH_FX double from_bits(uint64_t b) { double v; __builtin_memcpy(&v, &b, 8); return v; }
#endif

// High 64 bits of a * b, at most 3 too small: the low words' product and the
// carries of the cross products' low halves are left out (3 multiplies, not 4).
SPH_FX uint64_t mulhi64(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a;
  const uint32_t bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  return (uint64_t)ah * bh + mulhi32(ah, bl) + mulhi32(al, bh);
}

// a_k = pi^(2k) / (2k + 1)!, so S(v) = sum_k (-1)^k a_k y^k at y = t / 4 =
// v^2 / 4, in units of 2^-64 (a_1 in 2^-63); d_k = k a_k (d_1, d_2 in 2^-63).
// 16 terms: the first one left out is below 1.1e-21 (S) and 1.7e-20 (dS/dy).
struct Coefs {
  uint64_t a1 = 0xd28d3312983e9918u, a2 = 0xcfce5a015e236291u, a3 = 0x30d51c8e41b6cdaeu,
           a4 = 0x06b1a0173cd4298cu, a5 = 0x0099c0b552303d5bu, a6 = 0x0009ba38cfd59c8bu,
           a7 = 0x0000750926347382u, a8 = 0x0000043f264bfce8u, a9 = 0x0000001f5f9d970du;
  uint32_t a10 = 0xbcbc4342u, a11 = 0x03ae6a72u, a12 = 0x000f808bu, a13 = 0x000037cbu,
           a14 = 0x000000aeu, a15 = 0x00000002u;
};

// y = t / 4 in units of 2^-64 for 0 <= t < 4 (the mantissa shifted to its place;
// bits below 2^-64 are dropped).
SPH_FX uint64_t fraction(double t) {
  const uint64_t b = bits_of(t);
  const int s = 1024 - (int)(b >> 52);
  return ((b << 11) | 0x8000000000000000u) >> (s < 63 ? s : 63);
}

// S in units of 2^-63, 0 <= S < 2^63.
SPH_FX uint64_t sinc(uint64_t y) {
  constexpr Coefs C{};
  const uint32_t yh = (uint32_t)(y >> 32);
  // a_10 and beyond fit 32 bits
  uint32_t q = C.a14 - mulhi32(yh, C.a15);
  q = C.a13 - mulhi32(yh, q);
  q = C.a12 - mulhi32(yh, q);
  q = C.a11 - mulhi32(yh, q);
  q = C.a10 - mulhi32(yh, q);
  uint64_t s = C.a9 - mulhi32(yh, q);
  s = C.a8 - mulhi64(y, s);
  s = C.a7 - mulhi64(y, s);
  s = C.a6 - mulhi64(y, s);
  s = C.a5 - mulhi64(y, s);
  s = C.a4 - mulhi64(y, s);
  s = C.a3 - mulhi64(y, s);
  s = C.a2 - mulhi64(y, s);
  s = C.a1 - (mulhi64(y, s) >> 1);
  const int64_t r = (int64_t)(0x7fffffffffffffffu - mulhi64(y, s));
  return r > 0 ? (uint64_t)r : 0u;  // rounding may pass zero at the support's edge
}

// -dS/dy in units of 2^-63 (0.5 at y = 1, pi^2 / 6 at y = 0).
SPH_FX uint64_t sinc_slope(uint64_t y) {
  const uint32_t yh = (uint32_t)(y >> 32);
  uint32_t q = 0x0000097fu - mulhi32(yh, 0x0000001cu);  // d_14 - y d_15
  q = 0x0002d555u - mulhi32(yh, q);
  q = 0x00ba0682u - mulhi32(yh, q);
  q = 0x287e92ebu - mulhi32(yh, q);
  uint64_t s = 0x000000075f5aa095u - mulhi32(yh, q);
  s = 0x0000011a5c8a4f72u - mulhi64(y, s);
  s = 0x000021f9325fe73cu - mulhi64(y, s);
  s = 0x000333400b6f2891u - mulhi64(y, s);
  s = 0x003a5d54df01ab40u - mulhi64(y, s);
  s = 0x0300c38a9af132c8u - mulhi64(y, s);
  s = 0x1ac6805cf350a62fu - mulhi64(y, s);
  s = 0x927f55aac524690bu - mulhi64(y, s);
  s = 0xcfce5a015e236291u - (mulhi64(y, s) >> 1);
  return 0xd28d3312983e9918u - mulhi64(y, s);
}

// The double nearest (ties away from zero) to f 2^(e - 64) for f != 0.
SPH_FX double pack(uint64_t f, int e) {
  const int z = clz64(f);
  const uint64_t m = f << z;  // [2^63, 2^64): the implicit bit adds one to the exponent
  return from_bits(((uint64_t)(uint32_t)(1021 + e - z) << 52) + (m >> 11) + ((m >> 10) & 1u));
}

// S as a double, for t >= 0; 0 at and beyond the support's edge t = 4 (which
// rounding of r^2 / h^2 can reach), and for a NaN.
SPH_FX double S(double t) {
  if ((uint32_t)(bits_of(t) >> 32) >= 0x40100000u) return 0.0;
  const uint64_t s = sinc(fraction(t));
  return s ? pack(s, 1) : 0.0;
}

// S^6, the powers taken on the normalised mantissa (relative error below 2^-52.9).
SPH_FX double S6(double t) {
  if ((uint32_t)(bits_of(t) >> 32) >= 0x40100000u) return 0.0;
  const uint64_t s = sinc(fraction(t));
  if (s == 0) return 0.0;
  const int z = clz64(s);
  const uint64_t m = s << z;  // S = m 2^(1 - z - 64)
  const uint64_t m2 = mulhi64(m, m);
  return pack(mulhi64(mulhi64(m2, m2), m2), 6 - 6 * z);
}

// S^6 at the fraction y, and a S^6: the mantissas are multiplied before the one
// rounding to a double (a normal and not near the ends of the range, or the
// product is taken in FP64).
SPH_FX double S6_at(uint64_t y) {
  const uint64_t s = sinc(y);
  if (s == 0) return 0.0;
  const int z = clz64(s);
  const uint64_t m = s << z, m2 = mulhi64(m, m);
  return pack(mulhi64(mulhi64(m2, m2), m2), 6 - 6 * z);
}
SPH_FX double S6_at_times(uint64_t y, double a) {
  const uint64_t b = bits_of(a);
  const int E = (int)(b >> 52) & 0x7ff;
  if (E < 512 || E > 1535) return a * S6_at(y);
  const uint64_t s = sinc(y);
  if (s == 0) return 0.0;
  const int z = clz64(s);
  const uint64_t m = s << z, m2 = mulhi64(m, m);
  const uint64_t f = mulhi64(mulhi64(mulhi64(m2, m2), m2), (b << 11) | 0x8000000000000000u);
  return from_bits(bits_of(pack(f, 6 - 6 * z + E - 1022)) | (b & 0x8000000000000000u));
}

// S^6 and its derivative by t, 6 S^5 dS/dt (dS/dt = (dS/dy) / 4), at the
// fraction y = t / 4.
SPH_FX void S6_d_at(uint64_t y, double& w, double& dw) {
  w = dw = 0.0;
  const uint64_t s = sinc(y);
  if (s == 0) return;
  const int z = clz64(s);
  const uint64_t m = s << z;
  const uint64_t m2 = mulhi64(m, m), m4 = mulhi64(m2, m2);
  w = pack(mulhi64(m4, m2), 6 - 6 * z);
  // 1.5 S^5 D: D in units of 2^-63 and 1.5 = 0.75 * 2 add two to the exponent
  const uint64_t d = mulhi64(mulhi64(m4, m), sinc_slope(y));
  dw = -pack(d - (d >> 2), 7 - 5 * z);
}
SPH_FX void S6_d(double t, double& w, double& dw) {
  w = dw = 0.0;
  if ((uint32_t)(bits_of(t) >> 32) < 0x40100000u) S6_d_at(fraction(t), w, dw);
}

// --- vectors in block fixed point ---
// A vector's components share one power of two: component v is held as the
// integer X = v 2^(N - e) (rounded toward zero), 2^e above every |v|, N = 61 (60
// for the matrices), and used in two signed limbs, X = 2^32 h + l exactly.  A scalar product
// of two such vectors is then nine 32-bit multiply-adds into two 64-bit sums,
// with no carries: |X| < 2^61 leaves room for three terms.

// Power of two above |v| for finite v, as the exponent field of a double plus
// one (v = 0 and subnormal v give 1 and are taken as zero by fixed()); 2048 for a
// value that is not finite.
SPH_FX int exp_above(double v) { return (int)((bits_of(v) >> 52) & 0x7ffu) + 1; }

// In place of a power of two: a vector or matrix that is not finite.  fixed() makes
// it zero, and scaled<true>() of a product that it enters gives NaN.
constexpr int kNotFinite = 1 << 14;

// v 2^(N - (eb - 1023)), |v| < 2^(eb - 1023); zero and subnormals give zero for
// every eb (a zero vector has eb = 1, where shifting out the implicit bit would not do).
template <int N>
SPH_FX int64_t fixed(double v, int eb) {
  const uint64_t b = bits_of(v);
  const int f = (int)((b >> 52) & 0x7ffu);
  const int s = f ? eb - f : 63;  // >= 1 (63: m >> s is zero)
  uint64_t m = (b & 0xfffffffffffffu) << (N - 52) | (uint64_t)1 << N;
  m = shr64(m, s);
  if (s <= 0) m = ((uint64_t)1 << N) - 1;  // |v| not below the power of two: the largest value
  const int64_t g = (int64_t)b >> 63;
  return ((int64_t)m ^ g) - g;
}

struct Vec3 {
  int32_t h[3];
  int32_t l[3];
};

SPH_FX void put(Vec3& v, int i, int64_t x) {
  v.l[i] = (int32_t)x;
  v.h[i] = (int32_t)(x >> 32) - (v.l[i] >> 31);
}

// sum_i A_i B_i / 2^62 for |A_i|, |B_i| < 2^61, the products of the low limbs
// left out (at most 3 units, of either sign) and the rest rounded.
SPH_FX int64_t dot(const Vec3& a, const Vec3& b) {
  int64_t hh = (int64_t)a.h[0] * b.h[0];
  int64_t cr = (int64_t)a.h[0] * b.l[0];
  cr += (int64_t)a.l[0] * b.h[0];
  hh += (int64_t)a.h[1] * b.h[1];
  cr += (int64_t)a.h[1] * b.l[1];
  cr += (int64_t)a.l[1] * b.h[1];
  hh += (int64_t)a.h[2] * b.h[2];
  cr += (int64_t)a.h[2] * b.l[2];
  cr += (int64_t)a.l[2] * b.h[2];
  return (hh << 2) + ((cr + (1 << 29)) >> 30);
}

// The double nearest to x 2^k; zero where that is below the normal range.  ANY:
// infinity above it, and NaN past every finite vector's reach (kNotFinite), for factors
// of any size (the forward pair sums, whose products stay inside, would spend 2% on the
// compare).
template <bool ANY = false>
SPH_FX double scaled(int64_t x, int k) {
  const int64_t g = x >> 63;
  const uint64_t u = (uint64_t)((x ^ g) - g);
  const int z = clz64(u);
  const int f = 1085 + k - z;  // exponent field, less the implicit bit
  if (u == 0 || (ANY ? (uint32_t)f > 2045u : f < 0)) {
    if (ANY && f > kNotFinite / 2) return from_bits((uint64_t)0x7ff8000000000000);
    return ANY && u != 0 && f > 0
               ? from_bits((uint64_t)0x7ff0000000000000 | ((uint64_t)g << 63)) : 0.0;
  }
  const uint64_t m = u << z;
  return from_bits((((uint64_t)(uint32_t)f << 52) + (m >> 11) + ((m >> 10) & 1u)) |
                   ((uint64_t)g << 63));
}

// y = t / 4 = r^2 / (4 h^2) in units of 2^-64 from R = r^2 2^-k (R < 2^60) and
// 1 / h^2 (normal); false where t >= 4.
SPH_FX bool fraction_of(uint64_t R, int k, double hinv2, uint64_t& y) {
  const uint64_t b = bits_of(hinv2);
  // 1 / h^2 = H 2^(E - 1086), H in [2^63, 2^64)
  const uint64_t p = mulhi64(R << 3, (b << 11) | 0x8000000000000000u);  // R H 2^-61
  const int s = (int)(b >> 52) - 1086 + 61 + 62 + k;                    // y 2^64 = p 2^s
  y = 0;
  if (s <= 0) {
    y = p >> (s > -63 ? -s : 63);
    return true;
  }
  if (s > 63 ? p != 0 : (p >> (64 - s)) != 0) return false;
  y = s > 63 ? 0 : p << s;
  return true;
}

// A positive double of the middle of the range as m 2^(e - 64), m in [2^62, 2^64)
// (products of two such values included).
struct Mant {
  uint64_t m;
  int e;
};
SPH_FX bool middle(double a) {
  const uint64_t b = bits_of(a);
  return (b >> 52) - 823u < 400u;  // positive, 2^-200 <= a < 2^200
}
SPH_FX Mant mant(double a) {
  const uint64_t b = bits_of(a);
  return {(b << 11) | 0x8000000000000000u, (int)(b >> 52) - 1022};
}
SPH_FX Mant operator*(const Mant& a, const Mant& b) { return {mulhi64(a.m, b.m), a.e + b.e}; }

// a x for x in fixed point (units 2^k, |x| < 2^61).
SPH_FX double times(const Mant& a, int64_t x, int k) {
  const int64_t g = x >> 63;
  const uint64_t u = (uint64_t)((x ^ g) - g);
  const uint64_t f = mulhi64(a.m, u << 3);  // a x 2^-k 2^(3 - e)
  if (f == 0) return 0.0;
  return from_bits(bits_of(pack(f, a.e + k + 61)) | ((uint64_t)g << 63));
}

// v 2^kv / sqrt(R 2^kr) for v != 0 and R >= 2^52 (whose error of a unit is then
// below 2^-52): y0 from the FP32 reciprocal square root, and the factor
// 1 + e/2 + 3 e^2/8 with e = 1 - R y0^2, in 64-bit fixed point.  Zero below 2^-900; the
// callers' results end below 2^802.
SPH_FX double over_root(int64_t v, int kv, uint64_t R, int kr) {
  int z = clz64(R);
  uint64_t m = R << z;  // m 2^-62 in [2, 4)
  int x = 62 - z + kr;
  if (x & 1) {
    m >>= 1;            // [1, 2)
    ++x;
  }
  const float y0 = rsqrt32((float)(uint32_t)(m >> 32) * 9.313225746154785e-10f);  // 2^-30
  const uint32_t Y = (uint32_t)(y0 * 2147483648.0f);                             // y0 2^31, exact
  const int64_t e = (int64_t)0x2000000000000000 - (int64_t)mulhi64(m, ((uint64_t)Y * Y) << 1);
  const int64_t e20 = e >> 20;
  const int64_t q = (e >> 1) + ((3 * e20 * e20) >> 24);                          // 2^61
  const int64_t g = v >> 63;
  const uint64_t u = (uint64_t)((v ^ g) - g);
  const int zv = clz64(u);
  const uint64_t n = u << zv;
  uint64_t t = (uint64_t)(uint32_t)(n >> 32) * Y + mulhi32((uint32_t)n, Y);      // n y0 / 2
  t = q < 0 ? t - mulhi64(t, (uint64_t)-q << 3) : t + mulhi64(t, (uint64_t)q << 3);
  const int ex = 65 - zv + kv - (x >> 1);  // result t 2^(ex - 64)
  if (ex < -900 || ex > 900) return 0.0 * (double)g;
  return from_bits(bits_of(pack(t, ex)) | ((uint64_t)g << 63));
}

}  // namespace fx
}  // namespace sph
