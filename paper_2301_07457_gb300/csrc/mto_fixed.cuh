// 96-bit fixed-point arithmetic for the float64 element operator.
//
// On GB300 the FP64 pipe issues one add, multiply or FMA for about 38 integer
// instructions of the same warp, so a float64 stencil is bound by that pipe at
// a fifth of the memory bandwidth.  Almost all of the element operator is sums
// and differences, which integers do exactly once the values share a scale.
// The sweeps therefore convert the marched nodal values to integers with one
// scale per warp, add and multiply them on the integer pipe, and round once,
// when K v goes back to float64.
//
// Scales.  A nodal value is  F 2^(B - 1113)  with B the largest (biased)
// float64 exponent met by the warp so far: the value with exponent B has its
// 53 significant bits at bits 38..90 of F, four bits below the sign bit for the
// strain coordinates (sums of up to eight values).  A value of exponent e is
// represented exactly down to e = B - 38 and with an absolute error below
// 2^-90 of the warp's largest value under that.  Element coefficients are
// 61-bit integers with one exponent X per element; a product keeps the upper
// 96 of its 157 bits, so forces are  T 2^(B + Xm - 2132)  with Xm the largest X
// met so far (coarse elements: 59-bit integers, T 2^(B + Xm - 2130)): the last
// bit relates to the largest coefficient times the largest value of the window,
// not to the largest force.  Every sum of the operator fits: |K v| < 2^95
// (bounds at the kernel).
//
// A window (30 columns by the rows of a task, 14 columns by three rows, or a
// tile) shares its scales, so the error of a node's K v is absolute, whatever
// the size of its own terms: FX_SPAN_* below says from where on they are
// evaluated in float64 instead.
//
// The functions also compile as host code (checked against 128-bit
// arithmetic there).
#pragma once

#include "mto_common.cuh"

namespace mto {

struct Fx {
  unsigned lo, mid;
  int hi;
};

__host__ __forceinline__ __int128 fx_wide(const Fx& a) {
  return ((__int128)a.hi << 64) | ((unsigned long long)a.mid << 32) | a.lo;
}
__host__ __forceinline__ Fx fx_narrow(__int128 v) {
  return Fx{(unsigned)v, (unsigned)(v >> 32), (int)(v >> 64)};
}

__host__ __device__ __forceinline__ Fx fx_add(const Fx& a, const Fx& b) {
#ifdef __CUDA_ARCH__
  Fx r;
  asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
      : "=r"(r.lo), "=r"(r.mid), "=r"(r.hi)
      : "r"(a.lo), "r"(a.mid), "r"(a.hi), "r"(b.lo), "r"(b.mid), "r"(b.hi));
  return r;
#else
  return fx_narrow(fx_wide(a) + fx_wide(b));
#endif
}
__host__ __device__ __forceinline__ Fx fx_sub(const Fx& a, const Fx& b) {
#ifdef __CUDA_ARCH__
  Fx r;
  asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %7;\n\tsubc.u32 %2, %5, %8;"
      : "=r"(r.lo), "=r"(r.mid), "=r"(r.hi)
      : "r"(a.lo), "r"(a.mid), "r"(a.hi), "r"(b.lo), "r"(b.mid), "r"(b.hi));
  return r;
#else
  return fx_narrow(fx_wide(a) - fx_wide(b));
#endif
}
__host__ __device__ __forceinline__ Fx fx_zero() { return Fx{0u, 0u, 0}; }
__host__ __device__ __forceinline__ Fx fx_neg(const Fx& a) { return fx_sub(fx_zero(), a); }

// Low 32 bits of (hi:lo) >> s, 0 <= s < 32.
__host__ __device__ __forceinline__ unsigned fx_funnel(unsigned lo, unsigned hi, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_r(lo, hi, s);
#else
  return (unsigned)((((unsigned long long)hi << 32) | lo) >> s);
#endif
}

// High 32 bits of (hi:lo) << s, 0 <= s < 32.
__host__ __device__ __forceinline__ unsigned fx_funnel_left(unsigned lo, unsigned hi, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, s);
#else
  return (unsigned)(((((unsigned long long)hi << 32) | lo) << s) >> 32);
#endif
}

// a >> s (floor), 0 <= s < 32.
__host__ __device__ __forceinline__ Fx fx_sar31(const Fx& a, int s) {
  return Fx{fx_funnel(a.lo, a.mid, s), fx_funnel(a.mid, (unsigned)a.hi, s), a.hi >> s};
}
// a >> s by whole limbs: s - s mod 32 bits, any s >= 0.
__host__ __device__ __forceinline__ Fx fx_sar_limbs(Fx a, int s) {
  const int sg = a.hi >> 31;
  if (s >= 64) {
    a = Fx{(unsigned)a.hi, (unsigned)sg, sg};
    if (s >= 96) a = Fx{(unsigned)sg, (unsigned)sg, sg};
  } else if (s >= 32) {
    a = Fx{a.mid, (unsigned)a.hi, sg};
  }
  return a;
}
__host__ __device__ __forceinline__ Fx fx_sar(const Fx& a, int s) {
  return fx_sar31(fx_sar_limbs(a, s), s & 31);
}

// The significand of a finite float64 before the shift to the common scale
// (by B - max(exponent, 1)): times 2^38, upper two limbs (the lowest is zero),
// with sign.  With FLUSH subnormals give zero: where B > FX_FLUSH_B they lie
// more than 96 bits below the scale.
constexpr int FX_FLUSH_B = 97;
template <bool FLUSH> __host__ __device__ __forceinline__ Fx fx_significand(unsigned long long bits) {
  const unsigned hi = (unsigned)(bits >> 32);
  const bool normal = (hi & 0x7ff00000u) != 0u;
  const unsigned lo = FLUSH && !normal ? 0u : (unsigned)bits;
  const unsigned mh = normal ? (hi & 0xfffffu) | 0x100000u : (FLUSH ? 0u : hi & 0xfffffu);
  const unsigned sg = (unsigned)((int)hi >> 31);
  unsigned u1 = (lo << 6) ^ sg, u2 = ((mh << 6) | (lo >> 26)) ^ sg;
#ifdef __CUDA_ARCH__
  asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %2;" : "+r"(u1), "+r"(u2) : "r"(sg));
#else
  const unsigned long long t = (((unsigned long long)u2 << 32) | u1) - (((unsigned long long)sg << 32) | sg);
  u1 = (unsigned)t;
  u2 = (unsigned)(t >> 32);
#endif
  return Fx{0u, u1, (int)u2};
}

// Sign change by a mask (0 or -1).
__host__ __device__ __forceinline__ Fx fx_flip(const Fx& a, int mask) {
#ifdef __CUDA_ARCH__
  Fx r;
  const unsigned m = (unsigned)mask;
  asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %6;\n\tsubc.u32 %2, %5, %6;"
      : "=r"(r.lo), "=r"(r.mid), "=r"(r.hi)
      : "r"(a.lo ^ m), "r"(a.mid ^ m), "r"((unsigned)a.hi ^ m), "r"(m));
  return r;
#else
  return mask ? fx_neg(a) : a;
#endif
}

// (w c) >> 64 for 0 <= c < 2^61, up to 2 units low (the lowest of the six
// partial products and the lower halves of the next two are left out).
__host__ __device__ __forceinline__ Fx fx_mul(const Fx& w, unsigned long long c) {
  const unsigned c0 = (unsigned)c, c1 = (unsigned)(c >> 32);
#ifdef __CUDA_ARCH__
  const unsigned h0 = __umulhi(w.lo, c1), h1 = __umulhi(w.mid, c0);
  const unsigned long long x = (unsigned long long)w.mid * c1 + h0;
  const unsigned long long y = (unsigned long long)(unsigned)w.hi * c0 + h1;
  // The middle product takes w.hi as unsigned: 2^32 c0 too much when negative.
  const unsigned corr = (unsigned)(w.hi >> 31) & c0;
  const long long z = (long long)w.hi * (int)c1 - (long long)corr;
  const unsigned xl = (unsigned)x, xh = (unsigned)(x >> 32), yl = (unsigned)y, yh = (unsigned)(y >> 32);
  const unsigned zl = (unsigned)z, zh = (unsigned)((unsigned long long)z >> 32);
  Fx r;
  asm("add.cc.u32 %0, %3, %5;\n\taddc.cc.u32 %1, %4, %6;\n\taddc.u32 %2, %8, 0;\n\t"
      "add.cc.u32 %1, %1, %7;\n\taddc.u32 %2, %2, 0;"
      : "=&r"(r.lo), "=&r"(r.mid), "=&r"(r.hi)
      : "r"(xl), "r"(xh), "r"(yl), "r"(yh), "r"(zl), "r"(zh));
  return r;
#else
  const unsigned long long h0 = ((unsigned long long)w.lo * c1) >> 32, h1 = ((unsigned long long)w.mid * c0) >> 32;
  return fx_narrow((__int128)((unsigned long long)w.mid * c1 + h0) + (__int128)h1 +
                   (__int128)w.hi * c0 + (((__int128)w.hi * c1) << 32));
#endif
}

// v 2^u rounded to float64 (to nearest but for ties, and for the bits dropped
// below the 64th significant one); subnormal results and overflow as IEEE
// (rounded twice at most).
//
// CHECKED = false leaves the exponent's range to the caller, who knows that u
// lies in [FX_UNIT_MIN, FX_UNIT_MAX] (the result is normal or zero then).
constexpr int FX_UNIT_MIN = -1020, FX_UNIT_MAX = 920;
template <bool CHECKED = true> __host__ __device__ __forceinline__ double fx_to_double(const Fx& v, int u) {
  const unsigned sg = (unsigned)(v.hi >> 31);
#ifdef __CUDA_ARCH__
  unsigned a0 = v.lo ^ sg, a1 = v.mid ^ sg, a2 = (unsigned)v.hi ^ sg;
  asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;"
      : "+r"(a0), "+r"(a1), "+r"(a2)
      : "r"(sg));
#else
  const Fx mag = v.hi < 0 ? fx_neg(v) : v;
  unsigned a0 = mag.lo, a1 = mag.mid, a2 = (unsigned)mag.hi;
#endif
  int ex = u + 63 + 32 + 1022;  // biased exponent less one of a 64-bit significand (a2:a1) with its top bit set
  if (a2 == 0u) {
    a2 = a1;
    a1 = a0;
    a0 = 0u;
    ex -= 32;
  }
  if (a2 == 0u) {
    a2 = a1;
    a1 = a0;
    a0 = 0u;
    ex -= 32;
  }
#ifdef __CUDA_ARCH__
  const int lz = __clz((int)a2);
#else
  const int lz = a2 ? __builtin_clz(a2) : 32;
#endif
  a2 = fx_funnel_left(a1, a2, lz & 31);
  a1 = fx_funnel_left(a0, a1, lz & 31);
  ex -= lz;
  const unsigned long long m = ((unsigned long long)a2 << 32) | a1;
  const unsigned long long sign = (unsigned long long)(sg & 0x80000000u) << 32;
  if (CHECKED && a2 != 0u && (ex < 0 || ex >= 2045)) {  // outside the normal range
#ifdef __CUDA_ARCH__
    const double r = ldexp(__ull2double_rn(m), ex - 63 - 1022);
#else
    const double r = __builtin_ldexp((double)m, ex - 63 - 1022);
#endif
    return double_of(bits_of(r) | sign);
  }
  const double r = double_of(((m >> 11) + ((m >> 10) & 1u) + ((unsigned long long)(unsigned)ex << 52)) | sign);
  return a2 != 0u ? r : 0.0;
}

// (m << lift) aligned to exponent X, for a factor f of magnitude m 2^(e - 1075).
__host__ __device__ __forceinline__ unsigned long long fx_coef_word(double f, int X, int lift) {
  const unsigned long long b = bits_of(f);
  const int e = fx_exponent((unsigned)(b >> 32));
  unsigned long long m = b & 0xfffffffffffffull;
  if (e) m |= 0x10000000000000ull;
  const int s = X - (e ? e : 1);
  return s < 64 ? (m << lift) >> s : 0ull;
}
// Common exponent of n factors: the largest of theirs (0 only if all are zero).
__host__ __device__ __forceinline__ int fx_common_exponent(const double* f, int n) {
  int X = 0;
  for (int i = 0; i < n; ++i) {
    const unsigned hi = (unsigned)(bits_of(f[i]) >> 32);
    int e = fx_exponent(hi);
    if (e == 0 && f[i] != 0.0) e = 1;  // subnormal
    if (e > X) X = e;
  }
  return X;
}
// The low four bits of an element's first three words hold a 12-bit tag: the
// exponent X and, in bit 11, that a factor is negative that no positive
// modulus makes negative.  They are worth at most 2^-55 of the largest factor,
// below float64's rounding of it, and stay in the products.
constexpr unsigned FX_TAG_NEG = 0x800u;
__host__ __device__ __forceinline__ void fx_put_tag(unsigned long long* w, unsigned tag) {
  for (int i = 0; i < 3; ++i) w[i] = (w[i] & ~15ull) | ((tag >> (4 * i)) & 15u);
}
__host__ __device__ __forceinline__ unsigned fx_tag(const unsigned long long* w) {
  return ((unsigned)w[0] & 15u) | (((unsigned)w[1] & 15u) << 4) | (((unsigned)w[2] & 15u) << 8);
}

// Factor c 2^(X - bias) of an element with tag `tag`, NaN where the element is
// not finite (formed on the integer pipe).
__host__ __device__ __forceinline__ double fx_factor(unsigned long long c, bool neg, unsigned tag, int bias) {
  const int X = (int)(tag & 0x7ffu);
  const double f = fx_to_double(Fx{(unsigned)c, (unsigned)(c >> 32), 0}, X - bias);
  return double_of(X == 0x7ff ? 0x7ff8000000000000ull : bits_of(f) | (neg ? 0x8000000000000000ull : 0ull));
}

// Upper word of the larger magnitude of a pair.
__host__ __device__ __forceinline__ unsigned fx_magnitude(double x, double y) {
  const unsigned a = (unsigned)(bits_of(x) >> 32) & 0x7fffffffu, b = (unsigned)(bits_of(y) >> 32) & 0x7fffffffu;
  return a > b ? a : b;
}
// Whether scales of weight Q = B + Xm lose too much of an element of weight q,
// the sum of the (biased) exponents of its largest factor and of its largest
// nodal value: beyond span places the element is done in float64.
//
// The terms |K||v| of a node next to the element are at least about 2^(q - 2046).
// Its error is at most 18 units of the last place, so 2^(Q - q - 82) of them,
// and usually 2^-6 of that.  Measured on a soft block beside solids, random values
// of one size: error over the row's terms (largest / root mean square) 2.1e-16 /
// 5.7e-17 up to Q - q = 34, 2.9e-16 / 6.5e-17 at 36, 3.0e-16 / 7.7e-17 at 37,
// 3.5e-16 / 7.8e-17 at 38, against 4.1e-16 / 7.7e-17 in float64: the line lies at the
// last one that is better than float64 in both.  A coarse element's factors have
// two bits fewer and its terms are cut off more often: 3.6e-16 / 9.3e-17 at 33,
// 4.8e-16 / 1.0e-16 at 34, 5.7e-16 / 1.4e-16 at 35, 1.3e-15 / 2.3e-16 at 36, against
// 4.8e-16 / 9.0e-17 in float64.  With the line at 34 the whole sweep (elements on
// both sides of it) shows at most 4.8e-16 / 9.1e-17, at 36 5.2e-16 / 1.1e-16.
// A void of 1e-9 (2^-30) beside solids stays within it for values down to 1/64 of
// the window's largest on the finest level, 1/16 on a coarse one: a float64
// iteration on a smooth two-phase design with that void takes 61 us at 64^2 (57
// without the check) and 107 at 256^2 (104); with 36 on the coarse levels too 58 and
// 104, and on late designs of an optimiser's loop 184 / 421 at 512^2 / 1024^2 against
// 204 / 478.
// Float64 subnormals have no exponent of their own: next to values above 2^-986
// they may be lost.
constexpr int FX_SPAN_FINE = 36, FX_SPAN_COARSE = 34;
__host__ __device__ __forceinline__ bool fx_beyond(int Q, int q, int span) { return Q - q > span; }
constexpr int FX_NEVER = -(1 << 20);  // a weight that no scales hold

// A fine element: its three factors (p, c, g of mto_fsweep.cuh) as integers
// below 2^61, factor = c 2^(X - 1083); all of one sign (that of the modulus).
constexpr int FX_NFINE = 3;
__host__ __device__ __forceinline__ void fx_encode_fine(double p, double c, double g, unsigned long long* w) {
  const double f[FX_NFINE] = {p, c, g};
  const int X = fx_common_exponent(f, FX_NFINE);
  for (int i = 0; i < FX_NFINE; ++i) w[i] = X < 0x7ff ? fx_coef_word(f[i], X, 8) : 0ull;
  fx_put_tag(w, (unsigned)X | (bits_of(p) >> 63 ? FX_TAG_NEG : 0u));
}

// A coarse element: six factors (FxCoarse below) as magnitudes below 2^59 with
// the sign in bit 63, factor = c 2^(X - 1081).
constexpr int FX_NCOARSE = 6;
enum FxCoarse { FXC_M00 = 0, FXC_M10, FXC_M01, FXC_C3C3, FXC_D3D3, FXC_C3D3 };
__host__ __device__ __forceinline__ void fx_encode_coarse(const double* f, unsigned long long* w) {
  const int X = fx_common_exponent(f, FX_NCOARSE);
  for (int i = 0; i < FX_NCOARSE; ++i)
    w[i] = X < 0x7ff ? fx_coef_word(f[i], X, 6) | (bits_of(f[i]) & 0x8000000000000000ull) : 0ull;
  fx_put_tag(w, (unsigned)X | (f[FXC_M00] < 0.0 || f[FXC_C3C3] < 0.0 || f[FXC_D3D3] < 0.0 ? FX_TAG_NEG : 0u));
}

}  // namespace mto
