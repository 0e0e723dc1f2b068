// Host-side check of the 96-bit fixed-point arithmetic (mto_fixed.cuh)
// against 128-bit integers (compiled by nvcc as host code).  Prints
// "ok <count>" or the first mismatch and exits non-zero.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

#include "mto_fixed.cuh"

using namespace mto;
typedef __int128 i128;

static uint64_t state = 0x9E3779B97F4A7C15ull;
static uint64_t next_u64() {  // xorshift64*
  state ^= state >> 12;
  state ^= state << 25;
  state ^= state >> 27;
  return state * 0x2545F4914F6CDD1Dull;
}
static double make(uint64_t sign, int e, uint64_t m) {
  return double_of((sign << 63) | ((uint64_t)e << 52) | (m & 0xfffffffffffffull));
}
// Random 96-bit value of 1..bits significant bits.
static Fx random_fx(int bits) {
  i128 v = ((i128)(int64_t)next_u64() << 64) | next_u64();
  v >>= 128 - 1 - (int)(next_u64() % bits);
  return fx_narrow(v);
}
static int fail(const char* what, long long n) {
  std::printf("%s mismatch at case %lld\n", what, n);
  return 1;
}

int main() {
  long long n = 0;
  for (int t = 0; t < 1000000; ++t, ++n) {
    // Sums, differences, shifts.
    const Fx a = random_fx(94), b = random_fx(94);
    if (fx_wide(fx_add(a, b)) != fx_wide(a) + fx_wide(b)) return fail("add", n);
    if (fx_wide(fx_sub(a, b)) != fx_wide(a) - fx_wide(b)) return fail("sub", n);
    const int s = (int)(next_u64() % 130);
    if (fx_wide(fx_sar(a, s)) != (fx_wide(a) >> (s > 127 ? 127 : s))) return fail("shift", n);

    // float64 at a common scale: exact down to 38 binary places below it.
    const int B = 1 + (int)(next_u64() % 2046);
    const int e = B - (int)(next_u64() % (t % 2 ? 39 : 120));
    const double v = make(next_u64() & 1, e < 0 ? 0 : e, next_u64());
    const int ev = fx_exponent((unsigned)(bits_of(v) >> 32)), sh = B - (ev ? ev : 1);
    const Fx f = fx_sar(fx_significand<false>(bits_of(v)), sh);
    if (B > FX_FLUSH_B && fx_wide(fx_sar(fx_significand<true>(bits_of(v)), sh)) != (ev ? fx_wide(f) : 0))
      return fail("flushed", n);
    i128 m = (i128)(bits_of(v) & 0xfffffffffffffull) | (ev ? (i128)1 << 52 : 0);
    m = (v < 0 ? -m : m) << 38;
    if (fx_wide(f) != (m >> (sh > 127 ? 127 : sh))) return fail("from double", n);
    if (sh <= 38 && B > 60 && fx_to_double(f, B - 1113) != v) return fail("round trip", n);

    // Products keep the upper 96 bits, up to 2 units low.
    const Fx w = random_fx(95);
    const uint64_t c = next_u64() >> (3 + next_u64() % 61);
    const i128 W = fx_wide(w), wh = W >> 48, wl = W & (((i128)1 << 48) - 1);
    const i128 exact = (wh * c + ((wl * c) >> 48)) >> 16;
    const i128 d = exact - fx_wide(fx_mul(w, c));
    if (d < 0 || d > 2) return fail("product", n);

    // Back to float64: within half a unit in the last place (ties either way).
    const Fx r = random_fx(96);
    if (fx_to_double<false>(r, FX_UNIT_MAX) != fx_to_double(r, FX_UNIT_MAX) ||
        fx_to_double<false>(r, FX_UNIT_MIN) != fx_to_double(r, FX_UNIT_MIN))
      return fail("unchecked", n);
    const i128 R = fx_wide(r);
    const double got = fx_to_double(r, 0), want = (double)R;
    if (got != want) {
      const double up = std::nextafter(want, INFINITY), dn = std::nextafter(want, -INFINITY);
      const i128 dg = R - (i128)got, dw = R - (i128)want;
      const i128 ag = dg < 0 ? -dg : dg, aw = dw < 0 ? -dw : dw;
      if ((got != up && got != dn) || ag - aw > (aw >> 9)) return fail("to double", n);
    }
    const int u = -1100 + (int)(next_u64() % 2000);
    const double far = fx_to_double(r, u), ref = std::ldexp(want, u);
    if (!(std::fabs(far - ref) <= std::fabs(ref) * 2.3e-16 + 5e-324) && far != ref) return fail("scaled", n);
    if (fx_to_double(fx_zero(), u) != 0.0) return fail("zero", n);

    // Element factors: the doubles come back from words and exponent.
    const int ee = 1 + (int)(next_u64() % 2046);
    const double p = make(t & 1, ee, next_u64());
    const double k[3] = {p, p * 0.45, p * 0.69};
    unsigned long long q[FX_NCOARSE];
    fx_encode_fine(k[0], k[1], k[2], q);
    unsigned tag = fx_tag(q);
    if ((tag >> 11) != (unsigned)(t & 1)) return fail("factor sign", n);
    for (int i = 0; i < FX_NFINE; ++i) {
      if (q[i] >> 61) return fail("factor range", n);
      const double back = std::ldexp((double)(q[i] & ~15ull), (int)(tag & 0x7ff) - 1083);
      if (std::fabs(back - std::fabs(k[i])) > std::fabs(p) * 1.2e-16) return fail("factor", n);
    }
    const double c6[FX_NCOARSE] = {p, p * 0.01, -p * 0.02, p * 0.3, p * 0.31, (t & 2) ? -p * 1e-3 : p * 1e-3};
    fx_encode_coarse(c6, q);
    tag = fx_tag(q);
    if ((tag >> 11) != (unsigned)(t & 1)) return fail("coarse factor sign", n);
    for (int i = 0; i < FX_NCOARSE; ++i) {
      const unsigned long long mag = q[i] & ~(1ull << 63);
      if (mag >> 59) return fail("coarse factor range", n);
      double back = std::ldexp((double)(mag & ~15ull), (int)(tag & 0x7ff) - 1081);
      if (q[i] >> 63) back = -back;
      if (std::fabs(back - c6[i]) > std::fabs(p) * 1.2e-16) return fail("coarse factor", n);
    }
    // Reciprocal: within an ulp.
    const double rd = make(0, 30 + (int)(next_u64() % 1980), t % 5 ? next_u64() : (t % 3 ? 0 : ~0ull));
    const double rq = fx_reciprocal(rd), rw = 1.0 / rd;
    if (rq != rw && rq != std::nextafter(rw, INFINITY) && rq != std::nextafter(rw, 0.0)) return fail("reciprocal", n);
    if (fx_wide(fx_flip(a, -1)) != -fx_wide(a) || fx_wide(fx_flip(a, 0)) != fx_wide(a)) return fail("flip", n);
  }
  unsigned long long z[FX_NCOARSE];
  fx_encode_fine(0.0, 0.0, 0.0, z);
  if (z[0] || z[1] || z[2]) return fail("zero factor", n);
  fx_encode_fine(NAN, NAN, NAN, z);
  if ((fx_tag(z) & 0x7ff) != 0x7ff) return fail("nan factor", n);
  fx_encode_fine(INFINITY, 1.0, 1.0, z);
  if ((fx_tag(z) & 0x7ff) != 0x7ff) return fail("inf factor", n);
  std::printf("ok %lld\n", n);
  return 0;
}
