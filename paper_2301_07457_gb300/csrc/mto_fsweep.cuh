// Sweeps of the float64 levels with the element operator in 96-bit fixed
// point (mto_fixed.cuh): marching, and a row per warp on small grids.
//
// Same strips, chunks, modes and edge-force bookkeeping as mto_sweep.cuh, one
// node column per lane.  The marched vector, its update (p = z + beta p_old,
// v + P z_c, ...) and the node row's result (q, the smoothed z, the residual)
// are float64; between them every difference, product and sum of the element
// operator is an integer.  The core is evaluated on sums and differences of
// c1 and d2: with A[c1,c1] = A[d2,d2] = kA, A[c1,d2] = kB = nu kA and
// A[s,s] = kG = (kA - kB) / 2,
//   t_c1 = P + G, t_d2 = P - G,  P = (kA + kB)/2 E (c1 + d2),  G = kG E (c1 - d2),
// which takes five products of three factors per element instead of seven of
// four (24 bytes of element data instead of 32).
//
// Measured at 2048^2: K p 0.318 -> 0.115 ms (bound before by the FP64 pipe at
// 36 operations per node; now the ALU pipe is busy 67% of the time, instruction
// issue 63%, the FP64 pipe 43% with the 6 operations of the CG recurrence, DRAM
// 3.5 TB/s: 16 warps of 128 registers per SM do not fill any of them), the
// operator alone 0.325 -> 0.108 ms, relative error against exact arithmetic
// 2.3e-16 -> 1.8e-16.  With the coarse levels in fixed point too, a float64
// 4096^2 step takes 128 instead of 362 ms, a mixed 2048^2 step 13.1 instead of
// 21.7 ms.
//
// Bounds (mto_fixed.cuh; |F| < 2^91): edge differences < 2^92, c1, c3, c2, d1,
// d2, d3 < 2^93, s and c1 +- d2 < 2^94; factors < 2^61, so every product
// (>> 64) is < 2^91, a node sums at most 14 of them: |K v| < 2^95.
//
// Scales are uniform over the warp.  A row whose largest exponent is above B
// (or an element above Xm) raises it and shifts the carried state; this
// happens in the first rows of a task and hardly ever after.
//
// Where an element's terms lie too far below the scales (fx_beyond in
// mto_fixed.cuh) the task is done again in float64 (rows_f64).  The
// fixed-point loop only keeps the smallest weight of its elements, four or five
// integer instructions a row, and compares it with the scales at its end: a vote
// and a call in every row took K p at 2048^2 from 113 to 119 us, an early exit
// from the loop to 117, this to 115.  A non-finite nodal value or modulus takes
// the task to float64 too, and so reaches the nodes next to it alone.  With a
// void of 1e-9 the sweeps of a random or a smooth design do not get there, on an
// optimised one a task in a thousand of the first sweep of a cycle and of its
// residual does (w/D b spans more than a vector of the iteration); with a void of
// 1e-12 in half of a smooth design an iteration takes 141 instead of 104 us at
// 256^2 and 420 instead of 371 us at 1024^2 (278 and 992 us where all was in float64), and
// with factors some 2^-60 apart everywhere the operator at 2048^2 takes 407 us and a
// V-cycle 2.61 ms (318 us and 2.41 ms).
#pragma once

#include "mto_fixed.cuh"
#include "mto_sweep.cuh"

namespace mto {

struct Fx2 {
  Fx x, y;
};
__device__ __forceinline__ Fx2 fadd(const Fx2& a, const Fx2& b) { return {fx_add(a.x, b.x), fx_add(a.y, b.y)}; }
__device__ __forceinline__ Fx2 fsub(const Fx2& a, const Fx2& b) { return {fx_sub(a.x, b.x), fx_sub(a.y, b.y)}; }
__device__ __forceinline__ Fx2 fsar(const Fx2& a, int s) { return {fx_sar(a.x, s), fx_sar(a.y, s)}; }
__device__ __forceinline__ Fx fshfl_down(const Fx& a) {
  return {__shfl_down_sync(0xffffffffu, a.lo, 1), __shfl_down_sync(0xffffffffu, a.mid, 1),
          __shfl_down_sync(0xffffffffu, a.hi, 1)};
}
__device__ __forceinline__ Fx fshfl_up(const Fx& a) {
  return {__shfl_up_sync(0xffffffffu, a.lo, 1), __shfl_up_sync(0xffffffffu, a.mid, 1),
          __shfl_up_sync(0xffffffffu, a.hi, 1)};
}
__device__ __forceinline__ Fx2 fshfl_down(const Fx2& a) { return {fshfl_down(a.x), fshfl_down(a.y)}; }
__device__ __forceinline__ Fx2 fshfl_up(const Fx2& a) { return {fshfl_up(a.x), fshfl_up(a.y)}; }

// A finite pair of nodal values at scale B (all lanes of the warp together).
// Zeros take no shift, so that ghost and clamped nodes cost nothing extra.
__device__ __forceinline__ Fx2 fx2_from(const double2& v, int B) {
  const int ex = fx_exponent((unsigned)__double2hiint(v.x)), ey = fx_exponent((unsigned)__double2hiint(v.y));
  if (B <= FX_FLUSH_B)  // uniform over the warp: values near the subnormal range
    return {fx_sar(fx_significand<false>(bits_of(v.x)), B - max(ex, 1)),
            fx_sar(fx_significand<false>(bits_of(v.y)), B - max(ey, 1))};
  const int sx = ex ? B - ex : 0, sy = ey ? B - ey : 0;
  Fx2 r = {fx_significand<true>(bits_of(v.x)), fx_significand<true>(bits_of(v.y))};
  if (__any_sync(0xffffffffu, (sx | sy) >= 32)) {
    r.x = fx_sar_limbs(r.x, sx);
    r.y = fx_sar_limbs(r.y, sy);
  }
  return {fx_sar31(r.x, sx & 31), fx_sar31(r.y, sy & 31)};
}

// Strain-space forces of an element.
struct FxStrain {
  Fx c1, c3, d2, d3, s;
};

// The element operator of a source.  load(): the element's words.  core(): the
// forces t of the strains w (same basis), at the element's own scale; neg: a
// factor may be negative that is positive for every positive modulus.
template <int SRC> struct FxElem;
template <> struct FxElem<SRC_FINE64> {
  static constexpr int N = FX_NFINE, UNIT = -2132, SPAN = FX_SPAN_FINE;
  __device__ __forceinline__ static FxStrain core(const SweepParams<double>&, FxStrain w, const unsigned long long* k,
                                                  bool neg) {
    if (neg && (fx_tag(k) & FX_TAG_NEG))
      w = {fx_neg(w.c1), fx_neg(w.c3), fx_neg(w.d2), fx_neg(w.d3), fx_neg(w.s)};
    const Fx p = fx_mul(fx_add(w.c1, w.d2), k[0]), g = fx_mul(fx_sub(w.c1, w.d2), k[2]);
    return {fx_add(p, g), fx_mul(w.c3, k[1]), fx_sub(p, g), fx_mul(w.d3, k[1]), fx_mul(w.s, k[2])};
  }
  // The same in float64.
  __device__ __forceinline__ static Strain<double> core64(const SweepParams<double>&, const Strain<double>& w,
                                                          const unsigned long long* k) {
    const unsigned tag = fx_tag(k);
    const bool neg = tag & FX_TAG_NEG;
    const double P = fx_factor(k[0], neg, tag, 1083), C = fx_factor(k[1], neg, tag, 1083),
                 G = fx_factor(k[2], neg, tag, 1083);
    const double p = P * (w.c1 + w.d2), g = G * (w.c1 - w.d2);
    return {p + g, C * w.c3, p - g, C * w.d3, G * w.s};
  }
};
template <> struct FxElem<SRC_COARSE> {
  static constexpr int N = FX_NCOARSE, UNIT = -2130, SPAN = FX_SPAN_COARSE;
  __device__ __forceinline__ static FxStrain core(const SweepParams<double>& a, FxStrain w,
                                                  const unsigned long long* k, bool neg) {
    constexpr unsigned long long MAG = 0x7fffffffffffffffull;
    const unsigned long long m0 = k[FXC_M00] & MAG, m1 = k[FXC_M10] & MAG, m2 = k[FXC_M01] & MAG,
                             kc = k[FXC_C3C3] & MAG, kd = k[FXC_D3D3] & MAG, k9 = k[FXC_C3D3] & MAG;
    // g times the moments (g = (1 - nu) / 2 = gfix 2^-64, nu = 1 - 2 g).
    const unsigned long long g0 = __umul64hi(m0, a.gfix), g1 = __umul64hi(m1, a.gfix), g2 = __umul64hi(m2, a.gfix);
    const auto mask = [&](int i) -> int { return (int)(k[i] >> 32) >> 31; };
    const int s1 = mask(FXC_M10), s2 = mask(FXC_M01), s12 = s1 ^ s2, s9 = mask(FXC_C3D3) ^ s12;
    const Fx c3 = fx_flip(w.c3, s2), d3 = fx_flip(w.d3, s1), s = fx_flip(w.s, s12);
    const Fx sum = fx_add(w.c1, w.d2);
    Fx p = fx_mul(sum, m0 - g0), m = fx_mul(fx_sub(w.c1, w.d2), g0), tc = fx_mul(c3, kc), td = fx_mul(d3, kd),
       ts = fx_mul(s, g0);
    if (neg) {
      const int n0 = mask(FXC_M00);
      p = fx_flip(p, n0);
      m = fx_flip(m, n0);
      ts = fx_flip(ts, n0);
      tc = fx_flip(tc, mask(FXC_C3C3));
      td = fx_flip(td, mask(FXC_D3D3));
    }
    FxStrain t;
    {
      const Fx x2 = fx_mul(c3, m2), x1 = fx_mul(d3, m1), both = fx_add(x1, x2);
      const Fx y2 = fx_mul(c3, g2), y1 = fx_mul(d3, g1);
      t.c1 = fx_sub(fx_sub(fx_add(fx_add(p, m), both), y1), y1);
      t.d2 = fx_sub(fx_sub(fx_add(fx_sub(p, m), both), y2), y2);
    }
    {
      const Fx x = fx_mul(sum, m2), y = fx_mul(w.d2, g2);
      tc = fx_add(tc, fx_sub(fx_sub(x, y), y));
      tc = fx_add(tc, fx_mul(s, g1));
      t.c3 = fx_flip(fx_add(tc, fx_flip(fx_mul(d3, k9), s9)), s2);
    }
    {
      const Fx x = fx_mul(sum, m1), y = fx_mul(w.c1, g1);
      td = fx_add(td, fx_sub(fx_sub(x, y), y));
      td = fx_add(td, fx_mul(s, g2));
      t.d3 = fx_flip(fx_add(td, fx_flip(fx_mul(c3, k9), s9)), s1);
    }
    t.s = fx_flip(fx_add(ts, fx_add(fx_mul(c3, g1), fx_mul(d3, g2))), s12);
    return t;
  }
  // The same in float64.
  __device__ __forceinline__ static Strain<double> core64(const SweepParams<double>& a, const Strain<double>& w,
                                                          const unsigned long long* k) {
    const unsigned tag = fx_tag(k);
    double f[FX_NCOARSE];
#pragma unroll
    for (int n = 0; n < FX_NCOARSE; ++n) f[n] = fx_factor(k[n] & 0x7fffffffffffffffull, k[n] >> 63, tag, 1081);
    const double g = ldexp((double)a.gfix, -64), nu = 1.0 - 2.0 * g;
    const double m0 = f[FXC_M00], m1 = f[FXC_M10], m2 = f[FXC_M01], k9 = f[FXC_C3D3];
    Strain<double> t;
    t.c1 = m0 * (w.c1 + nu * w.d2) + (m2 * w.c3 + nu * (m1 * w.d3));
    t.d2 = m0 * (w.d2 + nu * w.c1) + (m1 * w.d3 + nu * (m2 * w.c3));
    t.c3 = f[FXC_C3C3] * w.c3 + m2 * (w.c1 + nu * w.d2) + (k9 * w.d3 + g * (m1 * w.s));
    t.d3 = f[FXC_D3D3] * w.d3 + m1 * (w.d2 + nu * w.c1) + (k9 * w.c3 + g * (m2 * w.s));
    t.s = g * (m0 * w.s + (m1 * w.c3 + m2 * w.d3));
    return t;
  }
};

// A warp's columns: lane `lane` has column i; rows from je0, coarse rows Jb .. Je
// of a restriction.
struct FTask {
  int i, lane, je0, Jb, Je;
  bool own_col;
};
// What a task sums: dot products, the coarse row in progress (RESTRICT).
struct FSums {
  double dot0, dot1;
  double2 racc;
};

template <int SRC, int MODE, bool DOT, typename ZT> struct FSweep {
  using S = Sweep<double, SRC, MODE, DOT, ZT>;
  using Elem = FxElem<SRC>;
  static constexpr bool SMOOTHING = S::SMOOTHING;
  // SMOOTH0 carries the right-hand side and w/D of its top row to the step
  // that completes it.
  static constexpr bool LOADS_B = S::NEEDS_B && MODE != MODE_SMOOTH0;
  static constexpr bool LOADS_D = SMOOTHING && MODE != MODE_SMOOTH0;

  // Loads of one step: node row je + 1, element row je, node row je.
  struct Pack {
    double2 v;
    ZT z;             // KP: z; RESID: the direction of a pending x step
    double2 c0, c1;   // PSMOOTH: coarse nodes (I, J), (I, J + 1)
    double2 dt;       // SMOOTH0: w/D of the top row
    unsigned long long k[Elem::N];
    double2 b;        // node row je (KP: of the top row, the iterate x to be advanced)
    double2 d;
    double2 rd, qd;
  };

  __device__ __forceinline__ static double2 load_d(const SweepParams<double>& a, long long k) {
    if constexpr (SRC == SRC_FINE64) {
      const double d = a.invd1[k];
      return make_double2(d, d);
    } else {
      return a.invd2[k];
    }
  }
  __device__ __forceinline__ static void load_top(const SweepParams<double>& a, long long k, int i, int jj,
                                                  bool lag, Pack& r) {
    if constexpr (MODE == MODE_KP) {
      r.z = static_cast<const ZT*>(a.zkp)[k];
      r.v = a.v[k];
      if (lag) r.b = a.xvec[k];
    } else if constexpr (MODE == MODE_PSMOOTH) {
      r.v = a.v[k];
      // Column i lies on coarse column I = i / 2 or halfway to I + 1 (the next
      // lane's), row jj on coarse row jj / 2 or halfway to the next.
      const long long kc = a.gc.at(max(i, 0) >> 1, max(jj, 0) >> 1);
      r.c0 = a.zc[kc];
      r.c1 = a.zc[kc + ((jj & 1) ? a.gc.pitch : 0)];
    } else if constexpr (MODE == MODE_SMOOTH0) {
      r.v = a.b[k];
      r.dt = load_d(a, k);
    } else if constexpr (MODE == MODE_RESID) {
      r.v = a.v[k];
      if (lag) r.z = a.xdir[k];
    } else if constexpr (MODE == MODE_APPLY) {
      if (a.dense) {  // the caller's vector: clamped nodes are read as zero, ghosts do not exist
        r.v = make_double2(0.0, 0.0);
        if (a.g.active(i, jj)) r.v = a.v[(long long)jj * (a.g.nx + 1) + i];
      } else {
        r.v = a.v[k];
      }
    } else {
      r.v = a.v[k];
    }
  }
  __device__ __forceinline__ static void load(const SweepParams<double>& a, long long k, int i, int je,
                                              bool lag, Pack& r) {
    load_top(a, k + a.g.pitch, i, je + 1, lag, r);
    const unsigned long long* E = static_cast<const unsigned long long*>(a.E) + k;
#pragma unroll
    for (int n = 0; n < Elem::N; ++n) r.k[n] = __ldg(E + n * a.cstride);
    if constexpr (LOADS_B) r.b = a.b[k];
    if constexpr (LOADS_D) r.d = load_d(a, k);
    if constexpr (DOT) {
      r.rd = a.rdot[k];
      if (a.qdot != nullptr) r.qd = a.qdot[k];
    }
  }

  // Marched value of node (i, jj).
  __device__ __forceinline__ static double2 value(const SweepParams<double>& a, const Pack& r, int i, int jj,
                                                  double beta, bool lag, double alag) {
    if constexpr (MODE == MODE_KP) {
      return make_double2(fma(beta, r.v.x, to_f64(r.z.x)), fma(beta, r.v.y, to_f64(r.z.y)));
    } else if constexpr (MODE == MODE_PSMOOTH) {
      // v + w (t + t of column I + 1 where i is odd, else t again), with
      // t = c0 or c0 + c1: two or three FP64 operations per component.
      double2 t = r.c0;
      double w = 0.5;
      if (jj & 1) {  // uniform over the warp
        t = make_double2(r.c0.x + r.c1.x, r.c0.y + r.c1.y);
        w = 0.25;
      }
      const double2 tr = shfl_down2(t);  // lane 31: its own value, used only for halo output
      const bool odd = i & 1;
      const double2 s = make_double2(t.x + (odd ? tr.x : t.x), t.y + (odd ? tr.y : t.y));
      return a.g.valid(i, jj) ? make_double2(fma(w, s.x, r.v.x), fma(w, s.y, r.v.y)) : make_double2(0.0, 0.0);
    } else if constexpr (MODE == MODE_SMOOTH0) {
      return make_double2(r.dt.x * r.v.x, r.dt.y * r.v.y);  // w/D is zero on clamped and ghost nodes
    } else if constexpr (MODE == MODE_RESID) {
      if (lag) return make_double2(fma(alag, r.z.x, r.v.x), fma(alag, r.z.y, r.v.y));
      return r.v;
    } else {
      return r.v;
    }
  }

  // What a mode does with K v of node (i, je); k: its offset, v: its marched
  // value, b, d: its right-hand side and w/D (all lanes of the warp).
  __device__ __forceinline__ static void finish_row(const SweepParams<double>& a, const FTask& t, long long k, int je,
                                                    bool inb, bool act, const double2& v, const double2& kv,
                                                    const double2& b, const double2& d, const Pack& cur,
                                                    FSums& sums) {
    const double2 zero2 = make_double2(0.0, 0.0);
    if constexpr (MODE == MODE_APPLY) {
      if (inb) a.out[a.dense ? (long long)je * (a.g.nx + 1) + t.i : k] = act ? kv : zero2;
    } else if constexpr (MODE == MODE_RESID) {
      double2 r = zero2;
      if (act) r = sub2(b, kv);
      if (inb) a.out[k] = r;
      if (inb && a.out32 != nullptr) a.out32[k] = make_float2(float(r.x), float(r.y));
      sums.dot0 = fma(r.x, r.x, fma(r.y, r.y, sums.dot0));
    } else if constexpr (MODE == MODE_KP) {
      const double2 q = act ? kv : zero2;
      if (inb) {
        a.p_out[k] = v;
        a.out[k] = q;
        sums.dot0 = fma(v.x, q.x, fma(v.y, q.y, sums.dot0));
      }
    } else if constexpr (SMOOTHING) {
      double2 zn = zero2;
      if (act) zn = make_double2(fma(d.x, b.x - kv.x, v.x), fma(d.y, b.y - kv.y, v.y));
      if (inb) a.out[k] = zn;
      if constexpr (DOT) {
        if (act) {
          sums.dot0 = fma(zn.x, cur.rd.x, fma(zn.y, cur.rd.y, sums.dot0));
          if (a.qdot != nullptr) sums.dot1 = fma(zn.x, cur.qd.x, fma(zn.y, cur.qd.y, sums.dot1));
        }
      }
    } else if constexpr (MODE == MODE_RESTRICT) {
      double2 r = zero2;
      if (act) r = sub2(b, kv);
      // Full weighting, vertically along the march (1/2, 1, 1/2 over fine
      // rows 2J - 1, 2J, 2J + 1), then horizontally once per coarse row.
      if (je > t.je0) {
        if (je & 1) {
          const int Jlo = (je - 1) / 2;
          const double2 col = make_double2(fma(0.5, r.x, sums.racc.x), fma(0.5, r.y, sums.racc.y));
          const double2 cu = shfl_up2(col), cd = shfl_down2(col);
          const double2 val = make_double2(fma(0.5, cu.x + cd.x, col.x), fma(0.5, cu.y + cd.y, col.y));
          const bool producer = (t.lane & 1) == 0 && t.lane >= 2 && t.lane <= 28;
          const int I = t.i >> 1;
          if (producer && Jlo >= t.Jb && Jlo <= t.Je && I >= 0 && I <= a.gc.nx)
            a.bc[a.gc.at(I, Jlo)] = a.gc.is_fixed(I, Jlo) ? zero2 : val;
          sums.racc = make_double2(0.5 * r.x, 0.5 * r.y);
        } else {
          sums.racc = add2(sums.racc, r);
        }
      }
    }
  }
};

// Rows je0 + 1 .. je1 of a warp's columns in float64 (all lanes of the warp):
// the marching sweep with the element operator on the FP64 pipe, at about three
// times the cost.  x has had its pending step (KP).  Without FINISH nothing is
// written and racc is K v of the last row.  A call of its own, so that its
// registers do not weigh on the kernels.
template <int SRC, int MODE, bool DOT, typename ZT, bool FINISH>
__device__ __noinline__ FSums rows_f64(const SweepParams<double>& a, FTask t0, int je1, double beta, bool lag,
                                       double alag) {
  using F = FSweep<SRC, MODE, DOT, ZT>;
  const Grid& g = a.g;
  const double2 zero2 = make_double2(0.0, 0.0);
  const int je0 = t0.je0;
  FSums sums = {0.0, 0.0, zero2};
  long long k = g.at(t0.i, je0);
  typename F::Pack cur;
  F::load_top(a, k, t0.i, je0, lag, cur);
  double2 vb = F::value(a, cur, t0.i, je0, beta, lag, alag), gbp = zero2, gsp = zero2, bc = zero2, dc = zero2, kv = zero2;
  if constexpr (MODE == MODE_SMOOTH0) {
    bc = cur.v;
    dc = cur.dt;
  }
#pragma unroll 1
  for (int je = je0; je <= je1; ++je, k += g.pitch) {
    F::load(a, k, t0.i, je, lag, cur);
    const double2 vt = F::value(a, cur, t0.i, je + 1, beta, lag, alag);
    const double2 ac = sub2(shfl_down2(vb), vb), bt = sub2(shfl_down2(vt), vt), dl = sub2(vt, vb);
    const double2 up = add2(dl, shfl_down2(dl));
    Strain<double> w;
    w.c1 = ac.x + bt.x;
    w.c3 = bt.x - ac.x;
    w.d2 = up.y;
    w.d3 = bt.y - ac.y;
    w.s = up.x + (ac.y + bt.y);
    const Strain<double> t = F::Elem::core64(a, w, cur.k);
    // Edge forces and node row je, as in the fixed-point loop.
    const double2 gh = add2(make_double2(t.c1 - t.c3, t.s - t.d3), gbp), gd = sub2(gsp, make_double2(t.s, t.d2));
    kv = add2(shfl_up2(add2(gd, gh)), sub2(gd, gh));
    if constexpr (FINISH) {
      const bool inb = je > je0 && t0.own_col && je >= 0 && je <= g.ny;
      const bool act = inb && !g.is_fixed(t0.i, je);
      const double2 b = MODE == MODE_SMOOTH0 ? bc : cur.b, d = MODE == MODE_SMOOTH0 ? dc : cur.d;
      F::finish_row(a, t0, k, je, inb, act, vb, kv, b, d, cur, sums);
    }
    gbp = make_double2(t.c1 + t.c3, t.s + t.d3);
    gsp = make_double2(t.s, t.d2);
    vb = vt;
    if constexpr (MODE == MODE_SMOOTH0) {
      bc = cur.v;
      dc = cur.dt;
    }
  }
  if constexpr (!FINISH) sums.racc = kv;
  return sums;
}

// The restriction's tasks of a block that are to be done again in float64
// (`lost`: this warp's is), their rows by all its warps: a row takes one warp about
// a microsecond of its FP64 pipe, and on an optimised design one or two tasks of
// a launch are waited for (a float64 iteration at 1024^2 433 -> 422 us, with
// FX_SPAN_COARSE at 36).  In the
// other sweeps the barrier at the end costs what this gains.
template <int SRC, bool DOT, typename ZT>
__device__ __noinline__ void restrict_f64(const SweepParams<double>& a, bool lost) {
  __shared__ unsigned mask;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  if (threadIdx.x == 0) mask = 0;
  __syncthreads();
  if (lost && lane == 0) atomicOr(&mask, 1u << warp);
  __syncthreads();
  // Each lost task is shared by `parts` warps, this warp has part `part` of the
  // one that is `mine`.
  unsigned m = mask;
  const int parts = nwarps / __popc(m), mine = warp / parts, part = warp % parts;
  for (int q = 0; q < mine; ++q) m &= m - 1;
  if (m == 0u) return;
  const int wg = blockIdx.x * nwarps + __ffs((int)m) - 1, strip = wg % a.nstrips, chunk = wg / a.nstrips;
  const int Jb = chunk * (a.H >> 1), n = min(a.H >> 1, a.gc.ny + 1 - Jb), per = (n + parts - 1) / parts;
  const int i = strip * SWEEP_RSTRIDE - 2 + lane, J0 = Jb + part * per, J1 = min(Jb + n, J0 + per) - 1;
  if (J0 > J1) return;
  const FTask t = {i, lane, max(2 * J0 - 2, -1), J0, J1, lane >= 1 && lane <= 30 && i >= 0 && i <= a.g.nx};
  rows_f64<SRC, MODE_RESTRICT, DOT, ZT, true>(a, t, 2 * J1 + 1, 0.0, false, 0.0);
}

// Two resident blocks per SM, as sweep2_kernel.
template <int SRC, int MODE, bool DOT, typename ZT, int PF>
__global__ void __launch_bounds__(SWEEP_NT, 2) fsweep_kernel(const __grid_constant__ SweepParams<double> a) {
  using F = FSweep<SRC, MODE, DOT, ZT>;
  using Pack = typename F::Pack;
  constexpr bool REDUCE = DOT || MODE == MODE_RESID || MODE == MODE_KP;
  pdl_wait();
  if (a.sc != nullptr && a.gate) {
    if (a.sc->done != RUNNING) return;  // uniform over the grid
    if (a.replace_gate && (a.sc->rr_every <= 0 || (a.sc->iter % a.sc->rr_every) != 0)) return;
  }
  const Grid g = a.g;
  const int lane = threadIdx.x & 31;
  const int wg = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int strip = wg % a.nstrips;
  const int chunk = wg / a.nstrips;
  const double2 zero2 = make_double2(0.0, 0.0);
  FSums sums = {0.0, 0.0, zero2};
  double beta = 0.0, alag = 0.0;
  bool vzero = false, lag = false, lost = false;
  if constexpr (MODE == MODE_KP) {
    beta = a.sc->beta;
    lag = a.sc->x_lag != 0;  // K p advances x by the pending step at its owned nodes
    alag = a.sc->alpha;
  }
  if constexpr (MODE == MODE_RESID) {
    vzero = a.zero_gate && a.sc->x_nonzero == 0;
    if (a.xlag && a.sc != nullptr && a.sc->x_lag != 0) {  // works on x + alpha p
      lag = true;
      alag = a.sc->alpha;
    }
  }

  if (vzero) {
    // Residual of a zero iterate: r = b on the free DOFs, no operator needed.
    const int i = strip * SWEEP_STRIDE - 1 + lane;
    if (chunk < a.nchunks && lane >= 1 && lane <= 30 && i >= 0 && i <= g.nx) {
      const int r0 = chunk * a.H, r1 = min(r0 + a.H - 1, g.ny);
      for (int j = r0; j <= r1; ++j) {
        const long long k = g.at(i, j);
        const double2 r = g.is_fixed(i, j) ? zero2 : a.b[k];
        a.out[k] = r;
        if (a.out32 != nullptr) a.out32[k] = make_float2(float(r.x), float(r.y));
        sums.dot0 = fma(r.x, r.x, fma(r.y, r.y, sums.dot0));
      }
    }
  } else if (chunk < a.nchunks) {
    constexpr int STRIDE = MODE == MODE_RESTRICT ? SWEEP_RSTRIDE : SWEEP_STRIDE;
    constexpr int SHIFT = MODE == MODE_RESTRICT ? 2 : 1;
    const int i = strip * STRIDE - SHIFT + lane;
    int je0, je1, Jb = 0, Je = 0;
    if constexpr (MODE == MODE_RESTRICT) {
      Jb = chunk * (a.H >> 1);
      Je = min(Jb + (a.H >> 1) - 1, a.gc.ny);
      je0 = max(2 * Jb - 2, -1);
      je1 = 2 * Je + 1;
    } else {
      const int r0 = chunk * a.H;
      je0 = r0 - 1;
      je1 = min(r0 + a.H - 1, g.ny);
    }
    const bool own_col = lane >= 1 && lane <= 30 && i >= 0 && i <= g.nx;
    const bool col_fixed = ((g.fixed & 2u) && i == 0) || ((g.fixed & 4u) && i == g.nx);
    const long long pitch = g.pitch;

    int B = 1, Xm = 0;             // scales of the nodal values and of the coefficients
    int eb = 0;                    // exponent of node (i, je)
    int low = 1 << 20;             // smallest weight of the column's elements
    const FTask t0 = {i, lane, je0, Jb, Je, own_col};
    // Carried from the row below: edge differences and sums (i + 1 minus / plus
    // i) of node row je, and the forces of element row je - 1 on its top and
    // left edges.
    Fx2 ac = {fx_zero(), fx_zero()}, sc = ac, gbp = ac, gsp = ac;
    // Marched values of a row at scale B, which the row raises if it has to;
    // e: the pair's larger exponent.
    auto to_fixed = [&](double2 v, int& e) -> Fx2 {
      e = max(fx_exponent((unsigned)__double2hiint(v.x)), fx_exponent((unsigned)__double2hiint(v.y)));
      if (__any_sync(0xffffffffu, e > B)) {
        const bool finite = e != 0x7ff;
        if (!finite) v = zero2;
        if (!__all_sync(0xffffffffu, finite)) low = FX_NEVER;
        const int Bn = (int)__reduce_max_sync(0xffffffffu, finite ? (unsigned)e : 0u);
        if (Bn > B) {
          ac = fsar(ac, Bn - B);
          sc = fsar(sc, Bn - B);
          gbp = fsar(gbp, Bn - B);
          gsp = fsar(gsp, Bn - B);
          B = Bn;
        }
      }
      return fx2_from(v, B);
    };

    const long long k0 = g.at(i, je0);
    double2 vbd;         // marched values of node row je in float64
    double2 bc = zero2;  // SMOOTH0: right-hand side and w/D of node row je
    double2 dc = zero2;
    {
      Pack r0;
      F::load_top(a, k0, i, je0, lag, r0);
      vbd = F::value(a, r0, i, je0, beta, lag, alag);
      const Fx2 vb = to_fixed(vbd, eb);
      const Fx2 vr = fshfl_down(vb);
      ac = fsub(vr, vb);
      sc = fadd(vr, vb);
      if constexpr (MODE == MODE_SMOOTH0) {
        bc = r0.v;
        dc = r0.dt;
      }
    }
    Pack ring[PF];
#pragma unroll
    for (int u = 0; u < PF; ++u)
      if (je0 + u <= je1) F::load(a, k0 + u * pitch, i, je0 + u, lag, ring[u]);

    long long k = k0;  // offset of node / element (i, je)
    for (int jb = je0; jb <= je1; jb += PF) {
#pragma unroll
      for (int u = 0; u < PF; ++u) {
        const int je = jb + u;
        if (je > je1) break;
        const Pack cur = ring[u];
        if (je + PF <= je1) F::load(a, k + PF * pitch, i, je + PF, lag, ring[u]);
        if constexpr (MODE == MODE_KP) {
          // Pending x step at the top row (owned rows only): x += alpha p_old.
          if (lag && je + 1 <= je1) {  // uniform over the warp
            if (own_col)
              a.xvec[k + pitch] = make_double2(fma(alag, cur.v.x, cur.b.x), fma(alag, cur.v.y, cur.b.y));
          }
        }
        // ---- element (i, je) from rows je (vb) and je + 1 (vt) ----
        const double2 vtd = F::value(a, cur, i, je + 1, beta, lag, alag);
        int et;
        const Fx2 vt = to_fixed(vtd, et);
        const Fx2 vr = fshfl_down(vt);  // lane 31: its own value, used only for halo output
        const Fx2 bt = fsub(vr, vt), st = fadd(vr, vt);
        const Fx2 up = fsub(st, sc);  // (c2, d2): left plus right edge
        const FxStrain w = {fx_add(ac.x, bt.x), fx_sub(bt.x, ac.x), up.y, fx_sub(bt.y, ac.y),
                            fx_add(up.x, fx_add(ac.y, bt.y))};
        // X above Xm, more than 31 below it, or an unexpected sign: one vote
        // for the three rare cases (ghost elements have tag 0).
        const unsigned tag = fx_tag(cur.k);
        const bool rare = __any_sync(0xffffffffu, tag != 0u && (unsigned)(Xm - (int)tag) >= 32u);
        const int X = (int)(tag & 0x7ffu);
        if (rare) {
          if (__any_sync(0xffffffffu, X == 0x7ff)) low = FX_NEVER;
          const int Xn = max(Xm, (int)__reduce_max_sync(0xffffffffu, X == 0x7ff ? 0u : (unsigned)X));
          gbp = fsar(gbp, Xn - Xm);
          gsp = fsar(gsp, Xn - Xm);
          Xm = Xn;
        }
        FxStrain t = F::Elem::core(a, w, cur.k, rare);
        const int sh = Xm - X;
        if (rare)
          t = {fx_sar_limbs(t.c1, sh), fx_sar_limbs(t.c3, sh), fx_sar_limbs(t.d2, sh), fx_sar_limbs(t.d3, sh),
               fx_sar_limbs(t.s, sh)};
        t = {fx_sar31(t.c1, sh & 31), fx_sar31(t.c3, sh & 31), fx_sar31(t.d2, sh & 31), fx_sar31(t.d3, sh & 31),
             fx_sar31(t.s, sh & 31)};
        // ---- edge forces and node row je ----
        const Fx2 gs = {t.s, t.d2};                                             // left and right edge of this element
        const Fx2 gb = {fx_add(t.c1, t.c3), fx_add(t.s, t.d3)};                 // its top edge
        const Fx2 gh = fadd(Fx2{fx_sub(t.c1, t.c3), fx_sub(t.s, t.d3)}, gbp);   // edge (i, je) -> (i + 1, je)
        // A node takes gh and the difference of the vertical forces from the
        // elements on its left (one shuffle for both) and on its right.
        const Fx2 gd = fsub(gsp, gs);
        const Fx2 kvf = fadd(fshfl_up(fadd(gd, gh)), fsub(gd, gh));
        const int unit = B + Xm + F::Elem::UNIT;
        double2 kv = make_double2(fx_to_double<false>(kvf.x, unit), fx_to_double<false>(kvf.y, unit));
        if (unit < FX_UNIT_MIN || unit > FX_UNIT_MAX)  // uniform over the warp
          kv = make_double2(fx_to_double(kvf.x, unit), fx_to_double(kvf.y, unit));

        // Weight of the element, where it is not zero on all corners (as most
        // are in the first cycle of a solve) and has material.
        const int ec = max(eb, et), e4 = max(ec, __shfl_down_sync(0xffffffffu, ec, 1));
        if (min(e4, X) != 0) low = min(low, e4 + X);
        eb = et;
        const bool inb = je > je0 && own_col && je >= 0 && je <= g.ny;
        const bool act = inb && !col_fixed && !(((g.fixed & 1u) && je == 0) || ((g.fixed & 8u) && je == g.ny));
        const double2 b = MODE == MODE_SMOOTH0 ? bc : cur.b, d = MODE == MODE_SMOOTH0 ? dc : cur.d;
        F::finish_row(a, t0, k, je, inb, act, vbd, kv, b, d, cur, sums);
        if constexpr (MODE == MODE_SMOOTH0) {
          bc = cur.v;
          dc = cur.dt;
        }
        ac = bt;
        gbp = gb;
        gsp = gs;
        sc = st;
        vbd = vtd;
        k += pitch;
      }
    }
    if constexpr (MODE == MODE_RESTRICT) {
      lost = __any_sync(0xffffffffu, lane <= 30 && fx_beyond(B + Xm, low, F::Elem::SPAN));
    } else {
      if (__any_sync(0xffffffffu, lane <= 30 && fx_beyond(B + Xm, low, F::Elem::SPAN)))
        sums = rows_f64<SRC, MODE, DOT, ZT, true>(a, t0, je1, beta, lag, alag);
    }
  }
  if constexpr (MODE == MODE_RESTRICT) {
    if (__syncthreads_or(lost)) restrict_f64<SRC, DOT, ZT>(a, lost);
  }
  if constexpr (REDUCE) {
    block_reduce_finish<SWEEP_NT, DOT>(sums.dot0, sums.dot1, a.partials, a.ticket, a.sc, a.finish, a.out_value, a.tag);
  }
}

// ---------------------------------------------------------------------------
// Small grids: one node row per warp, its two element rows side by side.
//
// Where a grid gives every warp one or two rows, a marching sweep is a chain
// of two or three element rows of about 600 instructions each, issued by one
// warp per scheduler at five clocks apiece: 3 us of a launch's 7, whatever the
// grid.  Here a warp completes one node row je of 14 columns: lanes 0-15
// evaluate the element row below it, lanes 16-31 the one above, both at once;
// the halves exchange their parts of K v, and the lower one finishes u_x, the
// upper one u_y.  The restriction uses a block of three warps for the three
// fine rows of a coarse row.  Element data and diagonals, which no kernel of
// the chain writes, are loaded before the wait for the previous kernel.
// ---------------------------------------------------------------------------
constexpr int SPLIT_STRIDE = 14;   // columns per warp
constexpr int SPLIT_RSTRIDE = 12;  // fine columns per warp of the restriction (6 coarse ones)
constexpr int SPLIT_RWARPS = 3;

// Resident blocks per SM that the fixed-point path's registers allow; rows_f64
// would take a few more (here and in the tiles together a float64 iteration at
// 256^2 99.1 -> 100.7 us, at 64^2, which does not fill the chip, 52.7 -> 52.3).
template <int SRC, int MODE, bool DOT> constexpr int split_blocks() {
  return SRC == SRC_COARSE ? 2 : (MODE == MODE_KP || DOT ? 3 : 4);
}

template <int SRC, int MODE, bool DOT, typename ZT>
__global__ void __launch_bounds__(SWEEP_NT, (split_blocks<SRC, MODE, DOT>()))
    fsplit_kernel(const __grid_constant__ SweepParams<double> a) {
  using F = FSweep<SRC, MODE, DOT, ZT>;
  using Pack = typename F::Pack;
  constexpr bool REDUCE = DOT || MODE == MODE_RESID || MODE == MODE_KP;
  constexpr bool RESTRICT = MODE == MODE_RESTRICT;
  pdl_trigger();
  const Grid g = a.g;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int half = lane >> 4, hl = lane & 15;
  // Task: a strip and a node row (restriction: a strip and a coarse row).
  const int wg = RESTRICT ? (int)blockIdx.x : blockIdx.x * (int)(blockDim.x >> 5) + warp;
  const int strip = wg % a.nstrips, row = wg / a.nstrips;
  const int i = strip * (RESTRICT ? SPLIT_RSTRIDE : SPLIT_STRIDE) - (RESTRICT ? 2 : 1) + hl;
  const int je = RESTRICT ? 2 * row - 1 + warp : row;
  const bool task = row < a.nchunks && je >= 0 && je <= g.ny;  // uniform over the warp
  const int jr = (task ? je : 0) - 1 + half;                   // this half's element row
  const long long ke = g.at(task ? i : 0, jr);                 // element (i, jr), node (i, jr)
  const long long kn = g.at(task ? i : 0, task ? je : 0);      // node (i, je)
  const int c = half;                                          // component this lane finishes
  const bool own = task && hl >= 1 && hl <= 14 && i >= 0 && i <= g.nx;
  const bool act = own && !g.is_fixed(i, je);

  Pack lo, hi;  // node rows jr and jr + 1
  {
    const unsigned long long* E = static_cast<const unsigned long long*>(a.E) + ke;
#pragma unroll
    for (int n = 0; n < F::Elem::N; ++n) lo.k[n] = __ldg(E + n * a.cstride);
  }
  double d = 0.0;
  if constexpr (F::SMOOTHING)
    d = SRC == SRC_FINE64 ? __ldg(a.invd1 + kn) : __ldg(reinterpret_cast<const double*>(a.invd2 + kn) + c);
  pdl_wait_prior();

  double beta = 0.0, alag = 0.0;
  bool lag = false, vzero = false, done = false;
  if (a.sc != nullptr) {
    if (a.gate) {
      done = a.sc->done != RUNNING;
      if (a.replace_gate) done = done || a.sc->rr_every <= 0 || (a.sc->iter % a.sc->rr_every) != 0;
    }
    if constexpr (MODE == MODE_KP) {
      beta = a.sc->beta;
      lag = a.sc->x_lag != 0;
      alag = a.sc->alpha;
    }
    if constexpr (MODE == MODE_RESID) {
      vzero = a.zero_gate && a.sc->x_nonzero == 0;
      lag = a.xlag && a.sc->x_lag != 0;
      alag = a.sc->alpha;
    }
  }
  // Without the pending step its operands are read all the same (unused).
  F::load_top(a, ke, task ? i : 0, jr, MODE == MODE_RESID && a.xlag, lo);
  F::load_top(a, ke + g.pitch, task ? i : 0, jr + 1, MODE == MODE_RESID && a.xlag, hi);
  double b = 0.0, rd = 0.0, qd = 0.0, x = 0.0;
  if constexpr (F::S::NEEDS_B) b = reinterpret_cast<const double*>(a.b + kn)[c];
  if constexpr (DOT) {
    rd = reinterpret_cast<const double*>(a.rdot + kn)[c];
    if (a.qdot != nullptr) qd = reinterpret_cast<const double*>(a.qdot + kn)[c];
  }
  if constexpr (MODE == MODE_KP) x = reinterpret_cast<const double*>(a.xvec + kn)[c];
  if (done) return;  // uniform over the grid

  FSums sums = {0.0, 0.0, make_double2(0.0, 0.0)};
  double res = 0.0;  // RESTRICT: b - K v of this lane's component
  if (task) {
    const double2 vlo = F::value(a, lo, i, jr, beta, lag, alag), vhi = F::value(a, hi, i, jr + 1, beta, lag, alag);
    // Scales of the warp.
    auto expo = [](double v) { return fx_exponent((unsigned)__double2hiint(v)); };
    const int e0 = max(expo(vlo.x), expo(vlo.y)), e1 = max(expo(vhi.x), expo(vhi.y));
    const int ec = max(e0, e1);
    const int B = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(ec, 1));
    const double2 zero2 = make_double2(0.0, 0.0);
    const Fx2 vb = fx2_from(vlo, B), vt = fx2_from(vhi, B);
    auto right = [](const Fx2& v) -> Fx2 {  // next column of the half (its last lane: its own value, halo only)
      return {{__shfl_down_sync(0xffffffffu, v.x.lo, 1, 16), __shfl_down_sync(0xffffffffu, v.x.mid, 1, 16),
               __shfl_down_sync(0xffffffffu, v.x.hi, 1, 16)},
              {__shfl_down_sync(0xffffffffu, v.y.lo, 1, 16), __shfl_down_sync(0xffffffffu, v.y.mid, 1, 16),
               __shfl_down_sync(0xffffffffu, v.y.hi, 1, 16)}};
    };
    const Fx2 vbr = right(vb), vtr = right(vt);
    const Fx2 ac = fsub(vbr, vb), bt = fsub(vtr, vt), up = fsub(fadd(vtr, vt), fadd(vbr, vb));
    const FxStrain w = {fx_add(ac.x, bt.x), fx_sub(bt.x, ac.x), up.y, fx_sub(bt.y, ac.y),
                        fx_add(up.x, fx_add(ac.y, bt.y))};
    const unsigned tag = fx_tag(lo.k);
    const int X = (int)(tag & 0x7ffu);
    const int Xm = (int)__reduce_max_sync(0xffffffffu, (unsigned)X);
    const int sh = Xm - X;
    const bool rare = __any_sync(0xffffffffu, tag != 0u && (sh >= 32 || (tag & FX_TAG_NEG)));
    FxStrain t = F::Elem::core(a, w, lo.k, rare);
    if (rare)
      t = {fx_sar_limbs(t.c1, sh), fx_sar_limbs(t.c3, sh), fx_sar_limbs(t.d2, sh), fx_sar_limbs(t.d3, sh),
           fx_sar_limbs(t.s, sh)};
    t = {fx_sar31(t.c1, sh & 31), fx_sar31(t.c3, sh & 31), fx_sar31(t.d2, sh & 31), fx_sar31(t.d3, sh & 31),
         fx_sar31(t.s, sh & 31)};
    // The node row is the top edge of the element row below (forces t_c1 + t_c3,
    // vertical forces +) and the bottom edge of the one above (t_c1 - t_c3, -).
    const int above = -half;
    const Fx2 h = {fx_add(t.c1, fx_flip(t.c3, above)), fx_add(t.s, fx_flip(t.d3, above))};
    const Fx2 v = {fx_flip(t.s, above), fx_flip(t.d2, above)};
    const Fx2 from_left = fadd(v, h);
    auto left = [](const Fx& f) -> Fx {
      return {__shfl_up_sync(0xffffffffu, f.lo, 1, 16), __shfl_up_sync(0xffffffffu, f.mid, 1, 16),
              __shfl_up_sync(0xffffffffu, f.hi, 1, 16)};
    };
    const Fx2 part = fadd(Fx2{left(from_left.x), left(from_left.y)}, fsub(v, h));
    // Each half sends the component that the other finishes.
    const Fx send = half ? part.x : part.y, keep = half ? part.y : part.x;
    const Fx got = {__shfl_xor_sync(0xffffffffu, send.lo, 16), __shfl_xor_sync(0xffffffffu, send.mid, 16),
                    __shfl_xor_sync(0xffffffffu, send.hi, 16)};
    const Fx sum = fx_add(keep, got);
    const int unit = B + Xm + F::Elem::UNIT;
    double kv = fx_to_double<false>(sum, unit);
    if (unit < FX_UNIT_MIN || unit > FX_UNIT_MAX) kv = fx_to_double(sum, unit);  // uniform over the warp
    // Whether the scales hold the terms of the elements, as in the marching
    // kernel; a non-finite value or modulus has made a scale non-finite.
    const int e4 = max(ec, __shfl_down_sync(0xffffffffu, ec, 1, 16));
    const bool again = (__any_sync(0xffffffffu, hl <= 14 && min(e4, X) != 0 && fx_beyond(B + Xm, e4 + X, F::Elem::SPAN)) ||
                        B == 0x7ff || Xm == 0x7ff) && !vzero;
    const double2 mid = half ? vlo : vhi;  // node row je
    const double vc = c ? mid.y : mid.x;
    if constexpr (MODE == MODE_KP) {
      const double2 old = half ? lo.v : hi.v;
      if (own && lag) reinterpret_cast<double*>(a.xvec + kn)[c] = fma(alag, c ? old.y : old.x, x);
    }
    if (again) {  // uniform over the warp: in float64, written from the lower half
      const FTask t0 = {i, lane, je - 1, 0, 0, own && half == 0};
      sums = rows_f64<SRC, MODE, DOT, ZT, !RESTRICT>(a, t0, je, beta, lag, alag);
      if constexpr (RESTRICT) kv = c ? sums.racc.y : sums.racc.x;
    }
    if (again && !RESTRICT) {
    } else if constexpr (MODE == MODE_APPLY) {
      double* out = reinterpret_cast<double*>(a.out + (a.dense ? (long long)je * (g.nx + 1) + i : kn));
      if (own) out[c] = act ? kv : 0.0;
    } else if constexpr (MODE == MODE_RESID) {
      const double r = act ? b - (vzero ? 0.0 : kv) : 0.0;
      if (own) {
        reinterpret_cast<double*>(a.out + kn)[c] = r;
        if (a.out32 != nullptr) reinterpret_cast<float*>(a.out32 + kn)[c] = float(r);
      }
      sums.dot0 = r * r;
    } else if constexpr (MODE == MODE_KP) {
      const double q = act ? kv : 0.0;
      if (own) {
        reinterpret_cast<double*>(a.p_out + kn)[c] = vc;
        reinterpret_cast<double*>(a.out + kn)[c] = q;
        sums.dot0 = vc * q;
      }
    } else if constexpr (F::SMOOTHING) {
      const double z = act ? fma(d, b - kv, vc) : 0.0;
      if (own) reinterpret_cast<double*>(a.out + kn)[c] = z;
      if constexpr (DOT) {
        sums.dot0 = z * rd;
        if (a.qdot != nullptr) sums.dot1 = z * qd;
      }
    } else if constexpr (RESTRICT) {
      res = act ? b - kv : 0.0;
    }
  }
  if constexpr (RESTRICT) {
    // Full weighting of the three rows, each column first.
    __shared__ double rows[SPLIT_RWARPS][32];
    rows[warp][lane] = res;
    __syncthreads();
    const int I = i >> 1;
    if (warp == 0 && row < a.nchunks && (hl & 1) == 0 && hl >= 2 && hl <= 12 && I >= 0 && I <= a.gc.nx) {
      auto column = [&](int l) { return fma(0.5, rows[2][l], fma(0.5, rows[0][l], rows[1][l])); };
      const double val = fma(0.5, column(lane - 1) + column(lane + 1), column(lane));
      reinterpret_cast<double*>(a.bc + a.gc.at(I, row))[c] = a.gc.is_fixed(I, row) ? 0.0 : val;
    }
  }
  if constexpr (REDUCE)
    block_reduce_finish<SWEEP_NT, DOT>(sums.dot0, sums.dot1, a.partials, a.ticket, a.sc, a.finish, a.out_value, a.tag);
}

}  // namespace mto
