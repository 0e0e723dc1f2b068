// Shared by the matrix-free stencil sweeps of the V-cycle and of the outer CG
// operator: sources, modes, parameters, and the element data of the float32
// coarse levels.  The kernels are in mto_sweep2.cuh (float32), mto_fsweep.cuh
// (float64, in fixed point), mto_fused.cuh, mto_tile.cuh and mto_ftile.cuh.
//
// A marching sweep: one warp owns a strip of node columns and a chunk of rows
// and marches upwards one element row per step.  A lane takes the node values
// of the new top row (its right neighbour's by shuffle), forms the element to
// its right once, and completes node row je.  The outer lanes' columns are halo
// shared with the neighbouring strips, so every lane runs the same
// instructions; every node value is read once plus one halo row per chunk, and
// there is no shared memory and no atomics.  Loads run PF steps ahead of the
// arithmetic (a register ring); addresses advance by one row pitch per step.
//
// The element operator works on edges (see mto_common.cuh for the strain
// basis).  Per element: the top-edge differences b, the left-edge differences
// dl (the bottom edge is the previous step's top edge), then c1 = a + b,
// c3 = b - a, c2 = dl + dr (u_x) and the same for u_y; after the 5x5 core, the
// forces go back through the edges: a horizontal edge collects ga = t_c1 - t_c3
// from the element above it and gb = t_c1 + t_c3 from the element below, a
// vertical edge collects t_s (u_x) or t_d2 (u_y) from its two elements, and a
// node sums its four edges with signs: about a third fewer operations than
// forming the four corner forces of every element.
//
// Modes (all masked by the clamped edges; ghost nodes are zero by layout):
//   APPLY    out = K v
//   RESID    out = b - K v,                        dot |out|^2
//   KP       p = z + beta p_old, q = K p,           dot p.q      (Alg. 2)
//   SMOOTH   out = v + w D^-1 (b - K v)                           (Sec. 2.3)
//   SMOOTH0  as SMOOTH with v = w D^-1 b formed on the fly (first sweep
//            from zero followed by the second, Alg. 1 pre-smoothing)
//   PSMOOTH  v' = v + P zc (Alg. 1 correction), out = v' + w D^-1 (b - K v')
//   RESTRICT bc = P^T (b - K v) on the next coarser grid          (Alg. 1)
// SMOOTH/PSMOOTH optionally accumulate z.r (and z.q for the flexible beta).
#pragma once

#include "mto_common.cuh"

namespace mto {

constexpr int SWEEP_NT = 256;
// Output columns per warp: 30 (lanes 1..30) for the stencil modes, 28 fine
// columns = 14 coarse columns for the restriction.
constexpr int SWEEP_STRIDE = 30;
constexpr int SWEEP_RSTRIDE = 28;

// SRC_FINE64, SRC_COARSE: the float64 finest and coarse levels, fixed-point
// element factors (mto_fixed.cuh).  SRC_FINEBF: the bf16 moduli of the mixed
// path's finest level.  SRC_CFINE: the first coarse level of the mixed path,
// whose Galerkin element matrices are rebuilt on the fly from the four bf16
// fine moduli they cover (8 bytes per coarse element instead of 13 stored
// coefficients).  SRC_CMOM: the deeper float32 coarse levels, which store the
// six scaled moments of each element (24 bytes) and form the 13 coefficients in
// registers.
enum Src { SRC_FINE64 = 0, SRC_FINEBF = 1, SRC_COARSE = 2, SRC_CFINE = 3, SRC_CMOM = 4 };
enum Mode {
  MODE_APPLY = 0,
  MODE_RESID,
  MODE_KP,
  MODE_SMOOTH,
  MODE_PSMOOTH,
  MODE_RESTRICT,
  MODE_SMOOTH0,
  // Two-stage passes of the float32 coarse levels (mto_fused.cuh, mto_tile.cuh),
  // of small bf16 finest levels and small float64 levels (mto_tile.cuh, mto_ftile.cuh):
  MODE_POST2,  // prolongation + two sweeps, fused
  MODE_PRE2    // two sweeps from zero + residual + restriction, fused
};

template <typename T> struct SweepParams {
  using T2 = typename V2<T>::t;
  Grid g;   // this level
  Grid gc;  // next coarser level (PSMOOTH source, RESTRICT target)
  int nstrips, nchunks, H;
  int gate;          // 1: skip the launch once the PCG has stopped (sc->done)
  int replace_gate;  // RESID as residual replacement: run only when iter % rr_every == 0
  int zero_gate;     // RESID of the initial guess: out = b when sc->x_nonzero == 0 (K 0 = 0)
  const T2* v;       // marched vector (z, x or p_old)
  const T2* zc;      // PSMOOTH: coarse correction
  const void* zkp;   // KP: z (double2 or float2)
  T2* p_out;         // KP: new search direction
  T2* xvec;          // KP: the iterate x, advanced by the pending step alpha p_old (x_lag)
  const T2* xdir;    // RESID with xlag: the direction p of the pending step
  int xlag;          // RESID: apply the pending step to v on the fly (v = x + alpha p) when x_lag
  int tag;           // KP: index of p_out among the two search-direction buffers
  const T2* b;       // right-hand side (SMOOTH, SMOOTH0, PSMOOTH, RESTRICT, RESID)
  T2* out;           // output vector (APPLY, RESID, KP: q, SMOOTH*, PSMOOTH)
  float2* out32;     // RESID: optional float32 copy of out (the mixed V-cycle's input)
  T2* bc;            // RESTRICT: coarse right-hand side
  const void* E;     // fixed-point factors (SRC_FINE64, SRC_COARSE: arrays of cstride words) or bf16 moduli
  const T* coef;     // SRC_CMOM: NMOM arrays of cstride scaled moments
  long long cstride;
  T cnu, cg;         // SRC_CMOM: nu and g = (1 - nu) / 2
  unsigned long long gfix;  // SRC_COARSE: g in units of 2^-64
  FineConst<T> kf;      // bf16 finest level / SRC_CFINE: scale factors of the element core
  Grid gfine;           // SRC_CFINE: the finer grid whose bf16 moduli E points to
  int redisc;           // SRC_CFINE: rediscretised (mean modulus) instead of Galerkin
  const double* invd1;  // float64 finest level: w / D per node
  const T2* invd2;      // coarse levels: w / D per DOF
  T wdiag;              // float32 finest level: w / (KE_00 at E = 1); D = sum of 4 moduli
  const double2* rdot;  // dot partner for z.r
  const double2* qdot;  // dot partner for z.q (flexible beta), may be null
  int dense;               // float64 APPLY: v and out in the caller's layout [ny + 1][nx + 1] (no padding)
  const double2* din;      // bf16 SMOOTH0 of a V-cycle called alone: b in the caller's layout
  double2* dout;           // bf16 SMOOTH: output in the caller's layout instead of out (may be null)
  double2* r64;            // bf16 SMOOTH0 with the CG update: r of this step (written)
  const double2* r64_prev;  // ... r of the last step, read while the update is pending
  const double2* q64;       // ... and q = K p of the last step
  double* partials;
  unsigned* ticket;
  DevScalars* sc;
  int finish;
  double* out_value;
};

template <typename T2> __device__ __forceinline__ T2 shfl_down2(T2 v) {
  v.x = __shfl_down_sync(0xffffffffu, v.x, 1);
  v.y = __shfl_down_sync(0xffffffffu, v.y, 1);
  return v;
}
template <typename T2> __device__ __forceinline__ T2 shfl_up2(T2 v) {
  v.x = __shfl_up_sync(0xffffffffu, v.x, 1);
  v.y = __shfl_up_sync(0xffffffffu, v.y, 1);
  return v;
}
template <typename T2> __device__ __forceinline__ T2 add2(T2 a, T2 b) {
  a.x += b.x;
  a.y += b.y;
  return a;
}
template <typename T2> __device__ __forceinline__ T2 sub2(T2 a, T2 b) {
  a.x -= b.x;
  a.y -= b.y;
  return a;
}
// float2 pairs use Blackwell's packed FP32 instructions (two correctly
// rounded operations per instruction): the float32 sweeps are bound by
// instruction issue, and most of their arithmetic treats u_x and u_y alike.
__device__ __forceinline__ unsigned long long pk2(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 upk2(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
template <> __device__ __forceinline__ float2 add2<float2>(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pk2(a)), "l"(pk2(b)));
  return upk2(r);
}
template <> __device__ __forceinline__ float2 sub2<float2>(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pk2(a)), "l"(pk2(b)));
  return upk2(r);
}
// a * b + c per component (float2: one packed FMA).
template <typename T2> __device__ __forceinline__ T2 fma2(T2 a, T2 b, T2 c) {
  c.x = fma(a.x, b.x, c.x);
  c.y = fma(a.y, b.y, c.y);
  return c;
}
template <> __device__ __forceinline__ float2 fma2<float2>(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pk2(a)), "l"(pk2(b)), "l"(pk2(c)));
  return upk2(r);
}
template <typename T2> __device__ __forceinline__ T2 mul2(T2 a, T2 b) {
  a.x *= b.x;
  a.y *= b.y;
  return a;
}
template <> __device__ __forceinline__ float2 mul2<float2>(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pk2(a)), "l"(pk2(b)));
  return upk2(r);
}

template <typename T, int SRC> struct ERaw;
template <typename T> struct ERaw<T, SRC_FINEBF> {
  T E;
};
template <typename T> struct ERaw<T, SRC_CFINE> {
  __nv_bfloat162 lo, hi;  // fine moduli of rows 2J and 2J+1, columns 2I and 2I+1
};
template <typename T> struct ERaw<T, SRC_CMOM> {
  T m[NMOM];
};

template <typename T, int SRC, int MODE, bool DOT, typename ZT> struct Sweep {
  using T2 = typename V2<T>::t;
  using ER = ERaw<T, SRC>;
  static constexpr bool NEEDS_B = MODE == MODE_RESID || MODE == MODE_SMOOTH ||
                                  MODE == MODE_SMOOTH0 || MODE == MODE_PSMOOTH ||
                                  MODE == MODE_RESTRICT;
  static constexpr bool SMOOTHING = MODE == MODE_SMOOTH || MODE == MODE_SMOOTH0 ||
                                    MODE == MODE_PSMOOTH;

  __device__ __forceinline__ static void load_e(const SweepParams<T>& a, long long e, int ii, int jj,
                                                ER& r) {
    if constexpr (SRC == SRC_FINEBF) {
      r.E = __bfloat162float(static_cast<const __nv_bfloat16*>(a.E)[e]);
    } else if constexpr (SRC == SRC_CFINE) {
      // Ghost and padding elements have no children: zero operator.
      if ((unsigned)ii < (unsigned)a.g.nx && (unsigned)jj < (unsigned)a.g.ny) {
        const __nv_bfloat162* Ef = static_cast<const __nv_bfloat162*>(a.E);
        const long long kf = a.gfine.at(2 * ii, 2 * jj);  // even: bf16 pairs are aligned
        r.lo = Ef[kf >> 1];
        r.hi = Ef[(kf + a.gfine.pitch) >> 1];
      } else {
        r.lo = r.hi = __floats2bfloat162_rn(0.f, 0.f);
      }
    } else {
      static_assert(SRC == SRC_CMOM, "elements read one by one: the float32 levels");
#pragma unroll
      for (int c = 0; c < NMOM; ++c) r.m[c] = a.coef[c * a.cstride + e];
    }
  }

  // Strain-space forces t = A w of one element.
  __device__ __forceinline__ static Strain<T> core(const SweepParams<T>& a, const ER& er,
                                                   const Strain<T>& w) {
    Strain<T> t;
    if constexpr (SRC == SRC_FINEBF) {
      t = fine_core<T>(w, er.E, a.kf);
    } else if constexpr (SRC == SRC_CFINE) {
      // Moments of the four child moduli (children at xi, eta = +-1/2 of the
      // parent): M00 = S/4, M10 = X/8, M01 = Y/8, M20 = M02 = M00/3,
      // M11 = Z/16, then the 13 coefficients of mto_common.cuh.
      const float2 l = __bfloat1622float2(er.lo), h = __bfloat1622float2(er.hi);
      const T e00 = l.x, e10 = l.y, e01 = h.x, e11 = h.y;
      const T M00 = T(0.25) * ((e00 + e10) + (e01 + e11));
      T M10 = T(0.125) * ((e10 + e11) - (e00 + e01));
      T M01 = T(0.125) * ((e01 + e11) - (e00 + e10));
      T M11 = T(0.0625) * ((e00 + e11) - (e10 + e01));
      if (a.redisc) M10 = M01 = M11 = T(0);
      const FineConst<T> k = a.kf;  // kappa, kappa nu, kappa (1+g)/3, kappa g
      T A[NCOEF];
      A[0] = k.kA * M00;
      A[1] = k.kA * M01;
      A[2] = k.kC * M00;
      A[3] = k.kA * M00;
      A[4] = k.kA * M10;
      A[5] = k.kC * M00;
      A[6] = k.kB * M00;
      A[7] = k.kB * M10;
      A[8] = k.kB * M01;
      A[9] = (k.kB + k.kG) * M11;
      A[10] = k.kG * M00;
      A[11] = k.kG * M10;
      A[12] = k.kG * M01;
      t = coarse_core<T>(w, A);
    } else {
      T A[NCOEF];
      coefs_from_kmom<T>(er.m, a.cnu, a.cg, A);
      t = coarse_core<T>(w, A);
    }
    return t;
  }
};

}  // namespace mto
