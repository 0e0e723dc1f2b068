// The two-stage passes of the small float64 levels (Alg. 1) in fixed point,
// one tile of nodes per block: PRE2 (two smoothing sweeps from zero, residual,
// restriction) and POST2 (prolongation, two sweeps, on the finest level with
// the dot products of the CG recurrence).
//
// The tiles, stages and halos are those of mto_tile.cuh, the arithmetic is that
// of mto_fsweep.cuh: one thread per element or node, the marched values and the
// corner forces of the elements as 96-bit integers in shared memory, one scale
// per tile and stage.  An element whose terms the scales do not hold (fx_beyond
// in mto_fixed.cuh) is evaluated in float64, and a node next to one sums the two
// kinds apart.  Most launches of a first sweep on an optimised design hold a few
// such elements in the void, and wait for the tile that does: a float64 iteration
// of the optimiser's loop at 512^2 takes 169 us with fixed point alone, 190 with the
// whole tile done again, 183 so (1024^2 366, 414, 410; all with FX_SPAN_COARSE at 36).
//
// Against two launches of the row-per-warp kernel a pass saves a launch and a
// trip through memory (a coarse level 10.4 -> 9.6 us, the finest 256^2 one with
// its dot products 25 -> 22 us; a float64 PCG iteration 114 -> 108 us at 256^2,
// 391 -> 375 us at 1024^2).  Both stages run the same copy of the operator's code:
// a block executes it once each, and fetching it is a good part of the kernel's
// time (a float64 iteration 57.9 -> 54.0 us at 64^2, 105.3 -> 99.7 us at 256^2).
#pragma once

#include "mto_fsweep.cuh"
#include "mto_tile.cuh"

namespace mto {

// N values of 96 bits per component, limbs apart (no bank conflicts).
template <int N> struct FxArray {
  unsigned lo[N], mid[N];
  int hi[N];
  __device__ __forceinline__ Fx get(int i) const { return {lo[i], mid[i], hi[i]}; }
  __device__ __forceinline__ void put(int i, const Fx& v) {
    lo[i] = v.lo;
    mid[i] = v.mid;
    hi[i] = v.hi;
  }
  // A float64 in the place of one, marked by an upper limb that no value has.
  static constexpr int WIDE = 0x7fffffff;
  __device__ __forceinline__ bool is64(int i) const { return hi[i] == WIDE; }
  __device__ __forceinline__ double get64(int i) const { return __hiloint2double((int)mid[i], (int)lo[i]); }
  __device__ __forceinline__ void put64(int i, double v) {
    lo[i] = (unsigned)__double2loint(v);
    mid[i] = (unsigned)__double2hiint(v);
    hi[i] = WIDE;
  }
};

// An element's words, passed by value.
template <int SRC> struct FxWords {
  unsigned long long k[FxElem<SRC>::N];
};

// One operator evaluation per stage over a tile of NW x NH nodes.
template <int SRC, int NW, int NH> struct FTile {
  static constexpr int N = NW * NH, EW = NW - 1, EH = NH - 1, NE = EW * EH;
  FxArray<N> vx, vy;             // nodal values at the stage's scale
  FxArray<NE> fx[4], fy[4];      // forces of element e on its corners BL, BR, TR, TL
  int B[2], X;                   // scales: nodal values of the two stages, coefficients
  double2 value[N];              // the nodal values themselves
  unsigned mag[N];               // their magnitudes
  int any_wide;                  // some element of the tile is evaluated in float64 (of either stage)

  __device__ __forceinline__ static int exponent(const double2& v) { return (int)(fx_magnitude(v.x, v.y) >> 20); }
  // All threads, before the first raise() (with a barrier between).
  __device__ __forceinline__ void init() {
    if (threadIdx.x < 2) B[threadIdx.x] = 1;
    if (threadIdx.x == 2) X = 0;
    if (threadIdx.x == 3) any_wide = 0;
  }
  // Raises the scale of stage s to the exponent e of a thread's value (0: none).
  __device__ __forceinline__ void raise(int s, int e) {
    if (e == 0x7ff) e = 0;
    const int m = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
    if ((threadIdx.x & 31) == 0) atomicMax(&B[s], m);
  }
  __device__ __forceinline__ void raise_elements(unsigned tag) {
    const unsigned x = tag & 0x7ffu;
    const int m = (int)__reduce_max_sync(0xffffffffu, x == 0x7ffu ? 0u : x);
    if ((threadIdx.x & 31) == 0) atomicMax(&X, m);
  }
  // Node n gets value v at the scale of stage s (whole warps).
  __device__ __forceinline__ void put(int s, int n, bool in, double2 v) {
    const unsigned m = fx_magnitude(v.x, v.y);
    const Fx2 f = fx2_from((m >> 20) == 0x7ffu ? make_double2(0.0, 0.0) : v, B[s]);
    if (!in) return;
    value[n] = v;
    mag[n] = m;
    vx.put(n, f.x);
    vy.put(n, f.y);
  }
  // The forces in float64.  A call of its own, so that its registers do not weigh on the kernels.
  __device__ __noinline__ void element_f64(const SweepParams<double>& a, int e, int c, FxWords<SRC> words) {
    const Strain<double> w =
        strain_coords<double, double2>(value[c], value[c + 1], value[c + NW + 1], value[c + NW]);
    double2 f[4];
    strain_forces<double, double2>(FxElem<SRC>::core64(a, w, words.k), f[0], f[1], f[2], f[3]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      fx[q].put64(e, f[q].x);
      fy[q].put64(e, f[q].y);
    }
  }
  // Forces of the thread's element e at stage s, whose BL node is c; tag, words: its factors.
  __device__ __forceinline__ void element(const SweepParams<double>& a, int s, int e, int c, unsigned tag,
                                          const FxWords<SRC>& words, bool rare) {
    const unsigned m = max(max(mag[c], mag[c + 1]), max(mag[c + NW], mag[c + NW + 1]));
    const int x = (int)(tag & 0x7ffu);
    const bool w64 = (m >> 20) == 0x7ffu || x == 0x7ff || (m != 0u && x != 0 && fx_beyond(B[s] + X, (int)(m >> 20) + x, FxElem<SRC>::SPAN));
    if (w64) {
      any_wide = 1;
      element_f64(a, e, c, words);
      return;
    }
    const Fx2 bl = {vx.get(c), vy.get(c)}, br = {vx.get(c + 1), vy.get(c + 1)};
    const Fx2 tl = {vx.get(c + NW), vy.get(c + NW)}, tr = {vx.get(c + NW + 1), vy.get(c + NW + 1)};
    const Fx2 ac = fsub(br, bl), bt = fsub(tr, tl), up = fsub(fadd(tr, tl), fadd(br, bl));
    const FxStrain w = {fx_add(ac.x, bt.x), fx_sub(bt.x, ac.x), up.y, fx_sub(bt.y, ac.y),
                        fx_add(up.x, fx_add(ac.y, bt.y))};
    FxStrain t = FxElem<SRC>::core(a, w, words.k, rare);
    const int sh = X - (int)(tag & 0x7ffu);
    if (rare)
      t = {fx_sar_limbs(t.c1, sh), fx_sar_limbs(t.c3, sh), fx_sar_limbs(t.d2, sh), fx_sar_limbs(t.d3, sh),
           fx_sar_limbs(t.s, sh)};
    t = {fx_sar31(t.c1, sh & 31), fx_sar31(t.c3, sh & 31), fx_sar31(t.d2, sh & 31), fx_sar31(t.d3, sh & 31),
         fx_sar31(t.s, sh & 31)};
    const Fx ga = fx_sub(t.c1, t.c3), gb = fx_add(t.c1, t.c3), ha = fx_sub(t.s, t.d3), hb = fx_add(t.s, t.d3);
    fx[0].put(e, fx_neg(fx_add(ga, t.s)));
    fx[1].put(e, fx_sub(ga, t.s));
    fx[2].put(e, fx_add(gb, t.s));
    fx[3].put(e, fx_sub(t.s, gb));
    fy[0].put(e, fx_neg(fx_add(ha, t.d2)));
    fy[1].put(e, fx_sub(ha, t.d2));
    fy[2].put(e, fx_add(hb, t.d2));
    fy[3].put(e, fx_sub(t.d2, hb));
  }
  // K v at the node whose upper right element is e.
  __device__ __forceinline__ double2 at_node(int s, int e) const {
    const int unit = B[s] + X + FxElem<SRC>::UNIT;
    if (any_wide) return at_node_mixed(unit, e);  // uniform over the block
    const Fx x = fx_add(fx_add(fx[0].get(e), fx[1].get(e - 1)), fx_add(fx[2].get(e - EW - 1), fx[3].get(e - EW)));
    const Fx y = fx_add(fx_add(fy[0].get(e), fy[1].get(e - 1)), fx_add(fy[2].get(e - EW - 1), fy[3].get(e - EW)));
    double2 kv = make_double2(fx_to_double<false>(x, unit), fx_to_double<false>(y, unit));
    if (unit < FX_UNIT_MIN || unit > FX_UNIT_MAX)  // uniform over the block
      kv = make_double2(fx_to_double(x, unit), fx_to_double(y, unit));
    return kv;
  }
  // The same where an element may be in float64.
  __device__ __noinline__ double2 at_node_mixed(int unit, int e) const {
    const int at[4] = {e, e - 1, e - EW - 1, e - EW};
    Fx x = fx_zero(), y = x;
    double2 w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      w[q] = make_double2(0.0, 0.0);
      if (fx[q].is64(at[q])) {
        w[q] = make_double2(fx[q].get64(at[q]), fy[q].get64(at[q]));
      } else {
        x = fx_add(x, fx[q].get(at[q]));
        y = fx_add(y, fy[q].get(at[q]));
      }
    }
    return make_double2(((w[0].x + w[1].x) + (w[2].x + w[3].x)) + fx_to_double(x, unit),
                        ((w[0].y + w[1].y) + (w[2].y + w[3].y)) + fx_to_double(y, unit));
  }
};

template <int SRC> struct FTileElem {
  FxWords<SRC> words;
  unsigned tag;
  __device__ __forceinline__ void load(const SweepParams<double>& a, bool in, int ei, int ej) {
    const bool valid = in && ei >= 0 && ei < a.g.nx && ej >= 0 && ej < a.g.ny;
    const unsigned long long* E = static_cast<const unsigned long long*>(a.E) + (valid ? a.g.at(ei, ej) : 0);
#pragma unroll
    for (int n = 0; n < FxElem<SRC>::N; ++n) words.k[n] = valid ? __ldg(E + n * a.cstride) : 0ull;
    tag = fx_tag(words.k);
  }
  // A scale far below the tile's or an unexpected sign (whole warps; once X is final).
  __device__ __forceinline__ bool rare(int X) const {
    return __any_sync(0xffffffffu, tag != 0u && ((tag & FX_TAG_NEG) || X - (int)(tag & 0x7ffu) >= 32));
  }
};

// w/D of a node.
template <int SRC> __device__ __forceinline__ double2 ftile_d(const SweepParams<double>& a, long long k) {
  if constexpr (SRC == SRC_FINE64) {
    const double d = __ldg(a.invd1 + k);
    return make_double2(d, d);
  } else {
    return __ldg(a.invd2 + k);
  }
}

// Blocks per SM that the fixed-point path's registers allow (as split_blocks()).
template <int SRC>
__global__ void __launch_bounds__(SWEEP_NT, SRC == SRC_FINE64 ? 4 : 2)
    ftile_pre2_kernel(const __grid_constant__ SweepParams<double> a) {
  pdl_trigger();
  constexpr int NW = TILE_X + 5, NH = TILE_Y + 5, EW = NW - 1, EH = NH - 1, ZW = NW - 2, ZH = NH - 2;
  __shared__ FTile<SRC, NW, NH> f;
  __shared__ double2 r[ZW * ZH];
  static_assert(EW * EH <= SWEEP_NT && ZW * ZH <= SWEEP_NT && NW * NH <= 2 * SWEEP_NT, "threads");
  const Grid g = a.g, gc = a.gc;
  const int t = threadIdx.x;
  f.init();
  const int I0 = ((int)blockIdx.x % a.nstrips) * TILE_CX, J0 = ((int)blockIdx.x / a.nstrips) * TILE_CY;
  const int x0 = 2 * I0 - 3, y0 = 2 * J0 - 3;
  const int ex = t % EW, ey = t / EW;
  const bool elem = t < EW * EH;
  FTileElem<SRC> er;
  er.load(a, elem, x0 + ex, y0 + ey);
  // The thread's z1 node.
  const int zx = 1 + t % ZW, zy = 1 + t / ZW, i = x0 + zx, j = y0 + zy;
  const bool node = t < ZW * ZH, valid = node && g.valid(i, j);
  const double2 zero2 = make_double2(0.0, 0.0);
  double2 d = zero2, b = zero2;
  if (valid) d = ftile_d<SRC>(a, g.at(i, j));
  double2 z0[2];  // of the nodes t and t + SWEEP_NT: w/D, then the value
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int n = t + u * SWEEP_NT, ii = x0 + n % NW, jj = y0 + n / NW;
    z0[u] = n < NW * NH && g.valid(ii, jj) ? ftile_d<SRC>(a, g.at(ii, jj)) : zero2;
  }
  pdl_wait_prior();
  const bool done = a.sc != nullptr && a.gate && a.sc->done != RUNNING;
  if (valid) b = a.b[g.at(i, j)];
  double2 bh[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int n = t + u * SWEEP_NT, ii = x0 + n % NW, jj = y0 + n / NW;
    bh[u] = n < NW * NH && g.valid(ii, jj) ? a.b[g.at(ii, jj)] : zero2;
  }
  if (done) return;  // uniform over the grid
#pragma unroll
  for (int u = 0; u < 2; ++u) z0[u] = make_double2(z0[u].x * bh[u].x, z0[u].y * bh[u].y);
  __syncthreads();
  f.raise(0, f.exponent(z0[0]));
  f.raise(0, f.exponent(z0[1]));
  f.raise_elements(er.tag);
  __syncthreads();
  f.put(0, t, t < NW * NH, z0[0]);
  if (t < ((NW * NH - SWEEP_NT + 31) / 32) * 32) f.put(0, t + SWEEP_NT, t + SWEEP_NT < NW * NH, z0[1]);
  const bool rare = er.rare(f.X);
  __syncthreads();
  // Stage 0: z1 = z0 + w/D (b - K z0); stage 1: the residual.
  const int c = ey * NW + ex;
  const int zn = zy * NW + zx, en = zy * EW + zx;  // node and its upper right element
  const bool act = node && g.active(i, j);
  const bool inner = node && zx >= 2 && zx < NW - 2 && zy >= 2 && zy < NH - 2;
  const bool inner_elem = elem && ex >= 1 && ex < EW - 1 && ey >= 1 && ey < EH - 1;
  double2 kv = zero2;
#pragma unroll 1
  for (int s = 0;; ++s) {
    if (s == 0 ? elem : inner_elem) f.element(a, s, t, c, er.tag, er.words, rare);
    __syncthreads();
    if (s == 0 ? act : inner && act) kv = f.at_node(s, en);
    if (s == 1) break;
    double2 z1 = zero2;
    if (act) z1 = make_double2(fma(d.x, b.x - kv.x, d.x * b.x), fma(d.y, b.y - kv.y, d.y * b.y));
    if (valid && zx >= 3 && zx < 3 + TILE_X && zy >= 3 && zy < 3 + TILE_Y) a.out[g.at(i, j)] = z1;
    f.raise(1, f.exponent(z1));
    __syncthreads();
    f.put(1, zn, node, z1);
    __syncthreads();
  }
  if (inner) r[t] = act ? make_double2(b.x - kv.x, b.y - kv.y) : zero2;
  __syncthreads();
  // Full weighting, over the three rows of each column first; one component per thread.
  if (t < 2 * TILE_CX * TILE_CY) {
    const int cc = t & 1, p = (t >> 1) % TILE_CX, q = (t >> 1) / TILE_CX, I = I0 + p, J = J0 + q;
    if (I <= gc.nx && J <= gc.ny) {
      const int n = (2 + 2 * q) * ZW + 2 + 2 * p;  // r at fine node (2 I, 2 J)
      auto at = [&](int k) { return cc ? r[k].y : r[k].x; };
      auto column = [&](int k) { return fma(0.5, at(k + ZW), fma(0.5, at(k - ZW), at(k))); };
      const double val = fma(0.5, column(n - 1) + column(n + 1), column(n));
      reinterpret_cast<double*>(a.bc + gc.at(I, J))[cc] = gc.is_fixed(I, J) ? 0.0 : val;
    }
  }
}

template <int SRC, bool DOT>
__global__ void __launch_bounds__(SWEEP_NT, SRC == SRC_FINE64 ? (DOT ? 3 : 4) : 2)
    ftile_post2_kernel(const __grid_constant__ SweepParams<double> a) {
  pdl_trigger();
  constexpr int NW = TILE_X + 4, NH = TILE_Y + 4, EW = NW - 1, EH = NH - 1, ZW = NW - 2, ZH = NH - 2;
  __shared__ FTile<SRC, NW, NH> f;
  static_assert(EW * EH <= SWEEP_NT && NW * NH <= SWEEP_NT, "threads");
  const Grid g = a.g, gc = a.gc;
  const int t = threadIdx.x;
  f.init();
  const int x0 = ((int)blockIdx.x % a.nstrips) * TILE_X - 2, y0 = ((int)blockIdx.x / a.nstrips) * TILE_Y - 2;
  const int ex = t % EW, ey = t / EW;
  const bool elem = t < EW * EH;
  FTileElem<SRC> er;
  er.load(a, elem, x0 + ex, y0 + ey);
  // The thread's z2 (and z3) node.
  const int zx = 1 + t % ZW, zy = 1 + t / ZW, i = x0 + zx, j = y0 + zy;
  const bool node = t < ZW * ZH, valid = node && g.valid(i, j);
  const bool own = valid && zx >= 2 && zx < 2 + TILE_X && zy >= 2 && zy < 2 + TILE_Y;
  const double2 zero2 = make_double2(0.0, 0.0);
  double2 d = zero2, b = zero2, rd = zero2, qd = zero2;
  const long long k = valid ? g.at(i, j) : 0;
  if (valid) d = ftile_d<SRC>(a, k);
  pdl_wait_prior();
  const bool done = a.sc != nullptr && a.gate && a.sc->done != RUNNING;
  if (valid) b = a.b[k];
  if constexpr (DOT) {
    if (own) {
      rd = a.rdot[k];
      if (a.qdot != nullptr) qd = a.qdot[k];
    }
  }
  // z = v + P z_c at node t (the interpolation of mto_fsweep.cuh).
  double2 v = zero2;
  {
    const int ii = x0 + t % NW, jj = y0 + t / NW;
    if (t < NW * NH && g.valid(ii, jj)) {
      v = a.v[g.at(ii, jj)];
      const long long kc = gc.at(ii >> 1, jj >> 1);
      double2 t0 = a.zc[kc], t1 = a.zc[kc + (ii & 1)];
      double w = 0.5;
      if (jj & 1) {
        const double2 u0 = a.zc[kc + gc.pitch], u1 = a.zc[kc + gc.pitch + (ii & 1)];
        t0 = add2(t0, u0);
        t1 = add2(t1, u1);
        w = 0.25;
      }
      v = make_double2(fma(w, t0.x + t1.x, v.x), fma(w, t0.y + t1.y, v.y));
    }
  }
  if (done) return;  // uniform over the grid
  __syncthreads();
  f.raise(0, f.exponent(v));
  f.raise_elements(er.tag);
  __syncthreads();
  f.put(0, t, t < NW * NH, v);
  const bool rare = er.rare(f.X);
  __syncthreads();
  const int c = ey * NW + ex;
  const int zn = zy * NW + zx, en = zy * EW + zx;
  const bool act = node && g.active(i, j);
  const bool inner_elem = elem && ex >= 1 && ex < EW - 1 && ey >= 1 && ey < EH - 1;
  double2 z = act ? f.value[zn] : zero2;
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    if (s == 0 ? elem : inner_elem) f.element(a, s, t, c, er.tag, er.words, rare);
    __syncthreads();
    if (s == 0 ? act : own && act) {
      const double2 kv = f.at_node(s, en);
      z = make_double2(fma(d.x, b.x - kv.x, z.x), fma(d.y, b.y - kv.y, z.y));
    }
    if (s == 1) break;
    f.raise(1, f.exponent(z));
    __syncthreads();
    f.put(1, zn, node, z);
    __syncthreads();
  }
  double dot0 = 0.0, dot1 = 0.0;
  if (own) {
    a.out[k] = z;
    if constexpr (DOT) {
      dot0 = fma(z.x, rd.x, z.y * rd.y);
      if (a.qdot != nullptr) dot1 = fma(z.x, qd.x, z.y * qd.y);
    }
  }
  if constexpr (DOT)
    block_reduce_finish<SWEEP_NT>(dot0, dot1, a.partials, a.ticket, a.sc, a.finish, a.out_value, a.tag);
}

}  // namespace mto
