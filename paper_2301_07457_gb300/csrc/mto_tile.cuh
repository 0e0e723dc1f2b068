// The two-stage passes of the small float32 levels (Alg. 1), one tile of nodes
// per block.
//
// Same passes as the marching kernels of mto_fused.cuh: PRE2 (two smoothing
// sweeps from zero, residual, restriction) and POST2 (prolongation, two
// sweeps).  On a small grid a marching task has one or two rows of output but
// marches five to seven, 300 instructions each, in one warp: 4.6 us of a
// launch's 7.5.  Here a block holds the tile and its halo in shared memory and
// takes one thread per element or node, so that a pass is a chain of two
// element evaluations and two node sums; the halo (about the tile again) is
// recomputed, which costs nothing while the grid does not fill the chip.
// Element data and diagonals are loaded before the wait for the previous
// kernel.
//
// Every value is formed by the same operations in the same order as there, so
// the results are those of the marching kernels bit for bit.
//
// On the bf16 finest level the passes replace two marching kernels each
// (mto_sweep2.cuh): PRE2 with DOT also carries the CG update of the outer
// iteration, POST2 with DOT forms the dot products (their partial sums are per
// tile, so these differ in the last bits).  Two launches and a trip through
// memory less per cycle at each end: a mixed iteration 56 -> 45 us at 200 x 136.
//
// The finest-level passes do not let the next kernel launch early: its blocks
// would wait in the registers and shared memory that this kernel's own tiles
// (one to five per SM, with a reduction at their end) and another load case's
// kernels still want.  With and without the early launch: mixed iteration at
// 200 x 136 47.4 -> 45.4 us, its two load cases at once 1590 -> 1316 us, 256^2
// 2115 -> 1980 us, one 64^2 solve 734 -> 748 us.  Coarse levels gain from it
// (mixed iteration at 2048^2 366.6 -> 363.6 us, at 1024^2 144.7 -> 142.2 us).
#pragma once

#include "mto_fused.cuh"

namespace mto {

constexpr int TILE_CX = 8, TILE_CY = 4;             // PRE2: coarse nodes per block
constexpr int TILE_X = 2 * TILE_CX, TILE_Y = 2 * TILE_CY;  // fine nodes per block (POST2: its output)

// Element forces in shared memory: bottom edge ga, top edge gb, vertical gs
// (the edge bookkeeping of mto_sweep.cuh), EW x EH elements.
template <int EW, int EH> struct TileForces {
  float2 ga[EW * EH], gb[EW * EH], gs[EW * EH];

  // Forces of element e from its corner values.
  template <int SRC>
  __device__ __forceinline__ void put(const SweepParams<float>& a, const ERaw<float, SRC>& er, int e, float2 bl,
                                      float2 br, float2 tl, float2 tr) {
    const float2 ac = sub2(br, bl), bt = sub2(tr, tl), dl = sub2(tl, bl), dr = sub2(tr, br);
    const float2 cd1 = add2(ac, bt), cd3 = sub2(bt, ac), cd2 = add2(dl, dr);
    Strain<float> w;
    w.c1 = cd1.x;
    w.c3 = cd3.x;
    w.d3 = cd3.y;
    w.d2 = cd2.y;
    w.s = cd2.x + cd1.y;
    const Strain<float> t = Sweep<float, SRC, MODE_SMOOTH, false, float2>::core(a, er, w);
    const float2 p = make_float2(t.c1, t.s), m = make_float2(t.c3, t.d3);
    ga[e] = sub2(p, m);
    gb[e] = add2(p, m);
    gs[e] = make_float2(t.s, t.d2);
  }
  // K v at the node whose upper right element is e.
  __device__ __forceinline__ float2 at_node(int e) const {
    const float2 gh = add2(ga[e], gb[e - EW]), ghl = add2(ga[e - 1], gb[e - EW - 1]);
    const float2 gv = add2(gs[e], gs[e - 1]), gvp = add2(gs[e - EW], gs[e - EW - 1]);
    return add2(sub2(ghl, gh), sub2(gvp, gv));
  }
};

// Element (ei, ej), zero outside the mesh.
template <int SRC>
__device__ __forceinline__ ERaw<float, SRC> tile_element(const SweepParams<float>& a, int ei, int ej) {
  ERaw<float, SRC> er{};
  if (ei >= 0 && ei < a.g.nx && ej >= 0 && ej < a.g.ny)
    Sweep<float, SRC, MODE_SMOOTH, false, float2>::load_e(a, a.g.at(ei, ej), ei, ej, er);
  return er;
}

// w/D at node (i, j) of the bf16 finest level, zero on clamped and ghost nodes.
__device__ __forceinline__ float2 tile_winv(const SweepParams<float>& a, int i, int j) {
  if (!a.g.active(i, j)) return make_float2(0.f, 0.f);
  const __nv_bfloat16* E = static_cast<const __nv_bfloat16*>(a.E) + a.g.at(i, j);
  const float own = __bfloat162float(E[-a.g.pitch]) + __bfloat162float(E[0]);
  const float left = __bfloat162float(E[-a.g.pitch - 1]) + __bfloat162float(E[-1]);
  const float w = __fdividef(a.wdiag, own + left);
  return make_float2(w, w);
}
template <int SRC> __device__ __forceinline__ float2 tile_d(const SweepParams<float>& a, int i, int j) {
  if constexpr (SRC == SRC_FINEBF) return tile_winv(a, i, j);
  else return __ldg(a.invd2 + a.g.at(i, j));
}

template <int SRC, bool DOT>
__global__ void __launch_bounds__(SWEEP_NT) tile_pre2_kernel(const SweepParams<float> a) {
  if constexpr (SRC != SRC_FINEBF) pdl_trigger();  // see the top of the file
  constexpr bool FBF = SRC == SRC_FINEBF;
  // z0 on NW x NH nodes from (x0, y0), elements one less each way; z1 inside.
  constexpr int NW = TILE_X + 5, NH = TILE_Y + 5, EW = NW - 1, EH = NH - 1, ZW = NW - 2, ZH = NH - 2;
  static_assert(EW * EH <= SWEEP_NT && ZW * ZH <= SWEEP_NT, "one element and one node per thread");
  __shared__ TileForces<EW, EH> f;
  __shared__ float2 z[NW * NH], r[ZW * ZH];
  const Grid g = a.g, gc = a.gc;
  const int t = threadIdx.x;
  const int I0 = ((int)blockIdx.x % a.nstrips) * TILE_CX, J0 = ((int)blockIdx.x / a.nstrips) * TILE_CY;
  const int x0 = 2 * I0 - 3, y0 = 2 * J0 - 3;
  const int ex = t % EW, ey = t / EW;
  const bool elem = t < EW * EH;
  ERaw<float, SRC> er{};
  if (elem) er = tile_element<SRC>(a, x0 + ex, y0 + ey);
  // The thread's z1 node.
  const int zx = 1 + t % ZW, zy = 1 + t / ZW, i = x0 + zx, j = y0 + zy;
  const bool node = t < ZW * ZH, valid = node && g.valid(i, j);
  const float2 zero2 = make_float2(0.f, 0.f);
  float2 d = zero2, b = zero2;
  if (valid) d = tile_d<SRC>(a, i, j);
  float2 dh[2], bh[2];  // of the z0 nodes t and t + SWEEP_NT
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int n = t + u * SWEEP_NT, ii = x0 + n % NW, jj = y0 + n / NW;
    dh[u] = n < NW * NH && g.valid(ii, jj) ? tile_d<SRC>(a, ii, jj) : zero2;
  }
  pdl_wait_prior();
  const bool done = a.sc != nullptr && a.gate && a.sc->done != RUNNING;
  double dot0 = 0.0;
  if constexpr (FBF) {
    // Right-hand side from float64, into shared memory for the z1 nodes: r
    // after the CG update (as in mto_sweep2.cuh), or the caller's vector.
    __shared__ float2 bs[NW * NH];
    bool upd = false;
    double aupd = 0.0;
    if constexpr (DOT) {
      upd = a.sc->upd_pending != 0;
      aupd = upd ? a.sc->alpha : 0.0;
    }
    if (done) return;  // uniform over the grid
    double2 rv[2], qv[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int n = t + u * SWEEP_NT, ii = x0 + n % NW, jj = y0 + n / NW;
      rv[u] = qv[u] = make_double2(0.0, 0.0);
      if constexpr (DOT) {
        if (n < NW * NH && g.valid(ii, jj)) {
          rv[u] = upd ? a.r64_prev[g.at(ii, jj)] : static_cast<const double2*>(a.r64)[g.at(ii, jj)];
          if (upd) qv[u] = a.q64[g.at(ii, jj)];  // else q is a leftover, perhaps not finite
        }
      } else {
        if (n < NW * NH && g.active(ii, jj)) rv[u] = a.din[(long long)jj * (g.nx + 1) + ii];
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int n = t + u * SWEEP_NT, nx = n % NW, ny = n / NW;
      const bool own = nx >= 3 && nx < 3 + TILE_X && ny >= 3 && ny < 3 + TILE_Y && g.valid(x0 + nx, y0 + ny);
      if constexpr (DOT) {
        const double2 rn = make_double2(fma(-aupd, qv[u].x, rv[u].x), fma(-aupd, qv[u].y, rv[u].y));
        bh[u] = make_float2(d2f_rn(rn.x), d2f_rn(rn.y));
        if (upd && own) {
          a.r64[g.at(x0 + nx, y0 + ny)] = rn;
          a.out32[g.at(x0 + nx, y0 + ny)] = bh[u];
          dot0 = fma(rn.x, rn.x, fma(rn.y, rn.y, dot0));
        }
      } else {
        bh[u] = make_float2((float)rv[u].x, (float)rv[u].y);
        if (own) a.out32[g.at(x0 + nx, y0 + ny)] = bh[u];
      }
      if (n < NW * NH) {
        z[n] = mul2(dh[u], bh[u]);
        bs[n] = bh[u];
      }
    }
    __syncthreads();
    if (node) b = bs[zy * NW + zx];
  } else {
    if (valid) b = a.b[g.at(i, j)];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int n = t + u * SWEEP_NT, ii = x0 + n % NW, jj = y0 + n / NW;
      bh[u] = n < NW * NH && g.valid(ii, jj) ? a.b[g.at(ii, jj)] : zero2;
    }
    if (done) return;  // uniform over the grid
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int n = t + u * SWEEP_NT;
      if (n < NW * NH) z[n] = mul2(dh[u], bh[u]);
    }
    __syncthreads();
  }
  // z1 = z0 + w/D (b - K z0).
  const int c = ey * NW + ex;
  if (elem) f.template put<SRC>(a, er, t, z[c], z[c + 1], z[c + NW], z[c + NW + 1]);
  __syncthreads();
  const int zn = zy * NW + zx, en = zy * EW + zx;  // node and its upper right element
  if (node) {
    const float2 z1 = fma2(d, sub2(b, f.at_node(en)), z[zn]);
    z[zn] = z1;
    if (valid && zx >= 3 && zx < 3 + TILE_X && zy >= 3 && zy < 3 + TILE_Y) a.out[g.at(i, j)] = z1;
  }
  __syncthreads();
  // Residual.
  if (elem && ex >= 1 && ex < EW - 1 && ey >= 1 && ey < EH - 1)
    f.template put<SRC>(a, er, t, z[c], z[c + 1], z[c + NW], z[c + NW + 1]);
  __syncthreads();
  if (node && zx >= 2 && zx < NW - 2 && zy >= 2 && zy < NH - 2) {
    const float m = g.active(i, j) ? 1.f : 0.f;
    r[t] = mul2(sub2(b, f.at_node(en)), make_float2(m, m));
  }
  __syncthreads();
  // Full weighting: across, then over the three rows.
  if (t < TILE_CX * TILE_CY) {
    const int p = t % TILE_CX, q = t / TILE_CX, I = I0 + p, J = J0 + q;
    if (I <= gc.nx && J <= gc.ny) {
      const int n = (2 + 2 * q) * ZW + 2 + 2 * p;  // r at fine node (2 I, 2 J)
      auto across = [&](int k) {
        const float2 r0 = r[k], r1 = r[k + 1], rl = r[k - 1];
        return make_float2(r0.x + 0.5f * (r1.x + rl.x), r0.y + 0.5f * (r1.y + rl.y));
      };
      const float2 lo = across(n - ZW), mid = across(n), hi = across(n + ZW);
      const float2 acc = add2(make_float2(0.5f * lo.x, 0.5f * lo.y), mid);
      const float2 val = make_float2(acc.x + 0.5f * hi.x, acc.y + 0.5f * hi.y);
      a.bc[gc.at(I, J)] = gc.is_fixed(I, J) ? zero2 : val;
    }
  }
  if constexpr (DOT)
    block_reduce_finish<SWEEP_NT, false>(dot0, 0.0, a.partials, a.ticket, a.sc, a.finish, a.out_value, a.tag);
}

template <int SRC, bool DOT>
__global__ void __launch_bounds__(SWEEP_NT) tile_post2_kernel(const SweepParams<float> a) {
  if constexpr (SRC != SRC_FINEBF) pdl_trigger();  // see the top of the file
  constexpr int NW = TILE_X + 4, NH = TILE_Y + 4, EW = NW - 1, EH = NH - 1, ZW = NW - 2, ZH = NH - 2;
  static_assert(EW * EH <= SWEEP_NT && NW * NH <= SWEEP_NT, "one element and one node per thread");
  __shared__ TileForces<EW, EH> f;
  __shared__ float2 z[NW * NH];
  const Grid g = a.g, gc = a.gc;
  const int t = threadIdx.x;
  const int x0 = ((int)blockIdx.x % a.nstrips) * TILE_X - 2, y0 = ((int)blockIdx.x / a.nstrips) * TILE_Y - 2;
  const int ex = t % EW, ey = t / EW;
  const bool elem = t < EW * EH;
  ERaw<float, SRC> er{};
  if (elem) er = tile_element<SRC>(a, x0 + ex, y0 + ey);
  // The thread's z2 (and z3) node.
  const int zx = 1 + t % ZW, zy = 1 + t / ZW, i = x0 + zx, j = y0 + zy;
  const bool node = t < ZW * ZH, valid = node && g.valid(i, j);
  const float2 zero2 = make_float2(0.f, 0.f);
  float2 d = zero2, b = zero2;
  if (valid) d = tile_d<SRC>(a, i, j);
  const bool own = valid && zx >= 2 && zx < 2 + TILE_X && zy >= 2 && zy < 2 + TILE_Y;
  double2 rd = make_double2(0.0, 0.0), qd = rd;
  pdl_wait_prior();
  const bool done = a.sc != nullptr && a.gate && a.sc->done != RUNNING;
  if (valid) b = a.b[g.at(i, j)];
  if constexpr (DOT) {
    if (own) {
      rd = a.rdot[g.at(i, j)];
      if (a.qdot != nullptr) qd = a.qdot[g.at(i, j)];
    }
  }
  // z = v + P z_c at node t (mto_sweep2.cuh's interpolation).
  float2 v = zero2;
  {
    const int ii = x0 + t % NW, jj = y0 + t / NW;
    if (t < NW * NH && g.valid(ii, jj)) {
      v = a.v[g.at(ii, jj)];
      const long long kc = gc.at(ii >> 1, jj >> 1);
      const long long up = (jj & 1) ? gc.pitch : 0;
      const float2 c00 = a.zc[kc], c01 = a.zc[kc + up], c10 = a.zc[kc + 1], c11 = a.zc[kc + 1 + up];
      const float2 cy0 = make_float2(0.5f * (c00.x + c01.x), 0.5f * (c00.y + c01.y));
      const float2 cy1 = make_float2(0.5f * (c10.x + c11.x), 0.5f * (c10.y + c11.y));
      v = (ii & 1) ? make_float2(v.x + 0.5f * (cy0.x + cy1.x), v.y + 0.5f * (cy0.y + cy1.y))
                   : make_float2(v.x + cy0.x, v.y + cy0.y);
    }
  }
  if (done) return;  // uniform over the grid
  if (t < NW * NH) z[t] = v;
  __syncthreads();
  const int c = ey * NW + ex;
  if (elem) f.template put<SRC>(a, er, t, z[c], z[c + 1], z[c + NW], z[c + NW + 1]);
  __syncthreads();
  const int zn = zy * NW + zx, en = zy * EW + zx;
  float2 z2 = zero2;
  if (node) {
    z2 = fma2(d, sub2(b, f.at_node(en)), z[zn]);
    z[zn] = z2;
  }
  __syncthreads();
  if (elem && ex >= 1 && ex < EW - 1 && ey >= 1 && ey < EH - 1)
    f.template put<SRC>(a, er, t, z[c], z[c + 1], z[c + NW], z[c + NW + 1]);
  __syncthreads();
  double dot0 = 0.0, dot1 = 0.0;
  if (own) {
    const float2 z3 = fma2(d, sub2(b, f.at_node(en)), z2);
    if (SRC == SRC_FINEBF && !DOT && a.dout != nullptr)
      a.dout[(long long)j * (g.nx + 1) + i] = make_double2(z3.x, z3.y);
    else
      a.out[g.at(i, j)] = z3;
    if constexpr (DOT) {
      const double zx64 = to_f64(z3.x), zy64 = to_f64(z3.y);
      dot0 = fma(zx64, rd.x, zy64 * rd.y);
      if (a.qdot != nullptr) dot1 = fma(zx64, qd.x, zy64 * qd.y);
    }
  }
  if constexpr (DOT)
    block_reduce_finish<SWEEP_NT>(dot0, dot1, a.partials, a.ticket, a.sc, a.finish, a.out_value, a.tag);
}

}  // namespace mto
