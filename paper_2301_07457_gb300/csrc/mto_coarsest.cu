// Explicit inverse of the coarsest matrix K_0 (Alg. 1 on the coarsest grid,
// Alg. 3's direct solve) by nested dissection over its node rows.
//
// In the row-major DOF numbering K_0 is block tridiagonal: J block rows (the
// free node rows) of m DOFs, neighbours coupled by sparse blocks B_j = K_0[j,
// j - 1] (three nodes wide).  A range of block rows [lo, hi) is split by its
// middle row s into two ranges that do not touch each other; with their
// inverses A1^-1 and A2^-1 known,
//   S   = K_ss - B_s G1 B_s^T - B_{s+1}^T G2 B_{s+1}
//         (G1: last diagonal block of A1^-1, G2: first one of A2^-1),
//   V_r = A1^-1[r, s-1] B_s^T or A2^-1[r, s+1] B_{s+1}, W = -V S^-1,
//   A^-1 = [A1^-1 + V S^-1 V^T in both parts and between them, W; W^T, S^-1],
// in which every correction of a diagonal part is positive semidefinite.
// With V = -I on the rows of s this is one formula, old - W V^T, over all
// rows of the range.
//
// Why: a band factorisation followed by substitutions is a chain of 2 n steps
// (n = 544 pivots on a 16 x 16 grid, 0.65 us each on one SM, then as many
// substitution steps: 354 + 265 us); here the chain is m pivots per level of
// the tree, all ranges of one depth run side by side, and the products, which
// hold the FP64 work, spread over the chip.
//
// The ranges follow from the depth and a path by halving, so no tables are
// kept.  Per depth, deepest first, three launches: (1) one block per range
// forms S and inverts it while other blocks form V, (2) W, (3) the update of
// K_0^-1 by 16 x 16 tiles of its lower triangle, mirrored.
#include "mto_fixed.cuh"
#include "mto_launch.h"

namespace mto {

namespace {

struct BlockRows {
  int n, m, J, bw;   // n = m J; bw: half bandwidth of the band storage
  const double* Kb;  // lower band, Kb[r (bw + 1) + d] = K_0[r][r - d]
  double* S;         // n x m: S^-1 of the range whose separator is the row's block
  double* V;         // n x m
  double* W;         // n x m
  double* Kinv;      // n x n
  int* err;
};

// The range of depth `depth` that holds block row j, or the one with path
// bits `path` (j < 0); false if j is a separator of a shallower range or the
// path ends in an empty one.
struct Range {
  int lo, s, hi;
};
__device__ __forceinline__ bool range_of(int J, int depth, int j, unsigned path, Range& r) {
  int lo = 0, hi = J;
  for (int d = 0; d < depth; ++d) {
    const int mid = (lo + hi) >> 1;
    bool right;
    if (j >= 0) {
      if (j == mid) return false;
      right = j > mid;
    } else {
      right = (path >> (depth - 1 - d)) & 1u;
    }
    if (right) lo = mid + 1;
    else hi = mid;
    if (lo >= hi) return false;
  }
  r.lo = lo;
  r.hi = hi;
  r.s = (lo + hi) >> 1;
  return true;
}

// K_0[r][c] from the band.
__device__ __forceinline__ double k0(const BlockRows& a, int r, int c) {
  const int hi = max(r, c), d = hi - min(r, c);
  return d <= a.bw ? a.Kb[(size_t)hi * (a.bw + 1) + d] : 0.0;
}

// DOF b of a block row is coupled to the DOFs first(b) .. first(b) + 5 of its
// neighbours: the three nodes around its own, where they exist.
constexpr int NCOUPLE = 6;
__device__ __forceinline__ int couple_first(int b) { return ((b >> 1) - 1) * 2; }
__device__ __forceinline__ double couple(const BlockRows& a, int q, int s, int b, int e) {  // K[q, l][s, b]
  const int l = couple_first(b) + e;
  return l >= 0 && l < a.m ? k0(a, q * a.m + l, s * a.m + b) : 0.0;
}
__device__ __forceinline__ int couple_at(int m, int b, int e) { return min(max(couple_first(b) + e, 0), m - 1); }

constexpr int SEP_NT = 224;   // threads that hold S: seven warps, so that with the
constexpr int SEP_BLOCK = SEP_NT + 32;  // diagonal's every scheduler has two (V blocks use them all)
constexpr int V_ROWS = 8;     // rows per V block
constexpr int W_ROWS = 2;     // rows per W block
constexpr int W_NT = 64 * W_ROWS;
constexpr int TILE = 16;      // update tiles
constexpr int TILE_NT = 128;  // 2 x 2 entries per thread, even and odd columns of W and V apart

// V rows [r0, r0 + V_ROWS) of the ranges of this depth.
__device__ __forceinline__ void form_v(const BlockRows& a, int depth, int r0) {
  const int m = a.m;
  for (int t = threadIdx.x; t < V_ROWS * m; t += SEP_BLOCK) {
    const int r = r0 + t / m, b = t % m;
    if (r >= a.n) return;
    const int j = r / m;
    Range g;
    if (!range_of(a.J, depth, j, 0u, g) || g.hi - g.lo == 1) continue;
    double v = 0.0;
    if (j == g.s) {
      v = (r - j * m) == b ? -1.0 : 0.0;
    } else {
      // Row r of the part's inverse at the block next to s, times K[block, s].
      const int q = j < g.s ? g.s - 1 : g.s + 1;
      const double* row = a.Kinv + (size_t)r * a.n + (size_t)q * m;
#pragma unroll
      for (int e = 0; e < NCOUPLE; ++e) v = fma(row[couple_at(m, b, e)], couple(a, q, g.s, b, e), v);
    }
    a.V[(size_t)r * m + b] = v;
  }
}

// S of the range, inverted in place by symmetric sweeps on its lower triangle
// (S -> -S^-1): pivot p = a_kk turns a_ij into a_ij - a_ik a_jk / p, column k
// into a_ik / p and a_kk into -1 / p.  The triangle lives in the registers of
// SEP_NT threads (E entries each); per pivot the column and its quotients pass
// through shared memory.  An extra warp keeps a second copy of the diagonal,
// so that the next pivot's reciprocal is formed while the others update.  Two
// barriers per pivot; the FP64 pipe bounds a pivot (three to six FMAs of two
// warps per scheduler at 64 clocks, and a latency of about 140): 25 -> 19 us
// for m = 34 against the triangle in shared memory.
template <int E>
__device__ __forceinline__ void form_s(const BlockRows& a, const Range& g, double* sm) {
  const int m = a.m, tid = threadIdx.x;
  double* G1 = sm;               // last diagonal block of the left part's inverse
  double* G2 = G1 + m * m;       // first one of the right part's
  double* X1 = G2 + m * m;       // G1 B_s^T
  double* X2 = X1 + m * m;       // G2 B_{s+1}
  double* C1 = X2 + m * m;       // couplings [b][e] to the left and the right
  double* C2 = C1 + NCOUPLE * m;
  double* u = C2 + NCOUPLE * m;  // pivot column, two buffers
  double* v = u + 2 * m;         // the same over the pivot
  double* diag = v + m;
  __shared__ double rec[2];
  const bool left = g.s > g.lo, right = g.s + 1 < g.hi;
  const int base = g.s * m;
  for (int t = tid; t < m * m; t += SEP_BLOCK) {
    const int i = t / m, b = t % m;
    G1[t] = left ? a.Kinv[(size_t)(base - m + i) * a.n + base - m + b] : 0.0;
    G2[t] = right ? a.Kinv[(size_t)(base + m + i) * a.n + base + m + b] : 0.0;
  }
  for (int t = tid; t < NCOUPLE * m; t += SEP_BLOCK) {
    const int b = t / NCOUPLE, e = t % NCOUPLE;
    C1[t] = left ? couple(a, g.s - 1, g.s, b, e) : 0.0;
    C2[t] = right ? couple(a, g.s + 1, g.s, b, e) : 0.0;
  }
  __syncthreads();
  if (left || right)
    for (int t = tid; t < m * m; t += SEP_BLOCK) {
      const int i = t / m, b = t % m;
      double x = 0.0, y = 0.0;
#pragma unroll
      for (int e = 0; e < NCOUPLE; ++e) {
        const int l = i * m + couple_at(m, b, e);
        x = fma(G1[l], C1[b * NCOUPLE + e], x);
        y = fma(G2[l], C2[b * NCOUPLE + e], y);
      }
      X1[t] = x;
      X2[t] = y;
    }
  __syncthreads();
  const int np = m * (m + 1) / 2;
  const bool worker = tid < SEP_NT;
  double A[E];
  int ij[E];  // i << 16 | j, i >= j
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int t = tid + e * SEP_NT;
    A[e] = 0.0;
    ij[e] = -1;
    if (!worker || t >= np) continue;
    int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= t) ++i;
    while (i * (i + 1) / 2 > t) --i;
    const int j = t - i * (i + 1) / 2;
    ij[e] = i << 16 | j;
    double x = k0(a, base + i, base + j), y = 0.0;
    if (left || right) {
#pragma unroll
      for (int c = 0; c < NCOUPLE; ++c) {
        const int l = couple_at(m, i, c) * m + j;
        x = fma(-C1[i * NCOUPLE + c], X1[l], x);
        y = fma(-C2[i * NCOUPLE + c], X2[l], y);
      }
    }
    A[e] = x + y;
    if (j == 0) u[i] = A[e];
    if (i == j) diag[i] = A[e];
  }
  __syncthreads();
  auto pivot = [&](double d, int k) {
    // Positive and between 2^-996 and 2^996, by the exponent (no comparison on
    // the FP64 pipe, whose latency the chain of pivots would see).
    if ((unsigned)(__double2hiint(d) - 0x01b00000) < 0x7c800000u) {
      rec[k & 1] = fx_reciprocal(d);
      return;
    }
    if (!(d > 0.0) || !(d < 1.0e300)) {
      *a.err = 1;
      d = 1.0;
    }
    rec[k & 1] = 1.0 / d;
  };
  constexpr int ND = (MAX_BLOCK_ROW + 31) / 32;
  double dg[ND];  // the extra warp's diagonal: entries lane, lane + 32, ...
  const int lane = tid & 31;
#pragma unroll
  for (int q = 0; q < ND; ++q) dg[q] = lane + 32 * q < m ? diag[lane + 32 * q] : 1.0;
  if (tid == SEP_NT) pivot(dg[0], 0);
  __syncthreads();
  for (int k = 0; k < m; ++k) {
    const double r = rec[k & 1];
    double* uk = u + (k & 1) * m;
    double* un = u + ((k + 1) & 1) * m;
    // With u_k = -1 and v_k = -r the pivot row, column and entry are -u_i v_j
    // (or its mirror image) too.
    if (tid < m) {
      v[tid] = tid == k ? -r : uk[tid] * r;
      if (tid == k) uk[tid] = -1.0;
    }
    __syncthreads();
    if (worker) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        if (ij[e] < 0) continue;
        const int i = ij[e] >> 16, j = ij[e] & 0xffff;
        // i >= j: in the pivot row (i = k) the -1 is in u_i, in the pivot
        // column (j = k) the -r in v_j.
        A[e] = fma(-uk[i], v[j], i == k || j == k ? 0.0 : A[e]);
        if (i == k + 1) un[j] = A[e];
        else if (j == k + 1) un[i] = A[e];
      }
    } else {
#pragma unroll
      for (int q = 0; q < ND; ++q) {
        const int d = lane + 32 * q;
        if (32 * q < m && d > k && d < m) {
          dg[q] = fma(-uk[d], v[d], dg[q]);
          if (d == k + 1) pivot(dg[q], k + 1);
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (ij[e] >= 0) X1[(ij[e] >> 16) * m + (ij[e] & 0xffff)] = A[e];
  __syncthreads();
  const bool leaf = g.hi - g.lo == 1;
  for (int t = tid; t < m * m; t += SEP_BLOCK) {
    const int i = t / m, j = t % m;
    const double x = -(i >= j ? X1[i * m + j] : X1[j * m + i]);
    a.S[(size_t)(base + i) * m + j] = x;
    if (leaf) a.Kinv[(size_t)(base + i) * a.n + base + j] = x;
  }
}

template <int E> __global__ void __launch_bounds__(SEP_BLOCK) separator_kernel(BlockRows a, int depth) {
  pdl_wait();
  extern __shared__ double dyn[];
  const int nranges = 1 << depth;
  if ((int)blockIdx.x < nranges) {
    Range g;
    if (range_of(a.J, depth, -1, blockIdx.x, g)) form_s<E>(a, g, dyn);
  } else {
    form_v(a, depth, ((int)blockIdx.x - nranges) * V_ROWS);
  }
}

// W = -V S^-1: W_ROWS rows per block, 64 threads per row.
__global__ void __launch_bounds__(W_NT) separator_column_kernel(BlockRows a, int depth) {
  pdl_wait();
  __shared__ double vrow[W_ROWS][MAX_BLOCK_ROW];
  const int m = a.m, u = threadIdx.x / 64, lane = threadIdx.x % 64;
  const int r = blockIdx.x * W_ROWS + u;
  Range g;
  const bool active = r < a.n && range_of(a.J, depth, r / m, 0u, g) && g.hi - g.lo > 1;  // uniform over a row's warps
  if (active)
    for (int l = lane; l < m; l += 64) vrow[u][l] = a.V[(size_t)r * m + l];
  __syncthreads();
  if (!active) return;
  const double* s = a.S + (size_t)g.s * m * m;
  for (int b = lane; b < m; b += 64) {
    double w0 = 0.0, w1 = 0.0;
#pragma unroll 16
    for (int l = 0; l < m; l += 2) {  // m is even
      w0 = fma(-vrow[u][l], s[(size_t)l * m + b], w0);
      w1 = fma(-vrow[u][l + 1], s[(size_t)(l + 1) * m + b], w1);
    }
    a.W[(size_t)r * m + b] = w0 + w1;
  }
}

// K_0^-1 of every range of this depth: old - W V^T (old: zero between the two
// parts and on the separator), one 16 x 16 tile of the lower triangle per
// block, mirrored.
__global__ void __launch_bounds__(TILE_NT) range_update_kernel(BlockRows a, int depth) {
  pdl_wait();
  // Tile (I, K), K <= I, from the linear index.
  const int t = blockIdx.x;
  int I = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((I + 1) * (I + 2) / 2 <= t) ++I;
  while (I * (I + 1) / 2 > t) --I;
  const int K = t - I * (I + 1) / 2;
  const int m = a.m, n = a.n;
  const int half = threadIdx.x >> 6, tx = threadIdx.x & 7, ty = (threadIdx.x & 63) >> 3;
  int r[2], c[2], side_r[2], side_c[2], lo_r[2], lo_c[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    r[u] = I * TILE + ty + 8 * u;
    c[u] = K * TILE + tx + 8 * u;
    // lo: identifies the range (-1: none at this depth); side: -1, 0, 1.
    Range g;
    lo_r[u] = lo_c[u] = -1;
    side_r[u] = side_c[u] = 0;
    if (r[u] < n && range_of(a.J, depth, r[u] / m, 0u, g) && g.hi - g.lo > 1) {
      lo_r[u] = g.lo;
      const int j = r[u] / m;
      side_r[u] = j < g.s ? -1 : (j > g.s ? 1 : 0);
    }
    if (c[u] < n && range_of(a.J, depth, c[u] / m, 0u, g) && g.hi - g.lo > 1) {
      lo_c[u] = g.lo;
      const int j = c[u] / m;
      side_c[u] = j < g.s ? -1 : (j > g.s ? 1 : 0);
    }
  }
  bool any = false;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) any = any || (lo_r[u] >= 0 && lo_r[u] == lo_c[w]);
  if (!__syncthreads_or(any)) return;
  // W of the tile's rows and V of its columns (row pitch odd: no bank conflicts
  // down a column of the tile).
  extern __shared__ double dyn[];
  const int pitch = m + 1;
  double *ws = dyn, *vs = dyn + TILE * pitch;
  for (int q = threadIdx.x; q < TILE * m; q += TILE_NT) {
    const int i = q / m, k = q - i * m;
    const int ri = I * TILE + i, ci = K * TILE + i;
    ws[i * pitch + k] = ri < n ? a.W[(size_t)ri * m + k] : 0.0;
    vs[i * pitch + k] = ci < n ? a.V[(size_t)ci * m + k] : 0.0;
  }
  __syncthreads();
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  const double *w0p = ws + ty * pitch, *w1p = w0p + 8 * pitch, *v0p = vs + tx * pitch, *v1p = v0p + 8 * pitch;
#pragma unroll 4
  for (int k = half; k < m; k += 2) {
    const double w0 = w0p[k], w1 = w1p[k], v0 = v0p[k], v1 = v1p[k];
    acc[0][0] = fma(-w0, v0, acc[0][0]);
    acc[0][1] = fma(-w0, v1, acc[0][1]);
    acc[1][0] = fma(-w1, v0, acc[1][0]);
    acc[1][1] = fma(-w1, v1, acc[1][1]);
  }
  __syncthreads();
  // The odd columns' sums join the even ones'.
  double* odd = dyn;
  if (half == 1) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int w = 0; w < 2; ++w) odd[(threadIdx.x & 63) + 64 * (2 * u + w)] = acc[u][w];
  }
  __syncthreads();
  if (half == 1) return;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) acc[u][w] += odd[threadIdx.x + 64 * (2 * u + w)];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      if (lo_r[u] < 0 || lo_r[u] != lo_c[w] || c[w] > r[u]) continue;
      double* dst = a.Kinv + (size_t)r[u] * n + c[w];
      const double old = side_r[u] != 0 && side_r[u] == side_c[w] ? *dst : 0.0;
      const double x = old + acc[u][w];
      *dst = x;
      if (c[w] != r[u]) a.Kinv[(size_t)c[w] * n + r[u]] = x;
    }
}

size_t update_smem(int m) { return sizeof(double) * (size_t)(2 * TILE * (m + 1) > 256 ? 2 * TILE * (m + 1) : 256); }

size_t separator_smem(int m) {
  return sizeof(double) * (4 * (size_t)m * m + (2 * NCOUPLE + 4) * m);
}

// Entries of S per thread: the fewest that hold m (m + 1) / 2 of them.
using SeparatorKernel = void (*)(BlockRows, int);
SeparatorKernel separator_for(int m) {
  const int np = m * (m + 1) / 2;
  if (np <= 3 * SEP_NT) return separator_kernel<3>;
  if (np <= 6 * SEP_NT) return separator_kernel<6>;
  if (np <= 10 * SEP_NT) return separator_kernel<10>;
  static_assert(MAX_BLOCK_ROW * (MAX_BLOCK_ROW + 1) / 2 <= 15 * SEP_NT, "widest block row");
  return separator_kernel<15>;
}

}  // namespace

bool block_inverse_fits(int n, int m) { return m >= 2 && m <= MAX_BLOCK_ROW && n >= m && n % m == 0; }

cudaError_t prepare_block_inverse(int m) {
  return raise_max_dynamic_smem((const void*)separator_for(m), separator_smem(m));
}

cudaError_t launch_block_inverse(int n, int m, int bw, const double* Kb, double* work, double* Kinv, int* err_flag,
                                 cudaStream_t s, long long* launches) {
  BlockRows a = {n, m, n / m, bw, Kb, work, work + (size_t)n * m, work + 2 * (size_t)n * m, Kinv, err_flag};
  int depth = 0;
  for (int size = a.J; size > 1; size >>= 1) ++depth;
  const int nt = (n + TILE - 1) / TILE, ntiles = nt * (nt + 1) / 2;
  for (int d = depth; d >= 0; --d) {
    // Ranges of the deepest level are single rows: no V.
    const int vblocks = d == depth ? 0 : (n + V_ROWS - 1) / V_ROWS;
    cudaError_t e = launch_pdl(separator_for(m), (1 << d) + vblocks, SEP_BLOCK, separator_smem(m), s, a, d);
    if (e != cudaSuccess) return e;
    *launches += 1;
    if (d == depth) continue;
    e = launch_pdl(separator_column_kernel, (n + W_ROWS - 1) / W_ROWS, W_NT, 0, s, a, d);
    if (e != cudaSuccess) return e;
    e = launch_pdl(range_update_kernel, ntiles, TILE_NT, update_smem(m), s, a, d);
    if (e != cudaSuccess) return e;
    *launches += 2;
  }
  return cudaSuccess;
}

}  // namespace mto
