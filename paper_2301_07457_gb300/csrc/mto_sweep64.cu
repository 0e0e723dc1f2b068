// float64 instantiations of the sweeps (fixed-point element factors on the
// finest and the coarse levels), and the launch-shape rule shared by all
// sweeps.  The float64 kernels are bound by integer issue, so one step of load
// lookahead suffices (two: K p at 2048^2 117 -> 137 us, for the registers).
#include "mto_launch.h"

namespace mto {

SweepShape sweep_shape(const Grid& g, int mode, int target_warps, int cols, int spread) {
  SweepShape sh;
  if (mode == MODE_PRE2) {
    // 29 output coarse columns per warp, coarse rows per task as for the
    // restriction sweep.
    const int nxc = g.nx / 2, nyc = g.ny / 2;
    sh.nstrips = (nxc + 1 + PRE2_CSTRIDE - 1) / PRE2_CSTRIDE;
    const int want = target_warps / sh.nstrips > 1 ? target_warps / sh.nstrips : 1;
    int hc = (nyc + 1 + want - 1) / want;
    hc = hc < 1 ? 1 : (hc > 32 ? 32 : hc);
    sh.H = 2 * hc;
    sh.nchunks = (nyc + 1 + hc - 1) / hc;
  } else if (mode == MODE_POST2) {
    // 60 output columns per warp, rows as for a smoothing sweep.
    sh.nstrips = (g.nx + 1 + POST2_STRIDE - 1) / POST2_STRIDE;
    const int want = target_warps / sh.nstrips > 1 ? target_warps / sh.nstrips : 1;
    int h = (g.ny + 1 + want - 1) / want;
    h = h < 1 ? 1 : (h > 64 ? 64 : h);
    sh.H = h;
    sh.nchunks = (g.ny + 1 + h - 1) / h;
  } else if (mode == MODE_RESTRICT) {
    // Coarse columns per warp: 14 (one column per lane) or 30 (two).
    const int cstride = cols == 2 ? SWEEP2_RSTRIDE / 2 : SWEEP_RSTRIDE / 2;
    const int nxc = g.nx / 2, nyc = g.ny / 2;
    sh.nstrips = (nxc + 1 + cstride - 1) / cstride;
    const int want = target_warps / sh.nstrips > 1 ? target_warps / sh.nstrips : 1;
    int hc = (nyc + 1 + want - 1) / want;
    hc = hc < 1 ? 1 : (hc > 32 ? 32 : hc);
    sh.H = 2 * hc;
    sh.nchunks = (nyc + 1 + hc - 1) / hc;
  } else {
    // Output node columns per warp: 30 ([30 s, 30 s + 29]) or 62 ([62 s - 1, 62 s + 60]).
    sh.nstrips = cols == 2 ? (g.nx + 2 + SWEEP2_STRIDE - 1) / SWEEP2_STRIDE
                           : (g.nx + 1 + SWEEP_STRIDE - 1) / SWEEP_STRIDE;
    const int want = target_warps / sh.nstrips > 1 ? target_warps / sh.nstrips : 1;
    // One row per task on small levels: with the halo step, two steps whose
    // loads all fit the lookahead ring, so the sweep costs one memory round
    // trip instead of two.
    int h = (g.ny + 1 + want - 1) / want;
    h = h < 1 ? 1 : (h > 64 ? 64 : h);
    sh.H = h;
    sh.nchunks = (g.ny + 1 + h - 1) / h;
  }
  const long long warps = (long long)sh.nstrips * sh.nchunks;
  long long per_block = SWEEP_NT / 32;
  if (spread > 0 && (warps + spread - 1) / spread < per_block) per_block = (warps + spread - 1) / spread;
  sh.nthreads = 32 * (int)per_block;
  sh.nblocks = (int)((warps + per_block - 1) / per_block);
  return sh;
}


// Small grids, where a marching task would have one or two rows, take the
// kernel that completes a row per warp (its two element rows side by side):
// per node it costs what two-row tasks do, and its chain is a third as long.
// PCG iterations: 256^2 168 -> 115 us, 1024^2 (coarse levels only) 446 -> 391
// us; a 64^2 solve 3.00 -> 1.92 ms.
constexpr int SPLIT_MAX_H = 2;

template <int SRC, int MODE, bool DOT, typename ZT>
static cudaError_t go(SweepParams<double> p, int tw, int num_sms, cudaStream_t s) {
  void (*kernel)(SweepParams<double>) = fsweep_kernel<SRC, MODE, DOT, ZT, 1>;
  if (tw <= 0) {
    static const int wave = full_wave_warps(kernel, num_sms);  // same for every device of a run
    tw = wave;
  }
  const SweepShape sh = sweep_shape(p.g, MODE, tw, SWEEP_COLS_F64, num_sms);
  p.nstrips = sh.nstrips;
  p.nchunks = sh.nchunks;
  p.H = sh.H;
  int nblocks = sh.nblocks, nthreads = sh.nthreads;
  if (sh.H <= SPLIT_MAX_H) {
    const bool restrict = MODE == MODE_RESTRICT;
    const int stride = restrict ? SPLIT_RSTRIDE : SPLIT_STRIDE;
    kernel = fsplit_kernel<SRC, MODE, DOT, ZT>;
    p.nstrips = (p.g.nx + 1 + stride - 1) / stride;
    p.nchunks = restrict ? p.gc.ny + 1 : p.g.ny + 1;
    const int tasks = p.nstrips * p.nchunks;
    int per_block = (tasks + num_sms - 1) / num_sms;
    per_block = per_block > SWEEP_NT / 32 ? SWEEP_NT / 32 : per_block;
    nblocks = restrict ? tasks : (tasks + per_block - 1) / per_block;
    nthreads = 32 * (restrict ? SPLIT_RWARPS : per_block);
  }
  return launch_pdl(kernel, nblocks, nthreads, 0, s, p);
}

static int tiles_across(const Grid& g) { return g.nx / TILE_X + 1; }
static long long tile_count(const Grid& g) { return (long long)tiles_across(g) * (g.ny / TILE_Y + 1); }

bool float64_tiles(const Grid& g, int target_warps, int num_sms) {
  return tile_count(g) <= FTILES_PER_SM * num_sms && (target_warps <= 0 || target_warps >= num_sms);
}

static cudaError_t go_tiles(void (*kernel)(SweepParams<double>), SweepParams<double> p, cudaStream_t s) {
  p.nstrips = tiles_across(p.g);
  return launch_pdl(kernel, (int)tile_count(p.g), SWEEP_NT, 0, s, p);
}

template <>
cudaError_t launch_sweep<double>(int src, int mode, bool dot, bool zfloat, SweepParams<double> p,
                                 int tw, int num_sms, cudaStream_t s) {
  if (src == SRC_FINE64) {
    switch (mode) {
      case MODE_APPLY: return go<SRC_FINE64, MODE_APPLY, false, double2>(p, tw, num_sms, s);
      case MODE_RESID: return go<SRC_FINE64, MODE_RESID, false, double2>(p, tw, num_sms, s);
      case MODE_KP:
        return zfloat ? go<SRC_FINE64, MODE_KP, false, float2>(p, tw, num_sms, s)
                      : go<SRC_FINE64, MODE_KP, false, double2>(p, tw, num_sms, s);
      case MODE_SMOOTH:
        return dot ? go<SRC_FINE64, MODE_SMOOTH, true, double2>(p, tw, num_sms, s)
                   : go<SRC_FINE64, MODE_SMOOTH, false, double2>(p, tw, num_sms, s);
      case MODE_SMOOTH0: return go<SRC_FINE64, MODE_SMOOTH0, false, double2>(p, tw, num_sms, s);
      case MODE_PSMOOTH:
        return dot ? go<SRC_FINE64, MODE_PSMOOTH, true, double2>(p, tw, num_sms, s)
                   : go<SRC_FINE64, MODE_PSMOOTH, false, double2>(p, tw, num_sms, s);
      case MODE_RESTRICT: return go<SRC_FINE64, MODE_RESTRICT, false, double2>(p, tw, num_sms, s);
      case MODE_PRE2: return go_tiles(ftile_pre2_kernel<SRC_FINE64>, p, s);
      case MODE_POST2:
        return go_tiles(dot ? ftile_post2_kernel<SRC_FINE64, true> : ftile_post2_kernel<SRC_FINE64, false>, p, s);
      default: return cudaErrorInvalidValue;
    }
  }
  if (src == SRC_COARSE) {
    switch (mode) {
      case MODE_APPLY: return go<SRC_COARSE, MODE_APPLY, false, double2>(p, tw, num_sms, s);
      case MODE_SMOOTH: return go<SRC_COARSE, MODE_SMOOTH, false, double2>(p, tw, num_sms, s);
      case MODE_SMOOTH0: return go<SRC_COARSE, MODE_SMOOTH0, false, double2>(p, tw, num_sms, s);
      case MODE_PSMOOTH: return go<SRC_COARSE, MODE_PSMOOTH, false, double2>(p, tw, num_sms, s);
      case MODE_RESTRICT: return go<SRC_COARSE, MODE_RESTRICT, false, double2>(p, tw, num_sms, s);
      case MODE_PRE2: return go_tiles(ftile_pre2_kernel<SRC_COARSE>, p, s);
      case MODE_POST2: return go_tiles(ftile_post2_kernel<SRC_COARSE, false>, p, s);
      default: return cudaErrorInvalidValue;
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace mto
