// Row passes: variant selection and launches (instantiated per precision by fft_rows_*.cu).
#pragma once

#include "fft_kernels.cuh"

namespace dps {

template <typename T>
bool fft_rows_allow() {
  return allow_smem(row_r2c_kernel<T, false>) && allow_smem(row_c2r_kernel<T, false>) &&
         allow_smem(row_r2c_kernel<T, true>) && allow_smem(row_c2r_kernel<T, true>) && allow_smem(row_r2c_reg_kernel<T, false>) &&
         allow_smem(row_r2c_reg_kernel<T, true>) && allow_smem(row_c2r_reg_kernel<T, false>) &&
         allow_smem(row_c2r_reg_kernel<T, true>);
}

namespace {

// Share of the lanes that a block issues which carry butterflies, over all stages, with 2^lb row pairs.
double lane_use(const FftPlan& fp, int lb) {
  const int th = fft_threads(fp.n << lb);
  double work = 0.0, issued = 0.0;
  for (int s = 0; s < fp.nstages; ++s) {
    const int bf = (fp.n << lb) / fp.radix[s], full = bf / th * th, rest = bf - full;
    work += (double)bf * fp.radix[s];
    issued += (double)(full + (rest + 31) / 32 * 32) * fp.radix[s];
  }
  return work / issued;
}

// log2 of the row pairs that a block of the shared-memory-staged passes transforms together (us of the
// forward pass on 33 planes FP64 at 1, 2, 4 and 8 pairs, 97 planes float).
//  - FP64: its instructions pay for idle lanes, so more pairs wherever they fill more of them, in at most 160
//    threads; four rather than two below 1024 points, where the barriers are then shared by more work.
//      64: 80 45 35 29   128: 182 106 80 84   210: 512 303 274 285   256: 559 344 309 311
//      384: 823 852 756 825   675: 4012 3446 3689   1024: 5831 6509 6082
//  - float: fours for short rows that leave a quarter of the lanes idle; longer rows, whose single-warp
//    blocks run their barriers for free and whose epilogue reads without bank conflicts, stay single.
//    (at 1 and 4 pairs) 64: 21 14   108: 33 31   160: 51 46   192: 68 55   200: 76 86   256: 93 101   384: 171 222
// No more than leaves two units for every SM when three fields are transformed.
template <typename T>
int row_batch(const Geometry& g, const FftPlan& fp) {
  int lb = 0;
  if (sizeof(T) == 8) {
    for (int l = 1; l <= 3 && (fp.n << l) <= 160 * kFftPer; ++l) {
      const double ratio = lane_use(fp, l) / lane_use(fp, lb);
      if (ratio > 1.04 || (lb == 1 && ratio > 0.999 && (fp.n << l) <= 1024)) lb = l;
    }
  } else if (fp.n <= 192 && lane_use(fp, 0) < 0.75) {
    lb = 2;
  }
  while (lb > 0 && 3ll * g.nz * ((g.ny + (2 << lb) - 1) >> (lb + 1)) < 2 * 152) --lb;
  return lb;
}

}  // namespace

template <typename T>
int fft_set_row_variant(Plan& p, int reg) {
  if (reg) {
    if (!reg_fits<T>(p.fxr, 0)) return 0;
    const int th = reg_threads(p.fxr, 0);
    const size_t sm = reg_smem<T>(p.g.nx);
    p.fft_reg[0] = 1;
    p.fft_grid[0] = r2c_split_ok(p.fxr) ? resident_grid(row_r2c_reg_kernel<T, true>, th, sm, p.device)
                                         : resident_grid(row_r2c_reg_kernel<T, false>, th, sm, p.device);
    p.fft_grid[1] = c2r_pair_ok(p.fxr) ? resident_grid(row_c2r_reg_kernel<T, true>, th, sm, p.device)
                                        : resident_grid(row_c2r_reg_kernel<T, false>, th, sm, p.device);
    return 1;
  }
  const int lb = row_batch<T>(p.g, p.fx);
  const size_t r2c = row_r2c_smem<T>(p.g, lb), c2r = row_c2r_smem<T>(p.g, lb);
  const int trow = fft_threads(p.g.nx << lb);
  if (trow > kFftMaxThreads || r2c > 220 * 1024 || c2r > 220 * 1024) return 0;
  p.fft_reg[0] = 0;
  p.row_lb = lb;
  p.fft_grid[0] = resident_grid(lb ? row_r2c_kernel<T, true> : row_r2c_kernel<T, false>, trow, r2c, p.device);
  p.fft_grid[1] = resident_grid(lb ? row_c2r_kernel<T, true> : row_c2r_kernel<T, false>, trow, c2r, p.device);
  return 1;
}

// Default shapes, from measurements on rollers and slit grids (3072^2, 768^2, 384^2): the
// register-staged row pass only for long float rows whose stages keep at least 3/4 of the block
// busy (3072 = 16 x 16 x 12: 10 % faster than the shared-memory-staged pass; 768 = 16 x 16 x 3 and
// 384 = 16 x 12 x 2 leave most threads idle in the radix-16 stages and run 1.5-2.5x slower, as does
// FP64).  Columns: the width of a block's per-row piece decides (3072 rows, mixed: 2 columns
// shared-memory-staged 18.1 ms per pass pair, 4 columns prefetched register-staged 14.5 ms, the
// latter at 2 columns 23.6 ms), so the prefetched register-staged pass where its two buffers fit a
// wider block than the staged pass's three, else the staged pass at its widest; the register-staged
// pass without prefetch (loads exposed; 1.3-1.5x slower at equal width) only by hand or autotuning.
template <typename T>
bool reg_rows_default(const FftPlan& fp) {
  if (sizeof(T) != 4 || fp.n < 2048 || !reg_fits<T>(fp, 0)) return false;
  int rmin = fp.radix[0], rmax = fp.radix[0];
  for (int s = 1; s < fp.nstages; ++s) {
    rmin = std::min(rmin, fp.radix[s]);
    rmax = std::max(rmax, fp.radix[s]);
  }
  return 3 * rmax <= 4 * rmin;
}

template <typename T>
bool fft_rows_default(Plan& p) {
  const bool rr = reg_rows_default<T>(p.fxr);
  return fft_set_row_variant<T>(p, rr ? 1 : 0) || fft_set_row_variant<T>(p, rr ? 0 : 1);
}

template <typename T>
void launch_fft_rows(const Plan& p, int dir, cudaStream_t s) {
  const Geometry& g = p.g;
  const cplx<T>* twx = reinterpret_cast<const cplx<T>*>(p.tab.twx);
  if (p.fft_reg[0]) {
    const int th = reg_threads(p.fxr, 0);
    const size_t sm = reg_smem<T>(g.nx);
    T* grid = reinterpret_cast<T*>(p.grid);
    if (dir < 0 && r2c_split_ok(p.fxr))
      row_r2c_reg_kernel<T, true><<<p.fft_grid[0], th, sm, s>>>(g, p.fxr, twx, grid, p.zrange);
    else if (dir < 0)
      row_r2c_reg_kernel<T, false><<<p.fft_grid[0], th, sm, s>>>(g, p.fxr, twx, grid, p.zrange);
    else if (c2r_pair_ok(p.fxr))
      row_c2r_reg_kernel<T, true><<<p.fft_grid[1], th, sm, s>>>(g, p.fxr, twx, grid, p.zrange);
    else
      row_c2r_reg_kernel<T, false><<<p.fft_grid[1], th, sm, s>>>(g, p.fxr, twx, grid, p.zrange);
    return;
  }
  const int lb = p.row_lb, th = fft_threads(g.nx << lb);
  T* grid = reinterpret_cast<T*>(p.grid);
  if (dir < 0) {
    const auto kernel = lb ? row_r2c_kernel<T, true> : row_r2c_kernel<T, false>;
    kernel<<<p.fft_grid[0], th, row_r2c_smem<T>(g, lb), s>>>(g, p.fx, twx, grid, p.zrange, lb);
  } else {
    const auto kernel = lb ? row_c2r_kernel<T, true> : row_c2r_kernel<T, false>;
    kernel<<<p.fft_grid[1], th, row_c2r_smem<T>(g, lb), s>>>(g, p.fx, twx, grid, p.zrange, lb);
  }
}

}  // namespace dps
