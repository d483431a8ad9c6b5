// Row passes: variant selection and launches (instantiated per precision by fft_rows_*.cu).
#pragma once

#include "fft_kernels.cuh"

namespace dps {

template <typename T>
bool fft_rows_allow() {
  return allow_smem(row_r2c_kernel<T>) && allow_smem(row_c2r_kernel<T>) && allow_smem(row_r2c_reg_kernel<T, false>) &&
         allow_smem(row_r2c_reg_kernel<T, true>) && allow_smem(row_c2r_reg_kernel<T, false>) &&
         allow_smem(row_c2r_reg_kernel<T, true>);
}

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
  const size_t r2c = row_r2c_smem<T>(p.g), c2r = row_c2r_smem<T>(p.g);
  const int trow = fft_threads(p.g.nx);
  if (trow > kFftMaxThreads || r2c > 220 * 1024 || c2r > 220 * 1024) return 0;
  p.fft_reg[0] = 0;
  p.fft_grid[0] = resident_grid(row_r2c_kernel<T>, trow, r2c, p.device);
  p.fft_grid[1] = resident_grid(row_c2r_kernel<T>, trow, c2r, p.device);
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
  const int th = fft_threads(g.nx);
  if (dir < 0)
    row_r2c_kernel<T><<<p.fft_grid[0], th, row_r2c_smem<T>(g), s>>>(g, p.fx, twx, reinterpret_cast<T*>(p.grid),
                                                                      p.zrange);
  else
    row_c2r_kernel<T><<<p.fft_grid[1], th, row_c2r_smem<T>(g), s>>>(g, p.fx, twx, reinterpret_cast<T*>(p.grid),
                                                                      p.zrange);
}

}  // namespace dps
