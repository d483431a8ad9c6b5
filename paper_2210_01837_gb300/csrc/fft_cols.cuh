// Column passes: variant selection and launches (instantiated per precision by fft_cols_*.cu).
#pragma once

#include <type_traits>

#include "fft_kernels.cuh"

namespace dps {

namespace {

// the column kernels' ODD instantiation for this factorisation (always, in double: compiled for 128
// registers a thread, they have room)
template <typename T>
bool odd_columns(const FftPlan& fp) {
  if (sizeof(T) == 8) return true;
  for (int s = 0; s < fp.nstages; ++s) {
    const int r = fp.radix[s];
    if (r % 5 == 0 || r % 7 == 0 || r == 9) return true;
  }
  return false;
}

// f(std::integral_constant<bool, ODD>) for it
template <typename T, typename F>
auto with_odd(const Plan& p, F&& f) {
  if constexpr (sizeof(T) == 8) return f(std::true_type());
  else return odd_columns<T>(p.fyr) ? f(std::true_type()) : f(std::false_type());
}

}  // namespace

template <typename T, bool ODD>
bool fft_cols_allow_odd() {
  return allow_smem(col_reg_kernel<T, -1, ODD>) && allow_smem(col_reg_kernel<T, +1, ODD>) &&
         allow_smem(col_pipe_kernel<T, -1, ODD>) && allow_smem(col_pipe_kernel<T, +1, ODD>) &&
         allow_smem(col_tma_kernel<T, -1, ODD>) && allow_smem(col_tma_kernel<T, +1, ODD>);
}
template <typename T>
bool fft_cols_allow() {
  if (!allow_smem(col_kernel<T, -1>) || !allow_smem(col_kernel<T, +1>)) return false;
  if constexpr (sizeof(T) == 4) {
    if (!fft_cols_allow_odd<T, false>()) return false;
  }
  return fft_cols_allow_odd<T, true>();
}

template <typename T>
int fft_set_col_width(Plan& p, int lcw, int reg) {
  if (lcw < 0 || lcw > 3 || reg < 0 || reg > 3) return 0;
  if (reg == 3) {
    const int maxth = sizeof(T) == 4 ? kPipeMaxThreadsF : kPipeMaxThreadsD;
    const int th = reg_threads(p.fyr, lcw);
    const size_t sm = tma_smem<T>(p.g.ny << lcw);
    const int bh = tma_box_rows<T>(p.g.ny, lcw);
    // box rows of 16-byte multiples; a block never reads past the padded row (pitch is a multiple
    // of 32 columns and a block starts at a multiple of its width)
    if (th > maxth || sm > 224 * 1024 || bh == 0 || ((2u << lcw) * sizeof(T)) % 16 != 0) return 0;
    if (!encode_col_tmap<T>(p, lcw, bh)) return 0;
    p.col_lcw = lcw;
    p.fft_reg[1] = 3;
    p.col_tma_rows = bh;
    with_odd<T>(p, [&](auto o) {
      constexpr bool ODD = decltype(o)::value;
      p.fft_grid[2] = resident_grid(col_tma_kernel<T, -1, ODD>, th, sm, p.device);
      p.fft_grid[3] = resident_grid(col_tma_kernel<T, +1, ODD>, th, sm, p.device);
    });
    return 1;
  }
  if (reg == 2) {
    if (!pipe_fits<T>(p.fyr, lcw)) return 0;
    const int th = reg_threads(p.fyr, lcw);
    const size_t sm = pipe_smem<T>(p.g.ny << lcw);
    p.col_lcw = lcw;
    p.fft_reg[1] = 2;
    with_odd<T>(p, [&](auto o) {
      constexpr bool ODD = decltype(o)::value;
      p.fft_grid[2] = resident_grid(col_pipe_kernel<T, -1, ODD>, th, sm, p.device);
      p.fft_grid[3] = resident_grid(col_pipe_kernel<T, +1, ODD>, th, sm, p.device);
    });
    return 1;
  }
  if (reg) {
    if (!reg_fits<T>(p.fyr, lcw)) return 0;
    const int th = reg_threads(p.fyr, lcw);
    const size_t sm = reg_smem<T>(p.g.ny << lcw);
    p.col_lcw = lcw;
    p.fft_reg[1] = 1;
    with_odd<T>(p, [&](auto o) {
      constexpr bool ODD = decltype(o)::value;
      p.fft_grid[2] = resident_grid(col_reg_kernel<T, -1, ODD>, th, sm, p.device);
      p.fft_grid[3] = resident_grid(col_reg_kernel<T, +1, ODD>, th, sm, p.device);
    });
    return 1;
  }
  const size_t col = col_smem<T>(p.g, lcw);
  const int tcol = fft_threads(p.g.ny << lcw);
  if (tcol > kFftMaxThreads || col > 220 * 1024) return 0;
  p.col_lcw = lcw;
  p.fft_reg[1] = 0;
  p.fft_grid[2] = resident_grid(col_kernel<T, -1>, tcol, col, p.device);
  p.fft_grid[3] = resident_grid(col_kernel<T, +1>, tcol, col, p.device);
  return 1;
}

template <typename T>
bool fft_cols_default(Plan& p) {
  // columns: the prefetched register-staged pass when it fits a wider block than the staged one,
  // prefetched by TMA where a box shape fits (3072^2: 12.2 -> 10.7 ms per pass pair), else cp.async
  const int ls = col_lwidth<T>(p);
  for (int l = sizeof(T) == 4 ? 3 : 2; l > ls; --l)
    if (fft_set_col_width<T>(p, l, 3) || fft_set_col_width<T>(p, l, 2)) return true;
  // at the staged pass's width, TMA from 320 rows on in float (8 columns, us per pass, staged / TMA: 216 rows
  // 58 / 60, 384 rows 235 / 219, 630 rows 475 / 478, 768 rows 578 / 538 at 65 nodes) and from 512 in double
  if (p.g.ny >= (sizeof(T) == 4 ? 320 : 512) && fft_set_col_width<T>(p, ls, 3)) return true;
  if (fft_set_col_width<T>(p, ls, 0)) return true;
  for (int l = 3; l >= 0; --l)
    if (fft_set_col_width<T>(p, l, 1)) return true;
  return false;
}

template <typename T>
void launch_fft_cols(const Plan& p, int dir, int kxs, int kxe, cudaStream_t s) {
  const Geometry& g = p.g;
  const cplx<T>* twy = reinterpret_cast<const cplx<T>*>(p.tab.twy);
  const int lcw = p.col_lcw;
  cplx<T>* grid = reinterpret_cast<cplx<T>*>(p.grid);
  const cplx<T>* tsy = reinterpret_cast<const cplx<T>*>(p.tab.tsy);
  if (p.fft_reg[1] == 3) {
    const int th = reg_threads(p.fyr, lcw);
    const size_t sm = tma_smem<T>(g.ny << lcw);
    const CUtensorMap& map = *reinterpret_cast<const CUtensorMap*>(p.col_tmap);
    with_odd<T>(p, [&](auto o) {
      constexpr bool ODD = decltype(o)::value;
      if (dir < 0)
        col_tma_kernel<T, -1, ODD><<<p.fft_grid[2], th, sm, s>>>(map, g, p.fyr, tsy, grid, p.zrange, p.status, lcw, kxs,
                                                                 kxe, p.col_tma_rows, p.inject == 3 ? 1 : 0);
      else
        col_tma_kernel<T, +1, ODD><<<p.fft_grid[3], th, sm, s>>>(map, g, p.fyr, tsy, grid, p.zrange, p.status, lcw, kxs,
                                                                 kxe, p.col_tma_rows, 0);
    });
    return;
  }
  if (p.fft_reg[1] == 2) {
    const int th = reg_threads(p.fyr, lcw);
    const size_t sm = pipe_smem<T>(g.ny << lcw);
    with_odd<T>(p, [&](auto o) {
      constexpr bool ODD = decltype(o)::value;
      if (dir < 0)
        col_pipe_kernel<T, -1, ODD><<<p.fft_grid[2], th, sm, s>>>(g, p.fyr, tsy, grid, p.zrange, lcw, kxs, kxe);
      else
        col_pipe_kernel<T, +1, ODD><<<p.fft_grid[3], th, sm, s>>>(g, p.fyr, tsy, grid, p.zrange, lcw, kxs, kxe);
    });
    return;
  }
  if (p.fft_reg[1]) {
    const int th = reg_threads(p.fyr, lcw);
    const size_t sm = reg_smem<T>(g.ny << lcw);
    with_odd<T>(p, [&](auto o) {
      constexpr bool ODD = decltype(o)::value;
      if (dir < 0)
        col_reg_kernel<T, -1, ODD><<<p.fft_grid[2], th, sm, s>>>(g, p.fyr, tsy, grid, p.zrange, lcw, kxs, kxe);
      else
        col_reg_kernel<T, +1, ODD><<<p.fft_grid[3], th, sm, s>>>(g, p.fyr, tsy, grid, p.zrange, lcw, kxs, kxe);
    });
    return;
  }
  const size_t sm = col_smem<T>(g, lcw);
  const int th = fft_threads(g.ny << lcw);
  if (dir < 0)
    col_kernel<T, -1><<<p.fft_grid[2], th, sm, s>>>(g, p.fy, twy, reinterpret_cast<cplx<T>*>(p.grid), p.zrange, lcw,
                                                    kxs, kxe);
  else
    col_kernel<T, +1><<<p.fft_grid[3], th, sm, s>>>(g, p.fy, twy, reinterpret_cast<cplx<T>*>(p.grid), p.zrange, lcw,
                                                    kxs, kxe);
}

}  // namespace dps
