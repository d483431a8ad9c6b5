// Chebyshev transforms of three fields in single precision (steps 2 and 6-7 of Sec. III.D, z part, for the routes
// without a spectral curl): forward DCT-I of the force density; backward, inverse DCT-I of the DP velocity plus
// the wall correction at the nodes, times 1/(Nx Ny).
//
// A thread owns one wavenumber of one field.  It loads the whole column to registers (a warp's row is 256
// contiguous bytes, nz rows of every thread in flight), so the memory stays busy without staging, barriers or a
// second copy.  By cos(pi n (n1 - c)/n1) = (-1)^n cos(pi n c/n1), n1 = nz - 1, the sums and differences of
// mirrored nodes give the even and the odd coefficients, and the sums over even and odd coefficients give two
// mirrored nodes: half of the dense product's FMAs.  The table is in shared memory, one broadcast 16-byte read
// per 8 FMAs.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "bvp_device.cuh"
#include "dps_internal.cuh"

namespace dps {
namespace {

constexpr int kColThreads = 128;
// blocks per SM to which a bucket's registers are limited: the column is 4 HP of them, and the compiler would
// keep the addresses of all rows besides
__host__ __device__ constexpr int col_blocks(int hp) { return hp <= 10 ? 6 : hp <= 18 ? 4 : hp <= 26 ? 3 : 2; }

// wavenumber of this lane: column in a plane of the grid (-1 beyond the end), index, components
struct ColLane {
  int64_t col, kid;
  int kxi, nyv;
  bool nyq;
};
__device__ __forceinline__ ColLane col_lane(const Geometry& g, unsigned it, unsigned total, int kx0, int w) {
  ColLane r{-1, 0, 0, 0, false};
  if (it < total) {
    const int kyi = (int)(it / (unsigned)w);
    r.kxi = kx0 + (int)(it - (unsigned)kyi * (unsigned)w);
    r.nyv = (kyi < (g.ny + 1) / 2) ? kyi : kyi - g.ny;
    r.col = (int64_t)kyi * g.pitch + r.kxi;
    r.kid = (int64_t)kyi * g.nkx + r.kxi;
    r.nyq = ((g.nx % 2 == 0) && r.kxi == g.nx / 2) || ((g.ny % 2 == 0) && kyi == g.ny / 2);
  }
  return r;
}

// HP: half of the column, (nz + 1) / 2, rounded up to a bucket.  Table: [(nz + 1) / 2][2 HP], zero past the
// column.
template <int HP>
__global__ void __launch_bounds__(kColThreads, col_blocks(HP)) cols_fwd_kernel(const __grid_constant__ Geometry g,
                                                              const float* __restrict__ ct, int npad,
                                                              const cplx<float>* __restrict__ grid,
                                                              cplx<float>* __restrict__ kbuf,
                                                              const int* __restrict__ zrange, int kx0, int w) {
  extern __shared__ __align__(16) unsigned char smraw[];
  float* tab = reinterpret_cast<float*>(smraw);  // row r: C[2r][c], C[2r + 1][c], c = 0 ..
  const int N = g.nz, n1 = N - 1, np = (N + 1) / 2;
  for (int i = threadIdx.x; i < np * 2 * HP; i += kColThreads) {
    const int r = i / (2 * HP), q = i - r * 2 * HP, n = 2 * r + (q & 1), c = q >> 1;
    tab[i] = n < N && c < np ? ct[(size_t)c * npad + n] : 0.f;
  }
  __syncthreads();
  const int clo = zrange[0], chi = zrange[1];
  const int64_t K = (int64_t)g.nkx * g.ny;
  const unsigned total = (unsigned)w * (unsigned)g.ny, per_field = (total + kColThreads - 1) / kColThreads;
  const size_t plane = (size_t)g.ny * g.pitch, fs = (size_t)N * plane;
  for (unsigned b = blockIdx.x; b < 3 * per_field; b += gridDim.x) {
    const int f = (int)(b / per_field);
    const ColLane L = col_lane(g, (b - (unsigned)f * per_field) * kColThreads + threadIdx.x, total, kx0, w);
    if (L.col < 0) continue;
    const cplx<float>* in = grid + f * fs + L.col;
    cplx<float> xe[HP], xo[HP];
#pragma unroll
    for (int c = 0; c < HP; ++c) {
      const int m = n1 - c;
      const cplx<float> lo = c <= m && c >= clo && c <= chi ? in[c * plane] : mk<float>(0.f, 0.f);
      const cplx<float> hi = c < m && m >= clo && m <= chi ? in[m * plane] : mk<float>(0.f, 0.f);
      xe[c] = lo + hi;
      xo[c] = c < m ? lo - hi : mk<float>(0.f, 0.f);
    }
    cplx<float>* out = kbuf + (size_t)f * N * K + L.kid;
    for (int r = 0; r < np; ++r) {
      const float4* t4 = reinterpret_cast<const float4*>(tab + r * 2 * HP);
      cplx<float> e = mk<float>(0.f, 0.f), o = e;
#pragma unroll
      for (int c = 0; c < HP; c += 2) {
        const float4 t = t4[c / 2];
        e.x = fmaf(t.x, xe[c].x, e.x);
        e.y = fmaf(t.x, xe[c].y, e.y);
        o.x = fmaf(t.y, xo[c].x, o.x);
        o.y = fmaf(t.y, xo[c].y, o.y);
        e.x = fmaf(t.z, xe[c + 1].x, e.x);
        e.y = fmaf(t.z, xe[c + 1].y, e.y);
        o.x = fmaf(t.w, xo[c + 1].x, o.x);
        o.y = fmaf(t.w, xo[c + 1].y, o.y);
      }
      out[(size_t)(2 * r) * K] = e;
      if (2 * r + 1 < N) out[(size_t)(2 * r + 1) * K] = o;
    }
  }
}

template <int HP, int CORR>  // CORR: 0 no wall, 1 bottom wall, 2 both walls
__global__ void __launch_bounds__(kColThreads, col_blocks(HP)) cols_bwd_kernel(const __grid_constant__ Geometry g,
                                                              const float* __restrict__ ict, int cpad,
                                                              const float* __restrict__ zeta,
                                                              const cplx<float>* __restrict__ kbuf,
                                                              const cplx<float>* __restrict__ kaux,
                                                              cplx<float>* __restrict__ grid,
                                                              const int* __restrict__ zrange, int kx0, int w, double hpx,
                                                              double hpy, float inv_nxny) {
  extern __shared__ __align__(16) unsigned char smraw[];
  float* tab = reinterpret_cast<float*>(smraw);  // row c: IC[c][n], n = 0 ..
  const int N = g.nz, n1 = N - 1, np = (N + 1) / 2;
  float* sz = tab + np * 2 * HP;  // [N] zeta
  for (int i = threadIdx.x; i < np * 2 * HP; i += kColThreads) {
    const int c = i / (2 * HP), n = i - c * 2 * HP;
    tab[i] = n < N ? ict[(size_t)n * cpad + c] : 0.f;
  }
  for (int i = threadIdx.x; i < N; i += kColThreads) sz[i] = zeta[i];
  __syncthreads();
  const int clo = zrange[0], chi = zrange[1];
  const int64_t K = (int64_t)g.nkx * g.ny;
  const unsigned total = (unsigned)w * (unsigned)g.ny, per_field = (total + kColThreads - 1) / kColThreads;
  const size_t plane = (size_t)g.ny * g.pitch, fs = (size_t)N * plane;
  for (unsigned b = blockIdx.x; b < 3 * per_field; b += gridDim.x) {
    const int f = (int)(b / per_field);
    const ColLane L = col_lane(g, (b - (unsigned)f * per_field) * kColThreads + threadIdx.x, total, kx0, w);
    if (L.col < 0) continue;
    cplx<float>* out = grid + f * fs + L.col;
    if (L.nyq) {
      for (int c = clo; c <= chi; ++c) out[c * plane] = mk<float>(0.f, 0.f);
      continue;
    }
    const cplx<float>* in = kbuf + (size_t)f * N * K + L.kid;
    cplx<float> y[2 * HP];
#pragma unroll
    for (int n = 0; n < 2 * HP; ++n) y[n] = n < N ? in[(size_t)n * K] : mk<float>(0.f, 0.f);
    cplx<float> cE = mk<float>(0.f, 0.f), cG = cE, tE = cE, tG = cE;
    float kk = 0.f;
    if (CORR) {
      if (L.kid > 0) {
        const cplx<float>* am = kaux + (size_t)4 * f * K + L.kid;
        cE = am[0];
        cG = am[K];
        if (CORR == 2) {
          tE = am[2 * K];
          tG = am[3 * K];
        }
      }
      const double hx = hpx * (double)L.kxi, hy = hpy * (double)L.nyv;
      // |k| = 2 sqrt(s) as a square root in double, rounded to float, gives it, without holding up the FP64
      // pipe: a float root and one Newton step with the residual formed in double
      const double s = hx * hx + hy * hy;
      const float r = sqrtf(d2f(s));
      if (r > 0.f) kk = fmaf(2.0f, r, __fdividef(d2f(fma(-f2d(r), f2d(r), s)), r));
    }
    for (int c = 0; c < np; ++c) {
      const int m = n1 - c;
      const bool low = c >= clo && c <= chi, high = m != c && m >= clo && m <= chi;
      if (!low && !high) continue;
      const float4* t4 = reinterpret_cast<const float4*>(tab + c * 2 * HP);
      cplx<float> e = mk<float>(0.f, 0.f), o = e;
#pragma unroll
      for (int n = 0; n < 2 * HP; n += 4) {
        const float4 t = t4[n / 4];
        e.x = fmaf(t.x, y[n].x, e.x);
        e.y = fmaf(t.x, y[n].y, e.y);
        o.x = fmaf(t.y, y[n + 1].x, o.x);
        o.y = fmaf(t.y, y[n + 1].y, o.y);
        e.x = fmaf(t.z, y[n + 2].x, e.x);
        e.y = fmaf(t.z, y[n + 2].y, e.y);
        o.x = fmaf(t.w, y[n + 3].x, o.x);
        o.y = fmaf(t.w, y[n + 3].y, o.y);
      }
      cplx<float> vl = e + o, vh = e - o;
      if (CORR) {
        const float zl = sz[c], zh = sz[m];
        const float el = expf(-kk * zl), eh = expf(-kk * zh);
        vl.x = fmaf(fmaf(cG.x, zl, cE.x), el, vl.x);
        vl.y = fmaf(fmaf(cG.y, zl, cE.y), el, vl.y);
        vh.x = fmaf(fmaf(cG.x, zh, cE.x), eh, vh.x);
        vh.y = fmaf(fmaf(cG.y, zh, cE.y), eh, vh.y);
        if (CORR == 2) {  // the top family's xi is the mirrored node's zeta
          vl.x = fmaf(fmaf(tG.x, zh, tE.x), eh, vl.x);
          vl.y = fmaf(fmaf(tG.y, zh, tE.y), eh, vl.y);
          vh.x = fmaf(fmaf(tG.x, zl, tE.x), el, vh.x);
          vh.y = fmaf(fmaf(tG.y, zl, tE.y), el, vh.y);
        }
      }
      if (low) out[c * plane] = mk<float>(vl.x * inv_nxny, vl.y * inv_nxny);
      if (high) out[m * plane] = mk<float>(vh.x * inv_nxny, vh.y * inv_nxny);
    }
  }
}

// blocks of a launch: of the chunk's columns, no more than the GPU holds at once
unsigned cols_blocks(const Plan& p, bool backward, int w) {
  const int64_t blocks = 3 * (((int64_t)w * p.g.ny + kColThreads - 1) / kColThreads);
  return (unsigned)std::min<int64_t>(blocks, p.cols_grid[backward]);
}
template <int HP>
size_t cols_smem(const Geometry& g, bool backward) {
  return ((size_t)(g.nz + 1) / 2 * 2 * HP + (backward ? g.nz : 0)) * sizeof(float);
}

template <int HP, int CORR>
void launch_bwd(const Plan& p, int kx0, int w, cudaStream_t s) {
  const Geometry& g = p.g;
  cols_bwd_kernel<HP, CORR><<<cols_blocks(p, true, w), kColThreads, cols_smem<HP>(g, true), s>>>(
      g, reinterpret_cast<const float*>(p.kt.ict), p.kt.cpad, reinterpret_cast<const float*>(p.tab.zeta),
      reinterpret_cast<const cplx<float>*>(p.kt.kbuf), reinterpret_cast<const cplx<float>*>(p.kt.kaux),
      reinterpret_cast<cplx<float>*>(p.grid), p.zrange, kx0, w, M_PI / g.Lx, M_PI / g.Ly,
      (float)(1.0 / ((double)g.nx * (double)g.ny)));
}

// f(std::integral_constant<int, HP>) for the column's bucket
template <typename F>
auto with_bucket(const Geometry& g, F&& f) {
  const int half = (g.nz + 1) / 2;
  if (half <= 10) return f(std::integral_constant<int, 10>());
  if (half <= 18) return f(std::integral_constant<int, 18>());
  if (half <= 26) return f(std::integral_constant<int, 26>());
  return f(std::integral_constant<int, 34>());  // (backward only)
}

template <int HP>
void launch_dir(const Plan& p, bool backward, int kx0, int w, cudaStream_t s) {
  const Geometry& g = p.g;
  if constexpr (HP <= 26) {
    if (!backward) {
      cols_fwd_kernel<HP><<<cols_blocks(p, false, w), kColThreads, cols_smem<HP>(g, false), s>>>(
          g, reinterpret_cast<const float*>(p.kt.ct), p.kt.npad, reinterpret_cast<const cplx<float>*>(p.grid),
          reinterpret_cast<cplx<float>*>(p.kt.kbuf), p.zrange, kx0, w);
      return;
    }
  }
  if (g.mode == DPS_FREE) {
    launch_bwd<HP, 0>(p, kx0, w, s);
  } else if (g.mode == DPS_SLIT) {
    launch_bwd<HP, 2>(p, kx0, w, s);
  } else {
    launch_bwd<HP, 1>(p, kx0, w, s);
  }
}

}  // namespace

// The forward transform up to 52 nodes, the backward one up to 68, the columns that leave two blocks an SM.  us
// against what ran before (forward on the tensor cores or, in brackets, by lane groups with staged planes;
// backward by lane groups), bottom wall:
//   1536 x 1536 x 9: forward 228 (131) -> 117, backward 421 -> 111    x 19: 404 (276) -> 203, 616 -> 184
//   x 33: 623 (668) -> 508, 874 -> 387    1024 x 1024 x 49: 410 (543) -> 289, 846 -> 328
//   1024 x 1024 x 65: 494 (846) against 569: tensor cores stay; 1188 -> 534
// (19 nodes: both ways at the rate of a copy.)  The kernel-derivative torque route keeps the tensor cores forward:
// its angular velocities came out 9 % further from double (33 nodes: 4.9e-7 against 5.4e-7; linear velocities
// 4.5e-7 against 3.8e-7).  Without torques both directions together are closer (19 nodes 3.7e-7 -> 3.5e-7, 49
// nodes 5.4e-7 -> 4.6e-7).
int cheb_columns_prepare(Plan& p) {
  const Geometry& g = p.g;
  p.cheb_columns = 0;
  if (p.precision != DPS_MIXED || g.spectral_curl) return 1;
  p.cheb_columns = (g.nz <= 52 && !g.with_torque ? 1 : 0) | (g.nz <= 68 ? 2 : 0);
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p.device) != cudaSuccess) return 0;
  return with_bucket(g, [&](auto hp) {
    constexpr int HP = decltype(hp)::value;
    const void* kernel[2] = {nullptr, g.mode == DPS_FREE   ? (const void*)cols_bwd_kernel<HP, 0>
                                      : g.mode == DPS_SLIT ? (const void*)cols_bwd_kernel<HP, 2>
                                                           : (const void*)cols_bwd_kernel<HP, 1>};
    if constexpr (HP <= 26) kernel[0] = (const void*)cols_fwd_kernel<HP>;
    for (int d = 0; d < 2; ++d) {
      int per_sm = 0;
      if (!(p.cheb_columns >> d & 1)) continue;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel[d], kColThreads, cols_smem<HP>(g, d == 1)) !=
              cudaSuccess || per_sm < 1)
        return 0;
      p.cols_grid[d] = per_sm * sms;
    }
    return 1;
  });
}

void launch_cheb_columns(const Plan& p, bool backward, int kx0, int w, cudaStream_t s) {
  with_bucket(p.g, [&](auto hp) { launch_dir<decltype(hp)::value>(p, backward, kx0, w, s); });
}

}  // namespace dps
