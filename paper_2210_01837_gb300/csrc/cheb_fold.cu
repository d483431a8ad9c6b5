// Chebyshev transforms by folding (steps 2 and 6-7 of Sec. III.D), for node counts with nz - 1 a multiple
// of 8: the double-precision plans' transforms, which as dense contractions were bound by the FP64 pipe.
//
// Both directions are a product with the matrix cos(pi n c / n1), n1 = nz - 1 = 2 M = 4 h.  Its symmetries
// split it, without any division or growth, into small dense parts, 0.15 of the work:
//   e_c = x_c + x_{n1-c}, o_c = x_c - x_{n1-c};  p_c = e_c + e_{M-c}, q_c = e_c - e_{M-c};
//   s_c = p_c + p_{h-c}, d_c = p_c - p_{h-c}
//   X_{8j}   from s (h/2 + 1 inputs and outputs), X_{8j+4} from d (h/2)
//   X_{4m+2} = G_m + H_m, X_{n1-(4m+2)} = G_m - H_m, m < h/2, from q at even and odd c (h/2 each)
//   X_{2m+1} = E_m + O_m, X_{n1-(2m+1)} = E_m - O_m, m < h, from o at even and odd c; E splits once more
//   by even and odd c/2 as X_{4m+2} does, O (odd c) is a dense h x h part.
// Derivatives are the recurrence on coefficients (O(n)) instead of dense matrices, and the wall correction
// enters as coefficients too: those of e^{-k zeta} and zeta e^{-k zeta}, a plan-time table per |k| (its mirror
// image at the other wall has them with alternating signs), so that no exponential is left.
//
// A block takes 16 wavenumbers, lanes 0-15 their real and 16-31 their imaginary parts (a 256-byte row of
// the spectra), all fields in shared memory, four warps per field: five fields make 20 warps, five on each
// sub-partition, the parts dealt so that their loads differ by a few per cent.  A part's outputs stay in
// registers until all inputs are read.  The table values are broadcast reads, each feeding one FMA: 64
// clocks of FP64 pipe, so the pipe is the bound.
//
// Measured (384 x 384 x 97, slit, torques, double; two levels of folding: 4.29 and 4.10): forward 15.5 -> 3.23
// ms, backward 19.6 -> 2.97 ms.
#include <math.h>

#include <type_traits>
#include <vector>

#include "bvp_device.cuh"
#include "dps_internal.cuh"

namespace dps {
namespace {

using T = double;           // the plans that fold
constexpr int kFoldK = 16;  // wavenumbers per block

__host__ __device__ constexpr int fold_pad(int hp) { return (hp + 1) / 2 * 2; }  // table row: whole 16-byte loads
// outputs of a part kept in registers: h/2 + 1, by buckets
__host__ __device__ inline int fold_bucket(int N) { return N <= 33 ? 5 : (N <= 65 ? 9 : (N <= 97 ? 13 : 17)); }

// A part: cnt inputs at slots x0 + i dx, outs outputs, table rows from `row`.  A warp's role r has two:
//   0: O_m, m < h/2, and X_{8j}      1: O_m, m >= h/2, and X_{8j+4}
//   2: G, H                          3: the halves of E
struct FoldPart {
  int x0, dx, cnt, outs, row;
};
__host__ __device__ inline FoldPart fold_part_of(int r, int q, int h) {
  const int n1 = 4 * h, M = 2 * h, k = h / 2;
  switch (2 * r + q) {
    case 0: return {n1 - 1, -2, h, k, 0};
    case 1: return {0, 1, k + 1, k + 1, h};
    case 2: return {n1 - 1, -2, h, k, h + k + 1};
    case 3: return {h, -1, k, k, 2 * h + k + 1};
    case 4: return {M, -2, k, k, 2 * h + 2 * k + 1};
    case 5: return {M - 1, -2, k, k, 2 * h + 3 * k + 1};
    case 6: return {n1, -4, k, k, 2 * h + 4 * k + 1};
    default: return {n1 - 2, -4, k, k, 2 * h + 5 * k + 1};
  }
}
__host__ __device__ inline int fold_rows(int h) { return 2 * h + 6 * (h / 2) + 1; }
__host__ __device__ inline size_t fold_table_values(int N) {
  return (size_t)fold_rows((N - 1) / 4) * fold_pad(fold_bucket(N));
}
// shared memory: fields, part tables, derivative factors
__host__ __device__ inline size_t fold_smem(int N, int nf) {
  return ((size_t)nf * N * 32 + fold_table_values(N) + N) * sizeof(T);
}

// x_c -> p_c, q_c, o_c, o_{M-c} of one column in place, c = 0 .. h: slots c, M - c, n1 - c, M + c; returns p_c
__device__ __forceinline__ T fold_quad(T* x, int c, int h) {
  const int M = 2 * h, n1 = 4 * h;
  const T a = x[c * 32], b = x[(n1 - c) * 32];
  const T e = a + b;
  x[(n1 - c) * 32] = a - b;
  if (c == h) return e;
  T f = x[(M - c) * 32];
  if (c) {
    const T u = x[(M + c) * 32];
    x[(M + c) * 32] = f - u;
    f = f + u;
  }
  x[(M - c) * 32] = e - f;
  return e + f;
}
// work item c = 0 .. h/2: the quadruples of c and h - c, then s_c in slot c and d_c in slot h - c
__device__ __forceinline__ void fold_in(T* x, int c, int h) {
  const T a = fold_quad(x, c, h);
  if (2 * c == h) {
    x[c * 32] = a;
  } else {
    const T b = fold_quad(x, h - c, h);
    x[c * 32] = a + b;
    x[(h - c) * 32] = a - b;
  }
}

// X_n from the parts' outputs: X_{4j} in slot j, X_{4j+2} in slot M - j, E_m in slot n1 - 2m, O_m below it
__device__ __forceinline__ T fold_out(const T* x, int n, int M) {
  if (!(n & 1)) return x[((n & 2) ? M - (n >> 2) : n >> 2) * 32];
  const bool up = n < M;
  const int m = up ? n >> 1 : (2 * M - n) >> 1;
  const T e = x[(2 * M - 2 * m) * 32], o = x[(2 * M - 2 * m - 1) * 32];
  return up ? e + o : e - o;
}

template <int HP>
__device__ __forceinline__ void fold_dot(const T* x, const T* __restrict__ tab, const FoldPart& p, T (&acc)[HP]) {
  constexpr int PAD = fold_pad(HP);
#pragma unroll
  for (int j = 0; j < HP; ++j) acc[j] = (T)0;
  const T* xi = x + p.x0 * 32;
  const T* row = tab + (size_t)p.row * PAD;
  const int step = p.dx * 32;
  for (int c = 0; c < p.cnt; ++c) {
    const T v = *xi;
    xi += step;
#pragma unroll
    for (int j = 0; j < PAD; j += 2) {
      const double2 t = *reinterpret_cast<const double2*>(row + j);
      acc[j] = fma(t.x, v, acc[j]);
      if (j + 1 < HP) acc[j + 1] = fma(t.y, v, acc[j + 1]);
    }
    row += PAD;
  }
}

// Folds the columns of all fields and applies their parts, in place; by the whole block, between barriers.
template <int HP>
__device__ __forceinline__ void fold_apply(T* sx, const T* tab, int N) {
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, f = wi >> 2, h = (N - 1) / 4, k = h / 2, M = 2 * h;
  const int r = (wi + f) & 3;  // a field's roles on all sub-partitions, a role of the fields too
  T* x = sx + (size_t)f * N * 32 + lane;
  for (int c = wi & 3; c <= k; c += 4) fold_in(x, c, h);
  __syncthreads();
  T a[HP], b[HP];
  fold_dot<HP>(x, tab, fold_part_of(r, 0, h), a);
  fold_dot<HP>(x, tab, fold_part_of(r, 1, h), b);
  __syncthreads();  // inputs read
#pragma unroll
  for (int j = 0; j < HP; ++j) {
    if (r < 2) {
      if (j < k) x[(4 * h - 2 * (j + r * k) - 1) * 32] = a[j];
      if (j < k + 1 - r) x[(2 * j + r) * 32] = b[j];
    } else if (j < k) {
      const T u = a[j] + b[j], v = a[j] - b[j];
      if (r == 2) {
        x[(M - j) * 32] = u;
        x[(M - (h - 1 - j)) * 32] = v;
      } else {
        x[(4 * h - 2 * j) * 32] = u;
        x[(4 * h - 2 * (h - 1 - j)) * 32] = v;
      }
    }
  }
  __syncthreads();
}

struct FoldLane {
  int64_t col;   // spectrum column in a plane (complex), -1 beyond the end
  int kid, kp;
  bool nyq;
  double hkx, hky;
};

// hx, hy: pi / Lx, pi / Ly (formed on the host: a division would take the FP64 pipe)
__device__ __forceinline__ FoldLane fold_lane(const Geometry& g, int64_t it, int kx0, int w, double hx, double hy) {
  FoldLane r;
  r.col = -1;
  r.kid = r.kp = 0;
  r.nyq = false;
  r.hkx = r.hky = 0.0;
  if (it < (int64_t)w * g.ny) {
    const int64_t kidx = chunk_kidx(g, it, kx0, w);
    const int kyi = (int)((unsigned)kidx / (unsigned)g.nkx), kxi = (int)((unsigned)kidx - (unsigned)kyi * (unsigned)g.nkx);
    r.nyq = ((g.nx % 2 == 0) && kxi == g.nx / 2) || ((g.ny % 2 == 0) && kyi == g.ny / 2);
    const int nyv = (kyi < (g.ny + 1) / 2) ? kyi : kyi - g.ny;
    r.col = (int64_t)kyi * g.pitch + kxi;
    r.kid = (int)kidx;
    r.kp = ((2 * kyi <= g.ny) ? kyi : g.ny - kyi) * g.nkx + kxi;
    r.hkx = hx * (double)kxi;
    r.hky = hy * (double)nyv;
  }
  return r;
}

// forward: kbuf[o][n][k] = (C a_o + D C b_o)[n] with a_o = f_o + (1/2)(i k x tau)_o, b_x = -tau_y / 2,
// b_y = tau_x / 2 (TQ; else a_o = f_o alone)
template <bool TQ, int HP>
__global__ void __launch_bounds__((TQ ? 20 : 12) * 32) fold_fwd_kernel(const __grid_constant__ Geometry g,
                                                                      const T* __restrict__ tab_g,
                                                                      const cplx<T>* __restrict__ grid,
                                                                      cplx<T>* __restrict__ kbuf,
                                                                      const int* __restrict__ zrange, int kx0, int w,
                                                                      double hx, double hy, int thin) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if (thin > 0 && zrange[1] - zrange[0] < thin) return;  // the dense transform's turn
  constexpr int NF = TQ ? 5 : 3, NW = 4 * NF;
  const int N = g.nz, M = (N - 1) / 2;
  T* sx = reinterpret_cast<T*>(smraw);  // [NF][N][32]
  T* tab = sx + (size_t)NF * N * 32;
  T* dn = tab + fold_table_values(N);  // [N] 2 (n + 1) d/dz s, times the half of the curl forward
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, part = lane >> 4, kc = lane & 15;
  const int nt = (int)fold_table_values(N);
  for (int i = threadIdx.x; i < nt; i += NW * 32) tab[i] = tab_g[i];
  for (int i = threadIdx.x; i < N; i += NW * 32) dn[i] = (T)((i + 1 == N - 1 ? 0.25 : 0.5) * (2 * (i + 1)) * g.sH);
  const int64_t K = (int64_t)g.nkx * g.ny, total = (int64_t)w * g.ny;
  const size_t plane = (size_t)g.ny * g.pitch, fs = 2 * (size_t)g.nz * plane;  // reals of a field
  const int clo = zrange[0], chi = zrange[1];
  const T sg = part ? (T)1 : (T)-1;
  for (int64_t tile = blockIdx.x; tile * kFoldK < total; tile += gridDim.x) {
    const FoldLane L = fold_lane(g, tile * kFoldK + kc, kx0, w, hx, hy);
    const T hkx = sg * (T)L.hkx, hky = sg * (T)L.hky;
    const T* base = reinterpret_cast<const T*>(grid) + 2 * (L.col < 0 ? 0 : L.col) + part;
    __syncthreads();  // the last tile's outputs have been read (and, first, the table is in place)
#pragma unroll 3
    for (int c = wi; c < N; c += NW) {
      T a[6];
#pragma unroll
      for (int f = 0; f < (TQ ? 6 : 3); ++f)
        a[f] = (c >= clo && c <= chi) ? base[f * fs + 2 * c * plane] : (T)0;
      T* x = sx + c * 32 + lane;
      if constexpr (TQ) {
        const T tx = __shfl_xor_sync(0xffffffffu, a[3], 16), ty = __shfl_xor_sync(0xffffffffu, a[4], 16),
                tz = __shfl_xor_sync(0xffffffffu, a[5], 16);
        a[0] = a[0] + hky * tz;
        a[1] = a[1] - hkx * tz;
        a[2] = a[2] + (hkx * ty - hky * tx);
      }
      if (c == 0 || c == N - 1) {  // the end nodes' weight
#pragma unroll
        for (int f = 0; f < (TQ ? 6 : 3); ++f) a[f] = a[f] * (T)0.5;
      }
      x[0] = a[0];
      x[(size_t)N * 32] = a[1];
      x[(size_t)2 * N * 32] = a[2];
      if constexpr (TQ) {  // -b_x, b_y without their halves (in dn and the recurrence's sign)
        x[(size_t)3 * N * 32] = a[4];
        x[(size_t)4 * N * 32] = a[3];
      }
    }
    if ((tile + gridDim.x) * kFoldK < total) {  // the next tile's rows into L2 while the parts run
      const FoldLane P = fold_lane(g, (tile + gridDim.x) * kFoldK + kc, kx0, w, hx, hy);
      const cplx<T>* q = grid + (P.col < 0 ? 0 : P.col);
      for (int c = clo + wi; c <= chi; c += NW)
        if ((kc & 7) == 0)
          for (int f = part; f < (TQ ? 6 : 3); f += 2) prefetch_l2(q + ((size_t)f * g.nz + c) * plane);
    }
    __syncthreads();
    fold_apply<HP>(sx, tab, N);
    // outputs: with torques the first two components add the derivative recurrence over their b, a warp
    // per (component, parity); the others are spread over the remaining warps
    const bool keep = L.col >= 0 && !L.nyq;
    T* out = reinterpret_cast<T*>(kbuf + L.kid) + part;
    auto put = [&](int o, int n, T v) {
      if (n == 0 || n == N - 1) v = v * (T)0.5;
      if (keep) out[2 * ((size_t)o * N + n) * K] = v;
    };
    if (TQ && wi < 4) {
      const int o = wi >> 1;
      const T *xa = sx + (size_t)o * N * 32 + lane, *xb = sx + (size_t)(3 + o) * N * 32 + lane;
      T d = (T)0;
      for (int n = N - 1 - ((N - 1 - (wi & 1)) & 1); n >= 0; n -= 2) {
        if (n + 1 < N) {  // (dn holds the last coefficient's half)
          const T b = fold_out(xb, n + 1, M);
          d = fma(o ? b : -b, dn[n], d);
        }
        T v = fold_out(xa, n, M);
        if (n == 0 || n == N - 1) v = v * (T)0.5;
        v = v + (n == 0 ? d * (T)0.5 : d);
        if (keep) out[2 * ((size_t)o * N + n) * K] = v;
      }
    } else {
      const int w0 = TQ ? 4 : 0, o0 = TQ ? 2 : 0;
      for (int i = wi - w0; i < (3 - o0) * N; i += NW - w0) {
        const int o = o0 + i / N, n = i % N;
        put(o, n, fold_out(sx + (size_t)o * N * 32 + lane, n, M));
      }
    }
  }
}

// backward: node values on the occupied planes of the DP velocity plus the wall correction (coefficients
// ecf of e^{-k zeta} and zeta e^{-k zeta}) and, with CURL, the half-curl from the coefficients' derivatives;
// times 1/(Nx Ny)
template <bool CURL, int HP>
__global__ void __launch_bounds__((CURL ? 20 : 12) * 32) fold_bwd_kernel(const __grid_constant__ Geometry g,
                                                                        const T* __restrict__ tab_g,
                                                                        const double2* __restrict__ ecf, int64_t KP,
                                                                        const cplx<T>* __restrict__ kbuf,
                                                                        const cplx<T>* __restrict__ kaux,
                                                                        cplx<T>* __restrict__ grid,
                                                                        const int* __restrict__ zrange, int kx0, int w,
                                                                        double hx, double hy, int thin) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if (thin > 0 && zrange[1] - zrange[0] < thin) return;  // the dense transform's turn
  constexpr int NF = CURL ? 5 : 3, NW = 4 * NF;
  const int N = g.nz, M = (N - 1) / 2;
  T* sx = reinterpret_cast<T*>(smraw);  // [NF][N][32]
  T* tab = sx + (size_t)NF * N * 32;
  T* dn = tab + fold_table_values(N);  // [N] 2 (n + 1) d/dz s
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, part = lane >> 4, kc = lane & 15;
  const int nt = (int)fold_table_values(N);
  for (int i = threadIdx.x; i < nt; i += NW * 32) tab[i] = tab_g[i];
  for (int i = threadIdx.x; i < N; i += NW * 32) dn[i] = 2.0 * (i + 1) * g.sH;
  const int64_t K = (int64_t)g.nkx * g.ny, total = (int64_t)w * g.ny;
  const size_t plane = (size_t)g.ny * g.pitch, fs = 2 * (size_t)g.nz * plane;
  const int clo = zrange[0], chi = zrange[1];
  const T sg = part ? (T)1 : (T)-1;
  for (int64_t tile = blockIdx.x; tile * kFoldK < total; tile += gridDim.x) {
    const FoldLane L = fold_lane(g, tile * kFoldK + kc, kx0, w, hx, hy);
    const T hkx = sg * (T)L.hkx, hky = sg * (T)L.hky;
    const bool live = L.col >= 0 && !L.nyq;
    __syncthreads();  // the last tile's outputs have been read (and, first, the table is in place)
    {
      // coefficients: a warp takes the rows of one field
      const int f = wi % 3;
      const T* yb = reinterpret_cast<const T*>(kbuf + (size_t)f * N * K + L.kid) + part;
      // amplitudes by the parity of n: bottom +- top
      T ae = (T)0, ge = (T)0, ao = (T)0, go = (T)0;
      if (ecf != nullptr && live && L.kid > 0) {
        const T* am = reinterpret_cast<const T*>(kaux + (size_t)4 * f * K + L.kid) + part;
        const T cE = am[0], cG = am[2 * K], tE = am[4 * K], tG = am[6 * K];
        ae = cE + tE;
        ao = cE - tE;
        ge = cG + tG;
        go = cG - tG;
      }
      T* x = sx + (size_t)f * N * 32 + lane;
      if (wi < NW / 3 * 3)
#pragma unroll 3
        for (int n = wi / 3; n < N; n += NW / 3) {
          T v = live ? yb[2 * (size_t)n * K] : (T)0;
          if (ecf != nullptr) {
            const double2 e = ecf[(size_t)n * KP + L.kp];
            v = fma((n & 1) ? ao : ae, (T)e.x, v);
            v = fma((n & 1) ? go : ge, (T)e.y, v);
          }
          x[n * 32] = v;
        }
    }
    if ((tile + gridDim.x) * kFoldK < total) {  // the next tile's rows into L2 while the parts run
      const FoldLane P = fold_lane(g, (tile + gridDim.x) * kFoldK + kc, kx0, w, hx, hy);
      for (int n = wi; n < N; n += NW)
        if ((kc & 7) == 0) {
          if (part) prefetch_l2(kbuf + (size_t)n * K + P.kid);
          else prefetch_l2(kbuf + ((size_t)N + n) * K + P.kid);
          if (part) prefetch_l2(kbuf + ((size_t)2 * N + n) * K + P.kid);
          else if (ecf != nullptr) prefetch_l2(ecf + (size_t)n * KP + P.kp);
        }
    }
    __syncthreads();
    if (CURL && wi < 4) {  // d/dz of the first two: a warp per (component, parity)
      const T* x = sx + (size_t)(wi >> 1) * N * 32 + lane;
      T* d = sx + (size_t)(3 + (wi >> 1)) * N * 32 + lane;
      T v = (T)0;
      for (int n = N - 1 - ((N - 1 - (wi & 1)) & 1); n >= 0; n -= 2) {
        if (n + 1 < N) v = fma(x[(n + 1) * 32], dn[n], v);
        d[n * 32] = n == 0 ? v * (T)0.5 : v;
      }
    }
    if (CURL) __syncthreads();
    fold_apply<HP>(sx, tab, N);
    T* out = reinterpret_cast<T*>(grid) + 2 * (L.col < 0 ? 0 : L.col) + part;
    for (int c = clo + wi; c <= chi; c += NW) {
      T v[5];
#pragma unroll
      for (int f = 0; f < NF; ++f) v[f] = live ? fold_out(sx + (size_t)f * N * 32 + lane, c, M) : (T)0;
      T* q = out + 2 * c * plane;
      const T ou = __shfl_xor_sync(0xffffffffu, v[0], 16), ov = __shfl_xor_sync(0xffffffffu, v[1], 16),
              ow = __shfl_xor_sync(0xffffffffu, v[2], 16);
      if (L.col >= 0) {
        q[0] = v[0];
        q[fs] = v[1];
        q[2 * fs] = v[2];
        if constexpr (CURL) {  // 1/2 (i ky w - v', u' - i kx w, i kx v - i ky u)
          q[3 * fs] = hky * ow - (T)0.5 * v[4];
          q[4 * fs] = (T)0.5 * v[3] - hkx * ow;
          q[5 * fs] = hkx * ov - hky * ou;
        }
      }
    }
  }
}

// the parts' matrices, a padded row of outputs per input, times s
std::vector<T> fold_table(int N, double s) {
  const int n1 = N - 1, h = n1 / 4, k = h / 2, pad = fold_pad(fold_bucket(N));
  std::vector<T> t(fold_table_values(N), (T)0);
  for (int r = 0; r < 4; ++r)
    for (int q = 0; q < 2; ++q) {
      const FoldPart p = fold_part_of(r, q, h);
      for (int i = 0; i < p.cnt; ++i)
        for (int j = 0; j < p.outs; ++j) {
          long long c = 0, n = 0;  // node and coefficient (or the other way round) of input i and output j
          if (r < 2 && q == 0) { c = 2 * i + 1; n = 2 * (j + r * k) + 1; }
          else if (r < 2) { c = i; n = 8 * j + 4 * r; }
          else if (r == 2) { c = 2 * i + q; n = 4 * j + 2; }
          else { c = 4 * i + 2 * q; n = 2 * j + 1; }
          t[(size_t)(p.row + i) * pad + j] = (T)(s * cos(M_PI * (double)((n * c) % (2 * n1)) / n1));
        }
    }
  return t;
}

// coefficients of e^{-k zeta} and zeta e^{-k zeta} per (kx, |ky|): a block per kp, a thread per coefficient, from
// the sums (even coefficients) and differences (odd) of mirrored nodes.  ct: [node][coefficient], so that a
// warp reads a row of it.
__global__ void fold_ecf_kernel(Geometry g, const double* __restrict__ zeta, const double* __restrict__ ct, int npad,
                                int64_t KP, double2* __restrict__ ecf) {
  extern __shared__ double2 ecf_sm[];
  const int N = g.nz, half = (N + 1) / 2;
  double2 *sum = ecf_sm, *dif = ecf_sm + half;  // [half] of both functions; the middle node (N odd) counts once
  for (int64_t kp = blockIdx.x; kp < KP; kp += gridDim.x) {
    const int kxi = (int)(kp % g.nkx), kyi = (int)(kp / g.nkx);
    const double kx = 2.0 * M_PI * (double)kxi / g.Lx, ky = 2.0 * M_PI * (double)kyi / g.Ly;
    const double kk = sqrt(kx * kx + ky * ky);
    __syncthreads();
    for (int c = threadIdx.x; c < half; c += blockDim.x) {
      const double za = zeta[c], zb = zeta[N - 1 - c], a = exp(-kk * za), b = exp(-kk * zb);
      const bool mid = c == N - 1 - c;
      sum[c] = mid ? make_double2(a, za * a) : make_double2(a + b, za * a + zb * b);
      dif[c] = mid ? make_double2(0.0, 0.0) : make_double2(a - b, za * a - zb * b);
    }
    __syncthreads();
    for (int n = threadIdx.x; n < N; n += blockDim.x) {
      const double2* f = n & 1 ? dif : sum;
      double a = 0.0, b = 0.0;
      for (int c = 0; c < half; ++c) {
        const double w = ct[(size_t)c * npad + n];
        a = fma(w, f[c].x, a);
        b = fma(w, f[c].y, b);
      }
      ecf[(size_t)n * KP + kp] = make_double2(a, b);
    }
  }
}

template <bool C, int HP>
bool fold_allow() {
  return allow_smem(fold_fwd_kernel<C, HP>) && allow_smem(fold_bwd_kernel<C, HP>);
}

template <typename F>
auto fold_dispatch(int bucket, F&& f) {
  switch (bucket) {
    case 5: return f(std::integral_constant<int, 5>());
    case 9: return f(std::integral_constant<int, 9>());
    case 13: return f(std::integral_constant<int, 13>());
    default: return f(std::integral_constant<int, 17>());
  }
}

}  // namespace

bool cheb_fold_applies(const Geometry& g, int precision) {
  return precision == DPS_FP64 && (g.nz - 1) % 8 == 0 && g.nz >= 9 && g.nz <= 129;
}

// Folding transforms whole columns; the dense kernels only read (forward) or form (backward) the occupied
// planes, whose number a call's particles decide on the device.  Where the dense ones can be the faster both are
// launched, and each leaves at once when it is the other's turn.  The largest number of planes at which the
// dense kernel is taken, from both over 17 to 129 nodes (dense over folded time at that number / at the next
// measured one; 256 x 240, forces only, free space if not said):
//   forward, any mode: 33 nodes 12: 0.95 / 1.1, 65 nodes 15: 0.93 / 1.04, 97 nodes 18: 0.98 / 1.10, 129 nodes
//   21: 0.93 / 1.10; with torques it wins by 5 to 20 % there.  All 9 planes of 9 nodes: 0.7 with torques.
//   backward: 33 nodes 8: 0.90 / 1.10, 65 nodes 16: 0.96 / 1.22, 97 nodes 16: 0.77 / 0.97, 121 nodes 24: 0.92 / 1.06,
//   129 nodes 8: 0.61 / 0.85.  Walls and curls cost the dense kernel terms for all nodes: 65 nodes 1.07 and up
//   with either; 97 nodes 0.83 with curl, 0.97 with walls, 1.09 with both; 121 nodes 16: bottom wall and curl 0.89,
//   two walls and curl 1.04; 129 nodes (per-thread kernel) 0.39 to 0.96 at 8, in free space with curl 0.76 at 16.
// Whole products of a sheet in a box 40 high (folded alone -> this): 256 x 256 x 129 with torques 5.52 -> 2.81 ms,
// 256 x 256 x 65 forces only 1.51 -> 1.02 ms.  The second launch costs 5 us.  The dense sums inside these kernels
// instead were up to three times slower backward (their table from global memory, few warps) and took registers
// from the folded form.
int fold_thin_planes(const Geometry& g, bool backward) {
  const int N = g.nz;
  if (!backward) return 9 + N / 10;
  const bool walls = g.mode != DPS_FREE, curl = g.spectral_curl != 0;
  if (N > 128) return !walls && curl ? 16 : 8;
  if (N > 97) return !walls ? 24 : (g.mode == DPS_SLIT && curl ? 0 : 16);
  if (N > 65) return walls && curl ? 0 : 16;
  if (walls || curl) return 0;
  return N > 33 ? 16 : 8;
}

size_t cheb_fold_bytes(const Geometry& g) {
  const size_t KP = (size_t)g.nkx * (g.ny / 2 + 1);
  return 2 * fold_table_values(g.nz) * sizeof(double) + (g.mode != DPS_FREE ? KP * g.nz * sizeof(double2) : 0);
}

dps_status cheb_fold_prepare(Plan& p) {
  const Geometry& g = p.g;
  const bool ok = fold_dispatch(fold_bucket(g.nz), [&](auto hp) {
    constexpr int HP = decltype(hp)::value;
    return g.spectral_curl ? fold_allow<true, HP>() : fold_allow<false, HP>();
  });
  if (!ok) return DPS_ERR_CUDA;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p.device) != cudaSuccess) return DPS_ERR_CUDA;
  const int nf = g.spectral_curl ? 5 : 3;
  p.fold_grid = sms * (2 * (fold_smem(g.nz, nf) + 1024) <= 228 * 1024 && nf == 3 ? 2 : 1);
  const size_t nt = fold_table_values(g.nz), bytes = cheb_fold_bytes(g);
  void* q = nullptr;
  if (cudaMalloc(&q, bytes) != cudaSuccess) {
    cudaGetLastError();
    return DPS_ERR_OOM;
  }
  p.kt.fold = reinterpret_cast<double*>(q);
  for (int d = 0; d < 2; ++d) p.fold_thin[d] = fold_thin_planes(g, d == 1);
  p.device_bytes += (int64_t)bytes;
  const std::vector<T> f = fold_table(g.nz, 2.0 / (g.nz - 1)), b = fold_table(g.nz, 1.0 / ((double)g.nx * (double)g.ny));
  if (cudaMemcpy(p.kt.fold, f.data(), nt * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(p.kt.fold + nt, b.data(), nt * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
    return DPS_ERR_CUDA;
  if (g.mode != DPS_FREE) {
    const int64_t KP = (int64_t)g.nkx * (g.ny / 2 + 1);
    fold_ecf_kernel<<<(unsigned)(KP < sms * 16 ? KP : sms * 16), 128, (g.nz + 1) / 2 * 2 * sizeof(double2)>>>(
        g, reinterpret_cast<const double*>(p.tab.zeta), reinterpret_cast<const double*>(p.kt.ct), p.kt.npad, KP,
        reinterpret_cast<double2*>(p.kt.fold + 2 * nt));
  }
  return cudaGetLastError() == cudaSuccess ? DPS_OK : DPS_ERR_CUDA;
}

void launch_cheb_fold(const Plan& p, bool backward, int kx0, int w, cudaStream_t s) {
  const Geometry& g = p.g;
  const int64_t tiles = ((int64_t)w * g.ny + kFoldK - 1) / kFoldK;
  const size_t nt = fold_table_values(g.nz);
  cplx<T>* grid = reinterpret_cast<cplx<T>*>(p.grid);
  cplx<T>* kbuf = reinterpret_cast<cplx<T>*>(p.kt.kbuf);
  const cplx<T>* kaux = reinterpret_cast<const cplx<T>*>(p.kt.kaux);
  const int nf = g.spectral_curl ? 5 : 3;
  const size_t smem = fold_smem(g.nz, nf);
  const unsigned blocks = (unsigned)(tiles < p.fold_grid ? tiles : p.fold_grid);
  const double2* ecf = g.mode != DPS_FREE ? reinterpret_cast<const double2*>(p.kt.fold + 2 * nt) : nullptr;
  const int64_t KP = (int64_t)g.nkx * (g.ny / 2 + 1);
  const double hx = M_PI / g.Lx, hy = M_PI / g.Ly;
  const int thin = p.fold_thin[backward];
  fold_dispatch(fold_bucket(g.nz), [&](auto hp) {
    constexpr int HP = decltype(hp)::value;
    const int th = 32 * 4 * nf;
    if (!backward && g.spectral_curl)
      fold_fwd_kernel<true, HP><<<blocks, th, smem, s>>>(g, p.kt.fold, grid, kbuf, p.zrange, kx0, w, hx, hy, thin);
    else if (!backward)
      fold_fwd_kernel<false, HP><<<blocks, th, smem, s>>>(g, p.kt.fold, grid, kbuf, p.zrange, kx0, w, hx, hy, thin);
    else if (g.spectral_curl)
      fold_bwd_kernel<true, HP><<<blocks, th, smem, s>>>(g, p.kt.fold + nt, ecf, KP, kbuf, kaux, grid, p.zrange, kx0, w,
                                                           hx, hy, thin);
    else
      fold_bwd_kernel<false, HP><<<blocks, th, smem, s>>>(g, p.kt.fold + nt, ecf, KP, kbuf, kaux, grid, p.zrange, kx0,
                                                            w, hx, hy, thin);
  });
}

}  // namespace dps
