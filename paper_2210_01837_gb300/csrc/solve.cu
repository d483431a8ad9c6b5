// Tiled solve of the per-wavenumber boundary-value problems (steps 3-5 of Sec. III.D) from a plan-time
// table, for nz <= 128.
//
// The FP64 pipe has half a lane per clock and SM sub-partition: a warp instruction keeps it busy for 64
// clocks.  A thread per wavenumber (solve_tab_kernel) runs 4 N dependent rows for its eight real right-hand
// sides, so a small problem waits on latency with most SMs idle, and at ordinary sizes the last pass of
// the resident grid is nearly empty.  Here the unit of work is one real right-hand side of one parity: a
// tile is 16 wavenumbers, lanes 0-15 their real and 16-31 their imaginary parts, and the eight
// (right-hand side, parity) systems of a tile are the eight warps of a block, two per sub-partition: warps
// 0-5 the three velocity components, 6-7 the pressure.  The velocities need the pressure, so the block is
// a pipeline over its tiles: in step s the pressure warps work on tile s and the velocity warps on tile
// s - 1, one barrier a step.  Sweep values live in shared memory, so the DRAM traffic falls from 4.8 to
// 1.3 GB at 768 x 768 x 65 (spectra and table).
//
// Measured (solve alone, GB300, thread per wavenumber -> this): 120 x 120 x 33 mixed 155 -> 46 us,
// 128 x 128 x 65 double 434 -> 170 us, 768 x 768 x 65 mixed 1.72 -> 1.38 ms, 3072 x 3072 x 65 mixed
// 23.2 -> 21.8 ms.  It is bound by the FP64 pipe, 77 % busy there (16 warps an SM, the slabs' shared memory, and
// a barrier a step leave the rest).  The sweeps run in double in float plans too, as the boundary sums do:
// 64-bit fixed-point sweeps on the integer pipe took the same time (1.40 and 22.3 ms), lost bits in the small
// entries of a column and turned an overflow into finite numbers.
#include "bvp_device.cuh"
#include "dps_internal.cuh"

namespace dps {
namespace {

constexpr int kSolveK = 16;       // wavenumbers per tile
constexpr int kSolveWarps = 8;    // 3 velocity components + pressure, two parities each
constexpr int kSolveThreads = 32 * kSolveWarps;
constexpr size_t kMaxBlockSmem = 227 * 1024;  // shared memory a block can have
// wavenumber constants and wall amplitudes are long serial chains on the FP64 pipe (a square root; up to
// divisions and an exponential): they are done for 8 tiles at a time, two tiles a warp, one warp on each
// sub-partition, so that they hold up one step in eight
constexpr int kGroup = 8;
constexpr int kVRing = kGroup + 1;

// one wavenumber of a tile; kid < 0: beyond the last wavenumber
struct KEnt {
  double kx, ky, kk, ik;
  int kid, kp;
};

template <typename T>
struct SolveSmem {
  double* sw;   // [8][(N + 1) / 2][32] a slab per warp: its system's right-hand sides, then sweep values
  double* pv;   // [2][2][32] pressure at the walls by parity
  double* vv;   // [kVRing][6][32] velocity at the walls by (component, parity)
  double* dv;   // [kVRing][4][32] its s derivative (slip)
  KEnt* ki;     // [2 kGroup][16]
  T* p;         // [2][N][32] pressure coefficients
  T* tl;        // [N] B B map in the transform precision
  T* td;
  T* tu;
  int n;        // N
};

__host__ __device__ inline int solve_rows(int N) { return (N + 1) / 2; }

template <typename T>
__host__ __device__ inline size_t solve_smem_bytes(int N, bool slip) {
  size_t d = (size_t)kSolveWarps * solve_rows(N) * 32 + 2 * 2 * 32 + kVRing * 6 * 32 + (slip ? kVRing * 4 * 32 : 0);
  return d * sizeof(double) + 2 * kGroup * kSolveK * sizeof(KEnt) + (2 * (size_t)N * 32 + 3 * (size_t)N) * sizeof(T);
}

template <typename T>
__device__ __forceinline__ SolveSmem<T> solve_smem(unsigned char* base, int N, bool slip) {
  SolveSmem<T> m;
  double* d = reinterpret_cast<double*>(base);
  m.sw = d; d += (size_t)kSolveWarps * solve_rows(N) * 32;
  m.pv = d; d += 2 * 2 * 32;
  m.vv = d; d += kVRing * 6 * 32;
  m.dv = d; if (slip) d += kVRing * 4 * 32;
  m.ki = reinterpret_cast<KEnt*>(d);
  m.p = reinterpret_cast<T*>(m.ki + 2 * kGroup * kSolveK);
  m.tl = m.p + 2 * (size_t)N * 32;
  m.td = m.tl + N;
  m.tu = m.td + N;
  m.n = N;
  return m;
}

// Rows in two batches of B in registers: while the rows of one are used, the loads of the other are in
// flight (a batch's loads are waited for together, so rows ahead of it never hold a wait back).  Rows run
// from `from` to `to` (at least one) in steps of D (1 or -1); load(r, more) reads the next row and, with
// more, moves on, so reads past the last row repeat it and nothing branches around a load.
template <int B, int D, typename R, typename Load>
__device__ __forceinline__ void rows_fetch(R (&r)[B], int i, int to, Load&& load) {
#pragma unroll
  for (int u = 0; u < B; ++u) load(r[u], D > 0 ? i + D * u < to : i + D * u > to);
}
// x: the first batch, fetched by the caller with rows_fetch (early, so that its latency is hidden too)
template <int B, int D, typename R, typename Load, typename Use>
__device__ __forceinline__ void rows_ahead(R (&x)[B], int from, int to, Load&& load, Use&& use) {
  R y[B];
  auto work = [&](R(&r)[B], int i) {
#pragma unroll
    for (int u = 0; u < B; ++u)
      if (D > 0 ? i + D * u <= to : i + D * u >= to) use(i + D * u, r[u]);
  };
#pragma unroll 1
  for (int i = from; D > 0 ? i <= to : i >= to; i += 2 * B * D) {
    rows_fetch<B, D, R>(y, i + B * D, to, load);
    work(x, i);
    rows_fetch<B, D, R>(x, i + 2 * B * D, to, load);
    work(y, i + B * D);
  }
}

// The plan-time table per (kx, |ky|), kp = |kyi| nkx + kxi: what the systems of a wavenumber need, which
// depends on |k| only.  Row n of parity par (n > par): gw = (gamma, omega), -V_n, -t_n, rho_n; per parity
// the boundary rows edge[par][7]: U, and with det = D' beta_a + k^2 b: beta_a / det, k^2 / det, D' / det,
// b / det, then the weight of c_par in the wall value and (slip) in the wall derivative.
template <typename T> struct Rows;
template <typename T>
struct SolveTable {
  double2* gw;     // [N][KP]
  double* edge;    // [2][7][KP]
  double* V;       // [N][KP]
  double* t;       // [N][KP]
  double* wd;      // [N][KP], slip only
  T* rho;          // [N][KP]
  int64_t KP;
  __device__ __forceinline__ Rows<T> rows(int par, int kp) const;
};

template <typename T>
__host__ inline size_t solve_table_bytes(const Geometry& g, int64_t KP) {
  return (size_t)KP * ((size_t)g.nz * (16 + 8 + 8 + (g.slip ? 8 : 0) + sizeof(T)) + 14 * sizeof(double));
}

template <typename T>
__host__ inline SolveTable<T> solve_table(const Plan& p) {
  const size_t n = (size_t)p.g.nz * p.kt.KP;
  SolveTable<T> t;
  t.KP = p.kt.KP;
  t.gw = reinterpret_cast<double2*>(p.kt.fac);
  t.edge = reinterpret_cast<double*>(t.gw + n);
  t.V = t.edge + 14 * (size_t)t.KP;
  t.t = t.V + n;
  t.wd = p.g.slip ? t.t + n : nullptr;
  t.rho = p.g.slip ? reinterpret_cast<T*>(t.wd + n) : reinterpret_cast<T*>(t.t + n);
  return t;
}

// the rows of one system's table entries (row n = par + 2 i), a lane's wavenumber
template <typename T>
struct Rows {
  const double2* gw;      // gamma, omega
  const double* wd;       // omega of the derivative (slip)
  const double *V, *t;    // -V_n and -t_n
  const T* rho;
  int64_t KP;
};

template <typename T>
__device__ __forceinline__ Rows<T> SolveTable<T>::rows(int par, int kp) const {
  const size_t o = (size_t)par * KP + kp;
  return Rows<T>{gw + o, wd ? wd + o : nullptr, V + o, t + o, rho + o, KP};
}

// A real system takes three passes.  Pass 1 forms the scaled right-hand sides r'_i = r_i rho_i in the transform precision
// (rhs(i, x) from the values that load(i, x) fetched), keeps them in the slab, widened, and adds up the boundary
// row and the wall value as functionals of them, in double: g -= sum gamma_i r'_i, q = sum omega_i r'_i
// (adjoints of the two sweeps, formed when the plan is made).  These sums have no serial part, so a warp
// can fill its FP64 pipe.  Pass 2 is the elimination s_i = r'_i - V_i s_{i+1}, i = il .. 1, pass 3 the
// substitution (sweeps).
template <typename T, bool SLIP, typename In, typename Load, typename Rhs>
__device__ __forceinline__ void functionals(int il, const Rows<T>& tb, double* slab, int lane, double& g, double& q,
                                            double& qd, Load&& load, Rhs&& rhs) {
  struct Row {
    double2 gw;
    double wd;
    T rho;
    In in;
  };
  double* rr = slab + lane;
  const size_t st = 2 * (size_t)tb.KP;
  const double2* pg = tb.gw + il * st;
  const double* pw = SLIP ? tb.wd + il * st : nullptr;
  const T* pr = tb.rho + il * st;
  auto fetch = [&](Row& x, bool more) {
    x.gw = *pg;
    x.rho = *pr;
    if (SLIP) x.wd = *pw;
    if (more) {
      pg -= st;
      pr -= st;
      if (SLIP) pw -= st;
    }
    load(x.in, more);
  };
  Row x[3];
  rows_fetch<3, -1, Row>(x, il, 1, fetch);
  rows_ahead<3, -1, Row>(x, il, 1, fetch, [&](int i, const Row& v) {
    const double d = widen<T>(rhs(i, v.in) * v.rho);
    rr[i * 32] = d;
    g = fma(-v.gw.x, d, g);
    q = fma(v.gw.y, d, q);
    if (SLIP) qd = fma(v.wd, d, qd);
  });
}

// a coefficient in the transform precision, to nearest (narrow truncates; these enter the output)
__device__ __forceinline__ void round_to(double d, double& v) { v = d; }
__device__ __forceinline__ void round_to(double d, float& v) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned s = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ffu) - 896;
  const unsigned m = ((unsigned)e << 23 | (hi & 0xfffffu) << 3 | lo >> 29) + (lo >> 28 & 1u);  // may carry into e
  v = __uint_as_float(s | (e <= 0 ? 0u : e >= 255 ? 0x7f800000u : m));
}

// Passes 2 and 3 of a system: the elimination in place and s_1 from it, the 2 x 2 boundary system for c_0 and
// a, and the substitution c_i = s_i - t_i c_{i-1} with y = B B c (+ a in row 0) handed to put(i, y) in the
// transform precision.  Returns the wall value's and (qd) the wall derivative's part of this parity.
template <typename T, bool SLIP, typename Put>
__device__ __forceinline__ double sweeps(int il, int par, const Rows<T>& tb, const double* __restrict__ edge,
                                         double* slab, int lane, const SolveSmem<T>& m, T r0, double g, double q,
                                         double& qd, Put&& put) {
  const size_t st = 2 * (size_t)tb.KP;
  const int64_t KP = tb.KP;
  const double* pv = tb.V + il * st;
  const double* pt = tb.t + st;
  auto fv = [&](double& x, bool more) {
    x = *pv;
    if (more) pv -= st;
  };
  auto ft = [&](double& x, bool more) {
    x = *pt;
    if (more) pt += st;
  };
  double v[4], t[4];
  rows_fetch<4, -1, double>(v, il, 1, fv);
  const double U = edge[0], cb = edge[KP], ck = edge[2 * KP], cd = edge[3 * KP], cc = edge[4 * KP], w0 = edge[5 * KP];
  const double w0d = SLIP ? edge[6 * KP] : 0.0;
  rows_fetch<4, 1, double>(t, 1, il, ft);
  double* sw = slab + lane;
  double s = 0.0;
  rows_ahead<4, -1, double>(v, il, 1, fv, [&](int i, double f) {
    s = fma(f, s, sw[i * 32]);
    sw[i * 32] = s;
  });
  const double rh = fma(-s, U, widen<T>(r0));
  const double c0 = fma(g, ck, rh * cb), a = fma(g, cd, -(rh * cc));
  T ta, c1, c2 = (T)0;
  round_to(a, ta);
  round_to(c0, c1);
  auto row = [&](int i, T cn) {  // row i of y, whose neighbours c_{i-1} and c_{i+1} = cn are known now
    const int n = par + 2 * i;
    const T y = (c1 * m.td[n] + cn * m.tu[n]) + c2 * m.tl[n];  // c2 = 0 in row 0
    put(i, y + (i == 0 ? ta : (T)0));
    c2 = c1;
    c1 = cn;
  };
  double c = c0;
  rows_ahead<4, 1, double>(t, 1, il, ft, [&](int i, double f) {
    c = fma(f, c, sw[i * 32]);
    T cn;
    round_to(c, cn);
    row(i - 1, cn);
  });
  row(il, (T)0);
  if (SLIP) {
    qd = fma(c0, w0d, qd);
    if (par) qd = qd + a;  // a1 T_1 has y_s = a1
  }
  return fma(c0, w0, q) + a;
}

// k = 0 (Sec. III.C, Eqs. 47-52; Appendix A, Eq. A12) by one warp, the rows over its lanes; the same
// rows as zero_mode of the thread-per-wavenumber solves.
template <typename T, bool SLIP>
__device__ __noinline__ void zero_mode_warp(const Geometry& g, const double* __restrict__ band, cplx<T>* __restrict__ kbuf,
                                            cplx<T>* __restrict__ kaux, cplx<double>* __restrict__ sc, int64_t K) {
  const int N = g.nz, lane = threadIdx.x & 31;
  const double *bl = band, *bd = band + N, *bu = band + 2 * N, *bP = band + 3 * N, *bQ = band + 4 * N;
  __syncwarp();  // sc is the warp's slab: its sweeps have read their columns before other lanes write over them
  auto sum = [](cplx<double> v) {
    for (int o = 16; o; o >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
  };
  for (int o = 0; o < 3; ++o) {
    cplx<T>* kb = kbuf + (size_t)o * N * K;
    if (g.mode == DPS_FREE || o == 2) {
      for (int n = lane; n < N; n += 32) kb[(size_t)n * K] = mk<T>((T)0, (T)0);
      continue;
    }
    cplx<double> Sp = mk<double>(0, 0), Sm = mk<double>(0, 0), Pd = mk<double>(0, 0), Pm = mk<double>(0, 0);
    for (int n = lane; n < N; n += 32) {
      const cplx<double> cn = scl(wid(kb[(size_t)n * K]), -g.inv_eta / (g.sH * g.sH));
      sc[n] = cn;
      const double sgn = (n & 1) ? -1.0 : 1.0;
      Sp = Sp + scl(cn, bQ[n]);
      Sm = Sm + scl(cn, sgn * bQ[n]);
      Pd = Pd + scl(cn, bP[n]);
      if (SLIP) Pm = Pm + scl(cn, sgn * bP[n]);
    }
    Sp = sum(Sp);
    Sm = sum(Sm);
    Pd = sum(Pd);
    if (SLIP) Pm = sum(Pm);
    __syncwarp();
    cplx<double> a0, a1;
    if (SLIP) {  // Robin rows, as in zero_mode
      const double nxy = (double)g.nx * (double)g.ny;
      const double al = 1.0 + g.slip0 * g.sH;
      const cplx<double> Rb = mk<double>(nxy * g.uw0[o], 0.0) - Sm - scl(Pm, g.slip0 * g.sH);
      if (g.mode == DPS_BOTTOM_WALL) {
        a1 = scl(Pd, -1.0);
        a0 = Rb + scl(a1, al);
      } else {
        const double be = 1.0 + g.slipH * g.sH;
        const cplx<double> Rt = mk<double>(nxy * g.uwH[o], 0.0) - Sp - scl(Pd, g.slipH * g.sH);
        a1 = scl(Rt - Rb, 1.0 / (al + be));
        a0 = Rb + scl(a1, al);
      }
    } else if (g.mode == DPS_BOTTOM_WALL) {  // y(-1) = 0, y_s(+1) = 0
      a1 = scl(Pd, -1.0);
      a0 = a1 - Sm;
    } else {  // y(-1) = y(+1) = 0
      a0 = scl(Sp + Sm, -0.5);
      a1 = scl(Sp - Sm, -0.5);
    }
    for (int n = lane; n < N; n += 32) {
      cplx<double> y = scl(sc[n], bd[n]);
      if (n >= 2) y = y + scl(sc[n - 2], bl[n]);
      if (n + 2 < N) y = y + scl(sc[n + 2], bu[n]);
      if (n == 0) y = y + a0;
      if (n == 1) y = y + a1;
      kb[(size_t)n * K] = nar<T>(y);
    }
    __syncwarp();
  }
  for (int q = lane; q < 12; q += 32) kaux[(size_t)q * K] = mk<T>((T)0, (T)0);
}

// wall amplitudes of one wavenumber per lane from the wall values by parity; out of line, so that its
// registers do not weigh on the sweeps
template <typename T, bool SLIP>
__device__ __noinline__ void tile_amplitudes(const Geometry& g, const KEnt& ent, const double* vv, const double* dv,
                                             cplx<T>* __restrict__ kaux, int64_t K) {
  const KEnt e = ent;
  if (e.kid <= 0) return;
  cplx<double> vtop[3], vbot[3], dtop[2], dbot[2];
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    const cplx<double> ev = mk<double>(vv[(2 * f) * 32], vv[(2 * f) * 32 + 16]);
    const cplx<double> od = mk<double>(vv[(2 * f + 1) * 32], vv[(2 * f + 1) * 32 + 16]);
    vtop[f] = ev + od;
    vbot[f] = ev - od;
  }
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    dtop[f] = dbot[f] = mk<double>(0, 0);
    if (SLIP) {  // T_n'(-1) = (-1)^(n+1) n^2
      const cplx<double> ev = mk<double>(dv[(2 * f) * 32], dv[(2 * f) * 32 + 16]);
      const cplx<double> od = mk<double>(dv[(2 * f + 1) * 32], dv[(2 * f + 1) * 32 + 16]);
      dtop[f] = ev + od;
      dbot[f] = od - ev;
    }
  }
  wall_amplitudes<T, SLIP>(g, e.kx, e.ky, e.kk, e.ik, vtop, vbot, dtop, dbot, kaux, e.kid, K);
}

template <typename T, bool SLIP>
__global__ void __launch_bounds__(kSolveThreads, 2) solve_tile_kernel(const __grid_constant__ Geometry g, const double* __restrict__ band,
                                                                     const T* __restrict__ bandT,
                                                                     const __grid_constant__ SolveTable<T> tab, cplx<T>* __restrict__ kbuf,
                                                                     cplx<T>* __restrict__ kaux, int kx0, int w,
                                                                     double tpx, double tpy) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int N = g.nz;
  const SolveSmem<T> m = solve_smem<T>(smraw, N, SLIP);
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int part = lane >> 4, kc = lane & 15;
  const int64_t K = (int64_t)g.nkx * g.ny, KP = tab.KP;
  // the wavenumbers to solve, in the order ky = 0, 1, -1, 2, -2, ... (the two that share table rows
  // within one pass of the grid, so the second read hits L2); Nyquist columns and rows are left out
  const int W = (g.nx % 2 == 0 && kx0 + w == g.nkx) ? w - 1 : w;
  const int rows = g.ny - (g.ny % 2 == 0 ? 1 : 0);
  const int64_t total = (int64_t)W * rows;
  const int64_t ntiles = (total + kSolveK - 1) / kSolveK;
  const int nt = (int)((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x);  // tiles of this block
  auto entry = [&](int t0) {  // by one warp: tiles t0 and t0 + 1 of the block into ki
    const int t = t0 + part;
    const int64_t i = ((int64_t)t * gridDim.x + blockIdx.x) * kSolveK + kc;
    KEnt e;
    e.kx = e.ky = e.kk = e.ik = 0.0;
    e.kid = -1;
    e.kp = 0;
    if (t < nt && i < total) {
      const int j = (int)((unsigned)i / (unsigned)W);
      const int kxi = kx0 + (int)((unsigned)i - (unsigned)j * (unsigned)W);
      const int kyi = (j == 0) ? 0 : ((j & 1) ? (j + 1) >> 1 : g.ny - (j >> 1));
      const int nyv = (kyi < (g.ny + 1) / 2) ? kyi : kyi - g.ny;
      e.kid = kyi * g.nkx + kxi;
      e.kp = ((2 * kyi <= g.ny) ? kyi : g.ny - kyi) * g.nkx + kxi;
      e.kx = tpx * (double)kxi;
      e.ky = tpy * (double)nyv;
      const double k2 = e.kx * e.kx + e.ky * e.ky;
      e.ik = (e.kid == 0) ? 0.0 : rsqrt(k2);
      e.kk = k2 * e.ik;
    }
    m.ki[(t & 15) * kSolveK + kc] = e;
  };
  for (int i = threadIdx.x; i < N; i += kSolveThreads) {
    m.tl[i] = bandT[i];
    m.td[i] = bandT[N + i];
    m.tu[i] = bandT[2 * N + i];
  }
  if (wi < kGroup / 2) entry(2 * wi);
  const T tsH = (T)g.sH, tie = (T)g.inv_eta;
  const int par = wi & 1;
  const int il = (N - 1 - par) >> 1;  // last row index of this parity
  double* slab = m.sw + (size_t)wi * solve_rows(N) * 32;
  const double* edge = tab.edge + (size_t)par * 7 * KP;

  for (int s = 0; s < nt + 2; ++s) {
    __syncthreads();  // tile s's and s + 1's constants, tile s - 1's pressure, tile s - 2's wall values
    if (s % kGroup == kGroup / 2 && wi >= kGroup / 2) entry(s + kGroup / 2 + 2 * (wi - kGroup / 2));
    if (s + 1 < nt) {  // the next tile's spectra and table rows into L2
      const KEnt* e = m.ki + ((s + 1) & 15) * kSolveK;
      const int a = e[0].kid, b = e[kSolveK - 1].kid < 0 ? a : e[kSolveK - 1].kid;
      const int pa = e[0].kp, pb = e[kSolveK - 1].kp;
      const int ke = part ? b : a, kq = part ? (b == a ? pa : pb) : pa;  // half of the lanes at either end
      if (wi == kSolveWarps - 1 && kc < 14) prefetch_l2(tab.edge + kc * KP + kq);
      for (int n = wi * 16 + kc; n < N; n += 16 * kSolveWarps) {
        prefetch_l2(kbuf + (size_t)n * K + ke);
        prefetch_l2(kbuf + (size_t)(N + n) * K + ke);
        prefetch_l2(kbuf + (size_t)(2 * N + n) * K + ke);
        prefetch_l2(tab.gw + n * KP + kq);
        prefetch_l2(tab.V + n * KP + kq);
        prefetch_l2(tab.t + n * KP + kq);
        prefetch_l2(tab.rho + n * KP + kq);
        if (SLIP) prefetch_l2(tab.wd + n * KP + kq);
      }
    }
    if (wi >= 6 && s < nt) {
      // ---- pressure of tile s: (D^2 - k^2) p = i kx f + i ky g + D h, DtN rows with zero data ------
      const KEnt& e = m.ki[(s & 15) * kSolveK + kc];
      const int kid = e.kid < 0 ? 0 : e.kid, kp = e.kp;
      const Rows<T> tb = tab.rows(par, kp);
      const T sx = part ? (T)e.kx : -(T)e.kx, sy = part ? (T)e.ky : -(T)e.ky;
      // f and g enter through their other part (i k), h through the lane's own
      const size_t rs = 2 * (size_t)K, fs = (size_t)N * rs;
      const T* fb = reinterpret_cast<const T*>(kbuf + kid) + (1 - part) + par * rs;
      const T* hb = reinterpret_cast<const T*>(kbuf + (size_t)2 * N * K + kid) + part + (par + 1) * rs;
      const T f0 = fb[0], q0 = fb[fs], h0 = (par + 1 < N) ? hb[0] : (T)0;
      struct In { T f, q, h; };
      fb += 2 * il * rs;
      bool no_h = par + 2 * il + 1 == N;  // the last row has no row of h above it
      hb += 2 * (no_h ? il - 1 : il) * rs;
      T dh = (T)0;  // derivative recurrence of h over the opposite parity
      double ga = 0.0, q = 0.0, qd = 0.0;
      functionals<T, false, In>(
          il, tb, slab, lane, ga, q, qd,
          [&](In& x, bool more) {
            x.f = fb[0];
            x.q = fb[fs];
            x.h = hb[0];
            if (more) {
              fb -= 2 * rs;
              if (!no_h) hb -= 2 * rs;
              no_h = false;
            }
          },
          [&](int i, const In& x) {
            const int n = par + 2 * i;
            dh = dh + x.h * (n + 1 < N ? (T)(2 * (n + 1)) : (T)0);
            return sx * x.f + sy * x.q + tsH * dh;
          });
      dh = dh + h0 * (T)(2 * (par + 1));
      if (par == 0) dh = dh * (T)0.5;
      T* po = m.p + (size_t)(s & 1) * N * 32 + par * 32 + lane;
      m.pv[((s & 1) * 2 + par) * 32 + lane] =
          sweeps<T, false>(il, par, tb, edge + kp, slab, lane, m, sx * f0 + sy * q0 + tsH * dh, ga, q, qd,
                           [&](int i, T y) {
                             po[i * 64] = y;
                           });
    } else if (wi < 6 && s >= 1 && s <= nt) {
      // ---- velocity of tile s - 1 -------------------------------------------------------------------
      const int t = s - 1, f = wi >> 1;
      const KEnt& e = m.ki[(t & 15) * kSolveK + kc];
      const int kid = e.kid < 0 ? 0 : e.kid, kp = e.kp;
      const Rows<T> tb = tab.rows(par, kp);
      const T* pi = m.p + (size_t)(t & 1) * N * 32;
      const double* pw = m.pv + (t & 1) * 2 * 32;
      const size_t rs = 2 * (size_t)K;
      T* const y0 = reinterpret_cast<T*>(kbuf + (size_t)f * N * K + kid) + part + par * rs;
      const T v0 = __ldcs(y0);
      double ga, q = 0.0, qd = 0.0;
      const T* yb = y0 + 2 * il * rs;
      T r0;
      if (f < 2) {
        // DtN data -(i k_f / (2 eta k)) p above, + below: (top +- bottom) / 2 by parity
        const double kf = (f == 0) ? e.kx : e.ky;
        const double z = kf * (0.5 * g.inv_eta * e.ik);
        ga = (part ? -z : z) * pw[par * 32 + (lane ^ 16)];
        const T sk = part ? (T)kf : -(T)kf;
        const T* po = pi + par * 32 + (lane ^ 16);
        functionals<T, SLIP, T>(
            il, tb, slab, lane, ga, q, qd,
            [&](T& x, bool more) {
              x = __ldcs(yb);
              if (more) yb -= 2 * rs;
            },
            [&](int i, T x) { return (po[i * 64] * sk - x) * tie; });
        r0 = (po[0] * sk - v0) * tie;
      } else {
        ga = (0.5 * g.inv_eta) * pw[(par ^ 1) * 32 + lane];
        const T* po = pi + (par + 1) * 32 + lane;
        T dp = (T)0;
        auto deriv = [&](int i) {  // the rows' derivative recurrence of p over the opposite parity
          const int n = par + 2 * i;
          if (n + 1 < N) dp = dp + po[i * 64] * (T)(2 * (n + 1));
        };
        functionals<T, false, T>(
            il, tb, slab, lane, ga, q, qd,
            [&](T& x, bool more) {
              x = __ldcs(yb);
              if (more) yb -= 2 * rs;
            },
            [&](int i, T x) {
              deriv(i);
              return (dp * tsH - x) * tie;
            });
        deriv(0);
        if (par == 0) dp = dp * (T)0.5;
        r0 = (dp * tsH - v0) * tie;
      }
      const bool keep = e.kid > 0;  // not beyond the end, not k = 0
      T* yo = y0;
      const int slot = t % kVRing;
      const double vw = sweeps<T, SLIP>(il, par, tb, edge + kp, slab, lane, m, r0, ga, q, qd, [&](int, T y) {
        if (keep) __stcs(yo, y);
        yo += 2 * rs;
      });
      m.vv[(slot * 6 + wi) * 32 + lane] = vw;
      if (SLIP && f < 2) m.dv[(slot * 4 + wi) * 32 + lane] = qd;
    }
    if (s == 2 && wi == 7 && blockIdx.x == 0 && kx0 == 0 && nt > 0)  // tile 0's readers are done
      zero_mode_warp<T, SLIP>(g, band, kbuf, kaux, reinterpret_cast<cplx<double>*>(slab), K);
    // ---- wall amplitudes of a finished group, a wavenumber per lane, two tiles a warp ------------------
    const bool last = s == nt + 1;
    if (wi < kGroup / 2 && (last || (s > kGroup && (s - 1) % kGroup == 0))) {
      const int t = (last ? (nt - 1) / kGroup * kGroup : s - 1 - kGroup) + 2 * wi + part;
      if (t < nt) tile_amplitudes<T, SLIP>(g, m.ki[(t & 15) * kSolveK + kc], m.vv + (t % kVRing) * 6 * 32 + kc,
                                           m.dv + (t % kVRing) * 4 * 32 + kc, kaux, K);
    }
  }
}

// The table, a thread per (kx, |ky|): the elimination from the last row down (as factor_kernel's), the folded
// weights b of the boundary row and w of the wall value on the way, then their adjoints over the
// elimination, gamma_n = b_n - V_{n-2} gamma_{n-2}, omega_n = w_n - V_{n-2} omega_{n-2}.
template <typename T>
__global__ void solve_table_kernel(Geometry g, const double* __restrict__ band, SolveTable<T> tab) {
  const int64_t KP = tab.KP, kp = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (kp >= KP) return;
  const int N = g.nz;
  const int kxi = (int)(kp % g.nkx), kyi = (int)(kp / g.nkx);
  const double *bl = band, *bd = band + N, *bu = band + 2 * N, *bP = band + 3 * N, *bQ = band + 4 * N;
  const double kx = 2.0 * M_PI * (double)kxi / g.Lx, ky = 2.0 * M_PI * (double)kyi / g.Ly;
  const double kk = sqrt(kx * kx + ky * ky), kap = kk * kk;
  const double sH = 2.0 / g.H, sig = sH * sH;
  for (int par = 0; par < 2; ++par) {
    const int nlast = ((N - 1 - par) & 1) ? N - 2 : N - 1;
    double t_next = 0.0, b = sH * bP[nlast] + kk * bQ[nlast], w = 0.0, wd = 0.0;
    for (int n = nlast; n > par; n -= 2) {
      const size_t o = (size_t)n * KP + kp;
      const double U = -kap * bu[n];
      const double rho = 1.0 / ((sig - kap * bd[n]) - U * t_next);
      const double t = rho * (-kap * bl[n]);
      w = bQ[n] - t_next * w;
      wd = bP[n] - t_next * wd;
      tab.gw[o] = make_double2(b, w);
      if (tab.wd) tab.wd[o] = wd;
      tab.V[o] = U * rho;
      tab.t[o] = -t;
      tab.rho[o] = (T)rho;
      b = (sH * bP[n - 2] + kk * bQ[n - 2]) - b * t;
      t_next = t;
    }
    double* e = tab.edge + (size_t)par * 7 * KP + kp;
    const double U = -kap * bu[par], Dp = (sig - kap * bd[par]) - U * t_next;
    const double beta = par == 0 ? kk : sH + kk;
    const double idet = kk > 0.0 ? 1.0 / (Dp * beta + kap * b) : 0.0;  // k = 0 is solved apart
    e[0] = U;
    e[KP] = beta * idet;
    e[2 * KP] = kap * idet;
    e[3 * KP] = Dp * idet;
    e[4 * KP] = b * idet;
    e[5 * KP] = bQ[par] - t_next * w;
    e[6 * KP] = bP[par] - t_next * wd;
    double V = 0.0, ga = 0.0, om = 0.0, od = 0.0;
    for (int n = par + 2; n <= nlast; n += 2) {
      const size_t o = (size_t)n * KP + kp;
      const double2 x = tab.gw[o];
      ga = x.x - V * ga;
      om = x.y - V * om;
      tab.gw[o] = make_double2(ga, om);
      if (tab.wd) {
        od = tab.wd[o] - V * od;
        tab.wd[o] = od;
      }
      V = tab.V[o];
      tab.V[o] = -V;
    }
  }
}

}  // namespace

// Where it is the faster one.  P: wavenumbers in passes of the thread-per-wavenumber solve's grid; figures are
// that solve's time over this one's, without walls / with (whose amplitudes lengthen its one thread's chain).
//  - Up to one pass the other solve waits on the latency of one thread's serial rows: 120 x 120 x 33 155 -> 47 us.
//    Where two blocks fit an SM (up to 70 nodes in float) this one wins at every size but the fullest pass:
//    33 nodes, P = 0.14 2.7 / 3.4, 0.57 1.3 / 1.8, 0.97 1.04 / 1.4; 33 in double 2.1 / 2.7, 1.07 / 1.3, 0.94 / 1.08.
//    Where only one fits, it covers less of its own latencies: 97 nodes, P = 0.28 1.46 / 2.2, 0.5 1.02 / 1.6,
//    0.57 0.86 / 1.3, 0.88 0.70 / 1.03; in double 1.3 / 1.7, 1.03 / 1.3, 0.88 / 1.14, 0.87 / 1.02.
//  - Beyond, it needs two blocks an SM (97 nodes, P = 5 0.72 / 0.78) and columns long enough to outweigh a tile's
//    fixed part.  Float from 33 nodes on wins at every size (P = 1.27 1.34 / 1.6, 5 1.15 / 1.16, 81 1.03 / 1.01).
//    Shorter columns and double win by the other's last pass while that counts: 25 nodes, P = 1.27 1.25 / 1.5,
//    5 1.06 / 1.07, 7 0.97 / 0.97, 81 0.94 / 0.94; 33 in double 1.2 / 1.3, 1.02 / 1.05, 0.97 / 0.97.
// In every case a block has to fit: in double with wall conditions, whose derivatives take 9 KB more, 127 and
// 128 nodes do not.
template <typename T>
bool solve_tile_applies_t(const Geometry& g) {
  const size_t b = solve_smem_bytes<T>(g.nz, g.slip != 0);
  if (g.nz > 128 || b > kMaxBlockSmem) return false;
  const bool two = 2 * (b + 1024) <= 228 * 1024;
  const double passes = (double)g.nkx * g.ny / (152.0 * 3 * kBvpThreads);
  if (passes <= 1.0) return two || passes <= (g.mode == DPS_FREE ? 0.5 : 0.9);
  return two && g.nz >= 25 && ((sizeof(T) == 4 && g.nz >= 33) || passes <= 6.0);
}

bool solve_tile_applies(const Geometry& g, int precision) {
  return precision == DPS_MIXED ? solve_tile_applies_t<float>(g) : solve_tile_applies_t<double>(g);
}

template <typename T>
int solve_tile_prepare(const Plan& p) {
  if (!allow_smem(solve_tile_kernel<T, false>) || !allow_smem(solve_tile_kernel<T, true>)) return 0;
  int per_sm = 0, sms = 0;
  const size_t b = solve_smem_bytes<T>(p.g.nz, p.g.slip != 0);
  const void* k = p.g.slip ? (const void*)solve_tile_kernel<T, true> : (const void*)solve_tile_kernel<T, false>;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kSolveThreads, b) != cudaSuccess || per_sm < 1) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p.device) != cudaSuccess) return 0;
  const int64_t tiles = ((int64_t)p.g.nkx * p.g.ny + kSolveK - 1) / kSolveK;
  const int64_t most = (int64_t)per_sm * sms;
  return (int)(tiles < most ? tiles : most);
}

size_t solve_tile_table_bytes(const Geometry& g, int precision) {
  const int64_t KP = (int64_t)g.nkx * (g.ny / 2 + 1);
  return precision == DPS_MIXED ? solve_table_bytes<float>(g, KP) : solve_table_bytes<double>(g, KP);
}

dps_status solve_tile_table(Plan& p) {
  const int64_t KP = (int64_t)p.g.nkx * (p.g.ny / 2 + 1);
  const bool mixed = p.precision == DPS_MIXED;
  const size_t bytes = solve_tile_table_bytes(p.g, p.precision);
  void* q = nullptr;
  if (cudaMalloc(&q, bytes) != cudaSuccess) {
    cudaGetLastError();
    return DPS_ERR_OOM;
  }
  p.kt.fac = reinterpret_cast<double*>(q);
  p.kt.KP = KP;
  p.device_bytes += (int64_t)bytes;
  const unsigned blocks = (unsigned)((KP + 127) / 128);
  if (mixed) solve_table_kernel<float><<<blocks, 128>>>(p.g, p.tab.band, solve_table<float>(p));
  else solve_table_kernel<double><<<blocks, 128>>>(p.g, p.tab.band, solve_table<double>(p));
  return cudaGetLastError() == cudaSuccess ? DPS_OK : DPS_ERR_CUDA;
}

template <typename T>
void launch_solve_tile(const Plan& p, int kx0, int w, cudaStream_t s) {
  const Geometry& g = p.g;
  const T* bandT = reinterpret_cast<const T*>(p.kt.bandT);
  cplx<T>* kbuf = reinterpret_cast<cplx<T>*>(p.kt.kbuf);
  cplx<T>* kaux = reinterpret_cast<cplx<T>*>(p.kt.kaux);
  const double tpx = 2.0 * M_PI / g.Lx, tpy = 2.0 * M_PI / g.Ly;
  const size_t b = solve_smem_bytes<T>(g.nz, g.slip != 0);
  if (g.slip)
    solve_tile_kernel<T, true><<<p.bvp_blocks, kSolveThreads, b, s>>>(g, p.tab.band, bandT, solve_table<T>(p), kbuf, kaux,
                                                                     kx0, w, tpx, tpy);
  else
    solve_tile_kernel<T, false><<<p.bvp_blocks, kSolveThreads, b, s>>>(g, p.tab.band, bandT, solve_table<T>(p), kbuf, kaux,
                                                                      kx0, w, tpx, tpy);
}

template int solve_tile_prepare<float>(const Plan&);
template int solve_tile_prepare<double>(const Plan&);
template void launch_solve_tile<float>(const Plan&, int, int, cudaStream_t);
template void launch_solve_tile<double>(const Plan&, int, int, cudaStream_t);

}  // namespace dps
