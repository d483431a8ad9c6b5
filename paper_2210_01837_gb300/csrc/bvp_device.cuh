// Device helpers shared by the per-wavenumber kernels (bvp.cu, solve.cu, cheb_fold.cu, cheb_columns.cu):
// conversions on the integer pipe, streaming accesses, the wavenumber of a spectrum column and the
// wall-correction amplitudes.
#pragma once

#include "dps_internal.cuh"

namespace dps {
namespace {

// ---------------------------------------------------------------------------------------------
// conversions on the integer pipe
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ double f2d(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned e = (b >> 23) & 0xffu;
  if (e == 0u) return 0.0;  // zero (float subnormals flush to zero)
  const unsigned m = b & 0x7fffffu;
  const unsigned hi = (b & 0x80000000u) | ((e + 896u) << 20) | (m >> 3);
  return __hiloint2double((int)hi, (int)(m << 29));
}

__device__ __forceinline__ float d2f(double d) { return narrow_bits(d); }

// 1/d for the pivots of the factorisation (|d| well inside the float range) by Newton-Raphson from a
// float seed: x0 = approximate float reciprocal of the narrowed d (relative error about 2^-22),
// then x <- x + x (1 - d x) twice in double, which squares the error each time (2^-44, then the
// double rounding level).  Four FP64 instructions instead of an IEEE double division; the result
// may differ from the correctly rounded quotient in the last bit.
__device__ __forceinline__ double recip_nr(double d) {
  double x = widen_bits(__fdividef(1.0f, narrow_bits(d)));
  x = fma(x, fma(-d, x, 1.0), x);
  x = fma(x, fma(-d, x, 1.0), x);
  return x;
}

template <typename T> __device__ __forceinline__ double widen(T v);
template <> __device__ __forceinline__ double widen<float>(float v) { return f2d(v); }
template <> __device__ __forceinline__ double widen<double>(double v) { return v; }
template <typename T> __device__ __forceinline__ T narrow(double v);
template <> __device__ __forceinline__ float narrow<float>(double v) { return d2f(v); }
template <> __device__ __forceinline__ double narrow<double>(double v) { return v; }

// loads and stores of data touched once (evict-first in L1 and L2)
__device__ __forceinline__ cplx<float> ld_stream(const cplx<float>* p) {
  const float2 v = __ldcs(reinterpret_cast<const float2*>(p));
  return mk<float>(v.x, v.y);
}
__device__ __forceinline__ cplx<double> ld_stream(const cplx<double>* p) {
  const double2 v = __ldcs(reinterpret_cast<const double2*>(p));
  return mk<double>(v.x, v.y);
}
__device__ __forceinline__ void st_stream(cplx<float>* p, cplx<float> v) {
  __stcs(reinterpret_cast<float2*>(p), make_float2(v.x, v.y));
}
__device__ __forceinline__ void st_stream(cplx<double>* p, cplx<double> v) {
  __stcs(reinterpret_cast<double2*>(p), make_double2(v.x, v.y));
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

template <typename T> __device__ __forceinline__ cplx<double> wid(cplx<T> a) { return mk<double>(widen<T>(a.x), widen<T>(a.y)); }
template <typename T> __device__ __forceinline__ cplx<T> nar(cplx<double> a) { return mk<T>(narrow<T>(a.x), narrow<T>(a.y)); }

__device__ __forceinline__ cplx<double> cdiv(cplx<double> a, cplx<double> b) {
  const double den = b.x * b.x + b.y * b.y;
  return mk<double>((a.x * b.x + a.y * b.y) / den, (a.y * b.x - a.x * b.y) / den);
}

// thread i of a chunk (columns [kx0, kx0 + w), every ky) -> wavenumber column; kidx = kyi*nkx + kxi
__device__ __forceinline__ int64_t chunk_kidx(const Geometry& g, int64_t i, int kx0, int w) {
  const unsigned ii = (unsigned)i;  // total wavenumbers < 2^31
  const int kyi = (int)(ii / (unsigned)w);
  return (int64_t)kyi * g.nkx + kx0 + (int)(ii - (unsigned)kyi * (unsigned)w);
}

struct KInfo {
  int kxi, kyi;
  bool nyq, zero;
  double kx, ky, kk;
};

// kinfo with the host's 2 pi / Lx and 2 pi / Ly, and 1 / |k| from one reciprocal square root (|k|
// as its product with |k|^2): no division on the FP64 pipe, which bounds the table solve
__device__ __forceinline__ KInfo kinfo_fast(const Geometry& g, int64_t kidx, double tpx, double tpy, double& ik) {
  KInfo r;
  const unsigned ku = (unsigned)kidx;  // wavenumbers < 2^31
  r.kyi = (int)(ku / (unsigned)g.nkx);
  r.kxi = (int)(ku - (unsigned)r.kyi * (unsigned)g.nkx);
  r.nyq = ((g.nx % 2 == 0) && r.kxi == g.nx / 2) || ((g.ny % 2 == 0) && r.kyi == g.ny / 2);
  r.zero = (r.kxi == 0 && r.kyi == 0);
  const int nyv = (r.kyi < (g.ny + 1) / 2) ? r.kyi : r.kyi - g.ny;
  r.kx = tpx * (double)r.kxi;
  r.ky = tpy * (double)nyv;
  const double k2 = r.kx * r.kx + r.ky * r.ky;
  ik = r.zero ? 0.0 : rsqrt(k2);
  r.kk = k2 * ik;
  return r;
}

// Wall-correction amplitudes (FP64 boundary rows) from the DP velocity at the walls (vtop, vbot)
// and, with slip, its z derivatives there: bottom wall Eqs. 41-44, slit Eqs. A4-A10 in closed
// form (reading B3), slip lengths and wall velocities Eqs. A3, A8.  Written to kaux as the
// node-value coefficients (cE + cG zeta) e^{-k zeta} + (tE + tG xi) e^{-k xi} per field.
template <typename T, bool SLIP>
__device__ __forceinline__ void wall_amplitudes(const Geometry& g, double kx, double ky, double kk, double ik,
                                                const cplx<double> (&vtop)[3], const cplx<double> (&vbot)[3],
                                                const cplx<double> (&dtop)[2], const cplx<double> (&dbot)[2],
                                                cplx<T>* __restrict__ kaux, int64_t kidx, int64_t K) {
  auto AUX = [&](int q) -> cplx<T>& { return kaux[(size_t)q * K + kidx]; };
  const double sH = g.sH;
  (void)dtop;
  (void)dbot;
  (void)sH;
  cplx<double> cE[3], cG[3], tE[3], tG[3];
#pragma unroll
  for (int f = 0; f < 3; ++f) { cE[f] = cG[f] = tE[f] = tG[f] = mk<double>(0, 0); }
  if (g.mode != DPS_FREE) {
    const double ex = kx * ik, ey = ky * ik;  // ik = 1 / k
    auto Lp = [&](cplx<double> u, cplx<double> v) { return scl(u, ex) + scl(v, ey); };
    auto Tp = [&](cplx<double> u, cplx<double> v) { return scl(v, ex) - scl(u, ey); };
    // wall data (Eq. A3): minus the DP velocity, and with slip u_DP - l0 du_DP/dz at the bottom,
    // u_DP + lH du_DP/dz at the top for the tangential parts
    cplx<double> eb0 = vbot[0], eb1 = vbot[1], et0 = vtop[0], et1 = vtop[1];
    if (SLIP) {
      eb0 = eb0 - scl(dbot[0], g.slip0 * sH);
      eb1 = eb1 - scl(dbot[1], g.slip0 * sH);
      et0 = et0 + scl(dtop[0], g.slipH * sH);
      et1 = et1 + scl(dtop[1], g.slipH * sH);
    }
    const cplx<double> u0L = scl(Lp(eb0, eb1), -1.0), u0T = scl(Tp(eb0, eb1), -1.0);
    const cplx<double> w0 = scl(vbot[2], -1.0);
    cplx<double> AL = u0L, Az = w0, AT = u0T;
    cplx<double> BL = mk<double>(0, 0), Bz = mk<double>(0, 0), BT = mk<double>(0, 0);
    if (SLIP && g.mode == DPS_BOTTOM_WALL) {
      // bottom family only: Robin rows u - l0 du/dz = u0 with w(0) = w0 give
      // AT (1 + k l0) = u0T and AL (1 + 2 k l0) + i k l0 Az = u0L
      const double kl0 = kk * g.slip0;
      AT = scl(u0T, 1.0 / (1.0 + kl0));
      AL = scl(u0L - scl(mul_i(w0), kl0), 1.0 / (1.0 + 2.0 * kl0));
    }
    if (SLIP && g.mode == DPS_SLIT) {
      const cplx<double> uHL = scl(Lp(et0, et1), -1.0), uHT = scl(Tp(et0, et1), -1.0);
      const cplx<double> wH = scl(vtop[2], -1.0);
      const double kH = kk * g.H, E = exp(-kH), E2 = E * E;
      const double kl0 = kk * g.slip0, klH = kk * g.slipH;
      // transverse: [1 + k l0, E (1 - k l0); E (1 - k lH), 1 + k lH] [AT; BT] = [u0T; uHT]
      {
        const double t11 = 1.0 + kl0, t12 = E * (1.0 - kl0), t21 = E * (1.0 - klH), t22 = 1.0 + klH;
        const double idt = 1.0 / (t11 * t22 - t12 * t21);
        AT = scl(scl(u0T, t22) - scl(uHT, t12), idt);
        BT = scl(scl(uHT, t11) - scl(u0T, t21), idt);
      }
      // longitudinal/normal: S0 A + E N1 B = a0, SH B + E N2 A = b0 with A = (AL, Az), B = (BL, Bz),
      // S0 = [1 + 2 k l0, i k l0; 0, 1], SH = [1 + 2 k lH, -i k lH; 0, 1],
      // N1 = [(1 - k l0)(1 - kH) - k l0, i k (H (1 - k l0) + l0); i kH, 1 + kH],
      // N2 = [(1 - kH)(1 - k lH) - k lH, -i k (H (1 - k lH) + lH); -i kH, 1 + kH];
      // (S0 - E^2 N1 SH^-1 N2) A = a0 - E N1 SH^-1 b0, then B = SH^-1 (b0 - E N2 A)
      const cplx<double> zc = mk<double>(0, 0);
      const double sh = 1.0 / (1.0 + 2.0 * klH);
      const cplx<double> h11 = mk<double>(sh, 0), h12 = mk<double>(0, klH * sh);  // SH^-1 = [h11 h12; 0 1]
      const cplx<double> n11 = mk<double>((1.0 - kl0) * (1.0 - kH) - kl0, 0), n12 = mk<double>(0, kk * (g.H * (1.0 - kl0) + g.slip0));
      const cplx<double> n21 = mk<double>(0, kH), n22 = mk<double>(1.0 + kH, 0);
      const cplx<double> m11 = mk<double>((1.0 - kH) * (1.0 - klH) - klH, 0), m12 = mk<double>(0, -kk * (g.H * (1.0 - klH) + g.slipH));
      const cplx<double> m21 = mk<double>(0, -kH), m22 = mk<double>(1.0 + kH, 0);
      // P = SH^-1 N2, Q = N1 P
      const cplx<double> p11 = h11 * m11 + h12 * m21, p12 = h11 * m12 + h12 * m22, p21 = m21, p22 = m22;
      const cplx<double> q11 = n11 * p11 + n12 * p21, q12 = n11 * p12 + n12 * p22;
      const cplx<double> q21 = n21 * p11 + n22 * p21, q22 = n21 * p12 + n22 * p22;
      const cplx<double> x11 = mk<double>(1.0 + 2.0 * kl0, 0) - scl(q11, E2), x12 = mk<double>(0, kl0) - scl(q12, E2);
      const cplx<double> x21 = zc - scl(q21, E2), x22 = mk<double>(1.0, 0) - scl(q22, E2);
      const cplx<double> hb0 = h11 * uHL + h12 * wH, hb1 = wH;  // SH^-1 b0
      const cplx<double> r0 = u0L - scl(n11 * hb0 + n12 * hb1, E);
      const cplx<double> r1 = w0 - scl(n21 * hb0 + n22 * hb1, E);
      const cplx<double> det = x11 * x22 - x12 * x21;
      AL = cdiv(x22 * r0 - x12 * r1, det);
      Az = cdiv(x11 * r1 - x21 * r0, det);
      const cplx<double> e0 = uHL - scl(m11 * AL + m12 * Az, E), e1 = wH - scl(m21 * AL + m22 * Az, E);
      BL = h11 * e0 + h12 * e1;
      Bz = e1;
    }
    if (!SLIP && g.mode == DPS_SLIT) {
      const cplx<double> uHL = scl(Lp(vtop[0], vtop[1]), -1.0), uHT = scl(Tp(vtop[0], vtop[1]), -1.0);
      const cplx<double> wH = scl(vtop[2], -1.0);
      const double kH = kk * g.H;
      const double E = exp(-kH);
      const double E2 = E * E;
      // transverse: [1 E; E 1] [AT; BT] = [u0T; uHT]
      AT = scl(u0T - scl(uHT, E), 1.0 / (1.0 - E2));
      BT = scl(uHT - scl(u0T, E), 1.0 / (1.0 - E2));
      // longitudinal/normal: A = a0 - E M1 B, B = b0 - E M2 A  =>  (I - E^2 M1 M2) A = a0 - E M1 b0,
      // M1 = [[1-kH, i kH], [i kH, 1+kH]], M2 = [[1-kH, -i kH], [-i kH, 1+kH]]
      const double k2H2 = kH * kH;
      const cplx<double> m11 = mk<double>(1.0 - E2 * (1.0 - 2.0 * kH + 2.0 * k2H2), 0.0);
      const cplx<double> m12 = mk<double>(0.0, -E2 * 2.0 * k2H2);
      const cplx<double> m21 = mk<double>(0.0, E2 * 2.0 * k2H2);
      const cplx<double> m22 = mk<double>(1.0 - E2 * (1.0 + 2.0 * kH + 2.0 * k2H2), 0.0);
      const cplx<double> M1b_L = scl(uHL, 1.0 - kH) + scl(mul_i(wH), kH);
      const cplx<double> M1b_z = scl(mul_i(uHL), kH) + scl(wH, 1.0 + kH);
      const cplx<double> rL = u0L - scl(M1b_L, E);
      const cplx<double> rz = w0 - scl(M1b_z, E);
      const cplx<double> det = m11 * m22 - m12 * m21;
      AL = cdiv(m22 * rL - m12 * rz, det);
      Az = cdiv(m11 * rz - m21 * rL, det);
      const cplx<double> M2a_L = scl(AL, 1.0 - kH) - scl(mul_i(Az), kH);
      const cplx<double> M2a_z = scl(mul_i(AL), -kH) + scl(Az, 1.0 + kH);
      BL = uHL - scl(M2a_L, E);
      Bz = wH - scl(M2a_z, E);
    }
    // pressure amplitudes over 2 eta: bottom k (Az - i AL), top -k (Bz + i BL)
    const cplx<double> pib = scl(Az - mul_i(AL), kk);
    const cplx<double> pit = scl(Bz + mul_i(BL), -kk);
    // u_L = (AL - i pib zeta) e^{-k zeta} + (BL - i pit xi) e^{-k xi};  u_T = AT e^{-k zeta} + BT e^{-k xi}
    // w   = (Az + pib zeta) e^{-k zeta} + (Bz - pit xi) e^{-k xi}
    const cplx<double> gbL = scl(mul_i(pib), -1.0), gtL = scl(mul_i(pit), -1.0);
    cE[0] = scl(AL, ex) - scl(AT, ey);  cG[0] = scl(gbL, ex);
    tE[0] = scl(BL, ex) - scl(BT, ey);  tG[0] = scl(gtL, ex);
    cE[1] = scl(AL, ey) + scl(AT, ex);  cG[1] = scl(gbL, ey);
    tE[1] = scl(BL, ey) + scl(BT, ex);  tG[1] = scl(gtL, ey);
    cE[2] = Az;                          cG[2] = pib;
    tE[2] = Bz;                          tG[2] = scl(pit, -1.0);
  }
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    AUX(4 * f + 0) = nar<T>(cE[f]);
    AUX(4 * f + 1) = nar<T>(cG[f]);
    AUX(4 * f + 2) = nar<T>(tE[f]);
    AUX(4 * f + 3) = nar<T>(tG[f]);
  }
}

// r rho in the transform precision (the right-hand side's own precision), widened exactly
template <typename T> __device__ __forceinline__ double prescale_one(T r, double rho);
template <> __device__ __forceinline__ double prescale_one<float>(float r, double rho) { return f2d(r * narrow_bits(rho)); }
template <> __device__ __forceinline__ double prescale_one<double>(double r, double rho) { return r * rho; }

}  // namespace
}  // namespace dps
