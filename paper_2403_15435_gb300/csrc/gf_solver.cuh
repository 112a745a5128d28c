// Device-side building blocks of the wave-propagation step: the augmented
// Riemann solver (Sec. 3.3), the MC limiter (Sec. 3.2) and the transverse
// eigen-split of the 2D extension (Sec. 3.2, leveque2002).  First the forms
// of the dimensionally split step, templates on the real type; then the
// unsplit step's own, in FP64 and in FP32.  The FP64 translation units are
// compiled with -fmad=false so that every operation rounds as written.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "gf_fp64.cuh"

namespace gfk {

template <typename R>
struct Side {
  R h, n, t, b;  // depth, normal momentum, transverse momentum, bed
  R w;           // surface-deviation form only: stored surface h + b - eta0
  bool wet;      // surface-deviation form only: exact wet test of the cell
};

// Quotient a / b.  FP64: the correctly rounded division (div_rn), so that the
// FP64 path rounds as written.  FP32: the approximate reciprocal times a (within
// 2 ulp for |b| below 2^126, far above any depth, momentum or speed here);
// the product is rounded on its own (never fused into a neighbouring
// addition), so that every kernel variant that inlines this code rounds it
// alike.  Zero numerators still give exact zeros, so a lake at rest keeps
// exactly zero waves.
template <typename R>
__device__ __forceinline__ R qdiv(R a, R b) { return div_rn(a, b); }
template <>
__device__ __forceinline__ float qdiv<float>(float a, float b) {
  return __fmul_rn(a, __fdividef(1.0f, b));
}

// Square root, correctly rounded in FP64.
__device__ __forceinline__ float qsqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double qsqrt(double x) { return sqrt_rn(x); }

// Product rounded on its own (FP32: never fused into a neighbouring addition).
template <typename R>
__device__ __forceinline__ R rmul(R a, R b) { return a * b; }
template <>
__device__ __forceinline__ float rmul<float>(float a, float b) { return __fmul_rn(a, b); }

template <typename R>
__device__ __forceinline__ R rmin(R a, R b) { return a < b ? a : b; }
template <typename R>
__device__ __forceinline__ R rmax(R a, R b) { return a > b ? a : b; }

// Augmented Riemann solve (Sec. 3.3).  Returns three f-waves Z[p*3 + k]
// (component k: mass, normal momentum, transverse momentum) and speeds s[p].
// Bed jump: a stationary wave whose momentum-flux part -g*hbar*db is the
// bathymetry source and whose depth jump is -db, bounded so no depth in the
// fan is negative.  Acoustic speeds: Einfeldt (HLLE) with Roe averages, or
// the dam-break front speeds at a wet/dry edge.  A dry cell whose bed is
// above the wet surface is tested with the mirrored (reflecting) problem.
//
// DEV = false: plain form, the state is (h, n, t) and the bed b; the wet test
// is h > drytol and the surface jump is formed from depths and beds.
// DEV = true: surface-deviation form, each side also carries its stored
// surface w = h + b - eta0 (b is then the bed minus eta0) and a wet flag
// decided exactly from the stored values; the surface jump is the difference
// of the stored surfaces, so a lake at rest gives exactly zero waves.
template <typename R, bool DEV = false>
__device__ __forceinline__ void riemann(Side<R> l, Side<R> r, R g, R drytol,
                                        R (&Z)[9], R (&s)[3]) {
#pragma unroll
  for (int k = 0; k < 9; ++k) Z[k] = R(0);
  s[0] = s[1] = s[2] = R(0);
  const bool wetl = DEV ? l.wet : (l.h > drytol);
  const bool wetr = DEV ? r.wet : (r.h > drytol);
  if (!wetl && !wetr) return;
  // surface depths: a dry cell keeps its stored depth in its surface so a
  // still shoreline stays at rest; fluxes and speeds see zero depth
  R el = l.h, er = r.h;
  if (!wetl) { l.h = R(0); l.n = R(0); l.t = R(0); }
  if (!wetr) { r.h = R(0); r.n = R(0); r.t = R(0); }

  int wall = 0;  // +1: right side is a wall, -1: left side is a wall
  if (!wetr && (DEV ? r.b > l.w : r.b > l.h + l.b)) {
    const R u = qdiv(l.n, l.h);
    const R c = qsqrt(g * l.h);
    const R sw = rmax(c - u, c);       // fastest wave of the mirrored problem
    const R hm = l.h + qdiv(l.n, sw);  // its HLL middle depth
    if (r.b >= l.b + hm) {
      wall = 1;
      r.h = l.h; r.n = -l.n; r.t = l.t; r.b = l.b; er = l.h; r.w = l.w;
    } else if (DEV) {
      r.w = l.w + er;                  // overtopped: step lowered to surface
      r.b = l.w;
    } else {
      r.b = l.h + l.b;
    }
  } else if (!wetl && (DEV ? l.b > r.w : l.b > r.h + r.b)) {
    const R u = qdiv(r.n, r.h);
    const R c = qsqrt(g * r.h);
    const R sw = rmax(u + c, c);
    const R hm = r.h - qdiv(r.n, sw);
    if (l.b >= r.b + hm) {
      wall = -1;
      l.h = r.h; l.n = -r.n; l.t = r.t; l.b = r.b; el = r.h; l.w = r.w;
    } else if (DEV) {
      l.w = r.w + el;
      l.b = r.w;
    } else {
      l.b = r.h + r.b;
    }
  }

  const R ul = l.h > R(0) ? qdiv(l.n, l.h) : R(0);
  const R ur = r.h > R(0) ? qdiv(r.n, r.h) : R(0);
  const R vl = l.h > R(0) ? qdiv(l.t, l.h) : R(0);
  const R vr = r.h > R(0) ? qdiv(r.t, r.h) : R(0);
  // FP32: the celerities from the square roots of the depths, which the
  // Roe average needs anyway (two square roots fewer per edge), each product
  // rounded on its own (not fused, so every inlining rounds it alike); FP64:
  // as written, sqrt(g h)
  constexpr bool F32 = std::is_same<R, float>::value;
  const R ql = F32 ? qsqrt(l.h) : R(0), qr = F32 ? qsqrt(r.h) : R(0);
  const R cl = F32 ? rmul(qsqrt(g), ql) : qsqrt(g * l.h);
  const R cr = F32 ? rmul(qsqrt(g), qr) : qsqrt(g * r.h);
  R s1, s3;
  if (l.h > R(0) && r.h > R(0)) {
    const R qlw = F32 ? ql : qsqrt(l.h), qrw = F32 ? qr : qsqrt(r.h);
    const R uhat = qdiv(qlw * ul + qrw * ur, qlw + qrw);
    const R chat = qsqrt(g * (R(0.5) * (l.h + r.h)));
    s1 = rmin(ul - cl, uhat - chat);
    s3 = rmax(ur + cr, uhat + chat);
  } else if (r.h == R(0)) {
    s1 = ul - cl;
    s3 = ul + R(2) * cl;
  } else {
    s1 = ur - R(2) * cr;
    s3 = ur + cr;
  }
  const R s2 = R(0.5) * (s1 + s3);

  const R hbar = R(0.5) * (l.h + r.h);
  const R db = r.b - l.b;
  const R deta = DEV ? r.w - l.w : (er + r.b) - (el + l.b);
  const R den = s3 - s1;
  const R dn = r.n - l.n;
  const R hhll = qdiv(s3 * r.h - s1 * l.h - dn, den);

  // depth jump of the stationary wave, bounded for non-negative depths
  R dhs = -db;
  bool clamped = false;
  if (s1 < R(0) && s3 > R(0)) {
    const R lo = qdiv(hhll * den, s1);
    const R hi = qdiv(hhll * den, s3);
    if (dhs < lo) { dhs = lo; clamped = true; }
    if (dhs > hi) { dhs = hi; clamped = true; }
  } else if (s1 >= R(0)) {
    const R hi = s1 > R(0) ? qdiv(hhll * den, s1) : dhs;
    if (dhs > hi) { dhs = hi; clamped = true; }
    if (dhs < -l.h) { dhs = -l.h; clamped = true; }
  } else {
    const R lo = s3 < R(0) ? qdiv(hhll * den, s3) : dhs;
    if (dhs < lo) { dhs = lo; clamped = true; }
    if (dhs > r.h) { dhs = r.h; clamped = true; }
  }
  const R d1 = clamped ? (r.h - l.h) - dhs : deta;
  const R d3 = (r.n * ur - l.n * ul) + g * hbar * deta;

  const R b1 = qdiv(s3 * d1 - dn, den);
  const R b3 = qdiv(dn - s1 * d1, den);
  const R b2 = d3 - (s1 * s1 * b1 + s3 * s3 * b3);

  Z[0] = s1 * b1;
  Z[1] = s1 * s1 * b1;
  Z[2] = vl * Z[0];
  Z[6] = s3 * b3;
  Z[7] = s3 * s3 * b3;
  Z[8] = vr * Z[6];
  Z[3] = R(0);
  Z[4] = b2;
  Z[5] = (r.n * vr - l.n * vl) - (Z[2] + Z[8]);
  s[0] = s1;
  s[1] = s2;
  s[2] = s3;
  if (wall == 1) {
#pragma unroll
    for (int k = 3; k < 9; ++k) Z[k] = R(0);
  } else if (wall == -1) {
#pragma unroll
    for (int k = 0; k < 6; ++k) Z[k] = R(0);
  }
}

// MC limiter.
template <typename R>
__device__ __forceinline__ R mc(R th) {
  const R a = R(0.5) * (R(1) + th);
  R m = a < R(2) ? a : R(2);
  const R b = R(2) * th;
  m = m < b ? m : b;
  return m > R(0) ? m : R(0);
}

template <typename R>
__device__ __forceinline__ R dot3(const R* a, const R* b) {
  return (a[0] * b[0] + a[1] * b[1]) + a[2] * b[2];
}

// Fluctuations A-dQ, A+dQ and the limited correction flux of one edge from
// its waves (Z, S) and the waves of its two neighbouring edges (Zm at the
// edge before, Zp at the edge after).  Component c of a wave array is at
// [c * ST] (ST = 1: packed; larger: one plane per component).  nodry = false
// switches the correction off (an edge touching a dry cell).
// Z3Z = true: the middle wave's mass component (Z[3], zero by construction
// of the solver) is neither read nor added, and A+dQ is formed as the wave
// minus its A-dQ part; both give the same values up to the sign of zeros.
template <typename R, int ST = 1, bool Z3Z = false>
__device__ __forceinline__ void edge_fluxes(const R* Z, const R* S,
                                            const R* Zm, const R* Zp, R nu,
                                            bool nodry, R (&am)[3],
                                            R (&ap)[3], R (&ff)[3]) {
  R cm[3][3], cp[3][3], cf[3][3];
  R z[9];
#pragma unroll
  for (int c = 0; c < 9; ++c) z[c] = (Z3Z && c == 3) ? R(0) : Z[c * ST];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const R sp = S[p * ST];
    const R wm = sp < R(0) ? R(1) : (sp == R(0) ? R(0.5) : R(0));
    const R wp = sp > R(0) ? R(1) : (sp == R(0) ? R(0.5) : R(0));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      cm[p][k] = z[3 * p + k] * wm;
      cp[p][k] = Z3Z ? z[3 * p + k] - cm[p][k] : z[3 * p + k] * wp;
      cf[p][k] = R(0);
    }
    if (sp != R(0) && nodry) {
      const bool m0 = Z3Z && p == 1;  // mass component known zero
      const R zz = m0 ? z[4] * z[4] + z[5] * z[5] : dot3(z + 3 * p, z + 3 * p);
      if (zz != R(0)) {
        const R* up = sp > R(0) ? Zm : Zp;
        const R u3[3] = {m0 ? R(0) : up[(3 * p) * ST], up[(3 * p + 1) * ST],
                         up[(3 * p + 2) * ST]};
        const R num = m0 ? u3[1] * z[4] + u3[2] * z[5] : dot3(u3, z + 3 * p);
        const R th = qdiv(num, zz);
        const R phi = mc(th);
        const R sg = sp > R(0) ? R(1) : R(-1);
        const R as = sp > R(0) ? sp : -sp;
        const R coef = R(0.5) * sg * (R(1) - nu * as) * phi;
#pragma unroll
        for (int k = 0; k < 3; ++k) cf[p][k] = coef * z[3 * p + k];
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (Z3Z && k == 0) {
      am[0] = cm[0][0] + cm[2][0];
      ap[0] = cp[0][0] + cp[2][0];
      ff[0] = cf[0][0] + cf[2][0];
    } else {
      am[k] = (cm[0][k] + cm[2][k]) + cm[1][k];
      ap[k] = (cp[0][k] + cp[2][k]) + cp[1][k];
      ff[k] = (cf[0][k] + cf[2][k]) + cf[1][k];
    }
  }
}

// ------------------------------------------------------------------------
// The FP64 step's own forms.  The FP64 pipe bounds that kernel, so whatever
// belongs to a cell (velocities, celerity, square root of the depth, surface)
// is computed once per cell instead of once per edge side, and everything but
// additions and products (comparisons, selections, scalings by two, quotients,
// roots) runs in the integer and FP32 pipes.  The operations and their order
// are those of riemann / edge_fluxes above, so the values agree bit for bit up
// to the sign of zeros.

// One side of an edge.  A dry cell has zero u, v, c and q; h, n, t, b and eta
// are its stored values.
struct Prim {
  double h, n, t, b, eta;  // depth, normal and transverse momentum, bed, h + b
  double u, v, c, q;       // n / h, t / h, sqrt(g h), sqrt(h)
  bool wet;
};

// Waves z[8]: (mass, normal, transverse) of the first and third wave and
// (normal, transverse) of the middle one, whose mass part is zero:
// z[0..2], z[3..4], z[5..7]; speeds s[3].
__device__ __forceinline__ void riemann_prim(Prim l, Prim r, double g, double (&z)[8],
                                             double (&s)[3]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) z[k] = 0.0;
  s[0] = s[1] = s[2] = 0.0;
  if (!l.wet && !r.wet) return;
  int wall = 0;
  bool pl = l.wet, pr = r.wet;  // sides with a positive depth
  if (!(l.wet && r.wet)) {
    // a wet/dry edge: see riemann
    const double el = l.h, er = r.h;
    if (!l.wet) l.h = l.n = l.t = 0.0;
    if (!r.wet) r.h = r.n = r.t = 0.0;
    if (!r.wet && dlt(l.eta, r.b)) {
      const double sw = dmax(l.c - l.u, l.c);
      const double hm = l.h + div_rn(l.n, sw);
      if (!dlt(r.b, l.b + hm)) {
        wall = 1;
        r = l;
        r.n = dneg(l.n);
        r.u = dneg(l.u);
        pr = true;
      } else {
        r.b = l.eta;
        r.eta = er + r.b;
      }
    } else if (!l.wet && dlt(r.eta, l.b)) {
      const double sw = dmax(r.u + r.c, r.c);
      const double hm = r.h - div_rn(r.n, sw);
      if (!dlt(l.b, r.b + hm)) {
        wall = -1;
        l = r;
        l.n = dneg(r.n);
        l.u = dneg(r.u);
        pl = true;
      } else {
        l.b = r.eta;
        l.eta = el + l.b;
      }
    }
  }
  const double hbar = half(l.h + r.h);
  const double ghb = g * hbar;
  double s1, s3;
  if (pl && pr) {
    const double uhat = div_rn(l.q * l.u + r.q * r.u, l.q + r.q);
    const double chat = sqrt_rn(ghb);
    s1 = dmin(l.u - l.c, uhat - chat);
    s3 = dmax(r.u + r.c, uhat + chat);
  } else if (pl) {
    rare();
    s1 = l.u - l.c;
    s3 = l.u + twice(l.c);
  } else {
    rare();
    s1 = r.u - twice(r.c);
    s3 = r.u + r.c;
  }
  const double s2 = half(s1 + s3);
  const double dhs0 = l.b - r.b;  // -(r.b - l.b)
  const double deta = r.eta - l.eta;
  const double den = s3 - s1;
  const double dn = r.n - l.n;
  const double hhll = div_rn(s3 * r.h - s1 * l.h - dn, den);
  // depth jump of the stationary wave, bounded for non-negative depths
  double dhs = dhs0;
  bool clamped = false;
  const double x = hhll * den;
  if (neg(s1) && pos(s3)) {
    // the bounds x / s1 < -db < x / s3, tested first in FP32 with a margin
    // far above its rounding; the exact test only where that cannot tell
    const float xf = trunc_f32(x), df = trunc_f32(dhs0);
    const bool inside = xf > 1e-25f && df * trunc_f32(s1) < 0.9999f * xf &&
                        df * trunc_f32(s3) < 0.9999f * xf;
    if (!inside) {
      rare();
      const double lo = div_rn(x, s1), hi = div_rn(x, s3);
      if (dlt(dhs, lo)) { dhs = lo; clamped = true; }
      if (dlt(hi, dhs)) { dhs = hi; clamped = true; }
    }
  } else if (!neg(s1)) {
    const double hi = pos(s1) ? div_rn(x, s1) : dhs;
    if (dlt(hi, dhs)) { dhs = hi; clamped = true; }
    if (dlt(dhs, dneg(l.h))) { dhs = dneg(l.h); clamped = true; }
  } else {
    const double lo = neg(s3) ? div_rn(x, s3) : dhs;
    if (dlt(dhs, lo)) { dhs = lo; clamped = true; }
    if (dlt(r.h, dhs)) { dhs = r.h; clamped = true; }
  }
  double d1 = deta;
  if (clamped) {
    rare();
    d1 = (r.h - l.h) - dhs;
  }
  const double d3 = (r.n * r.u - l.n * l.u) + ghb * deta;
  const double b1 = div_rn(s3 * d1 - dn, den);
  const double b3 = div_rn(dn - s1 * d1, den);
  const double z1 = s1 * s1 * b1, z3 = s3 * s3 * b3;
  z[0] = s1 * b1;
  z[1] = z1;
  z[2] = l.v * z[0];
  z[5] = s3 * b3;
  z[6] = z3;
  z[7] = r.v * z[5];
  z[3] = d3 - (z1 + z3);
  z[4] = (r.n * r.v - l.n * l.v) - (z[2] + z[7]);
  s[0] = s1;
  s[1] = s2;
  s[2] = s3;
  if (wall == 1) {
#pragma unroll
    for (int k = 3; k < 8; ++k) z[k] = 0.0;
  } else if (wall == -1) {
#pragma unroll
    for (int k = 0; k < 5; ++k) z[k] = 0.0;
  }
}

// MC limiter of a ratio num / zz with num > 0, times one half
__device__ __forceinline__ double half_mc(double num, double zz) {
  const double th = div_rn(num, zz);
  const double m = dmin(dmin(half(1.0 + th), 2.0), twice(th));
  return half(m);
}

// Fluctuations and limited correction flux of one edge from the wave planes
// (component k at [k * ST]; planes 8..10 the speeds; Zm, Zp the edges before
// and after).  See edge_fluxes.
template <int ST>
__device__ __forceinline__ void edge_fluxes_prim(const double* Z, const double* Zm,
                                                 const double* Zp, double nu, bool nodry,
                                                 double (&am)[3], double (&ap)[3],
                                                 double (&ff)[3]) {
  double z[8], s[3];
#pragma unroll
  for (int c = 0; c < 8; ++c) z[c] = Z[c * ST];
#pragma unroll
  for (int p = 0; p < 3; ++p) s[p] = Z[(8 + p) * ST];
  const bool n2 = neg(s[1]);
  if (neg(s[0]) && pos(s[2]) && !iszero(s[1])) {
    // first wave leftwards, third rightwards, the middle one to one side
    const double x1 = (n2 ? z[1] : z[6]) + z[3];
    const double x2 = (n2 ? z[2] : z[7]) + z[4];
    am[0] = z[0];
    am[1] = n2 ? x1 : z[1];
    am[2] = n2 ? x2 : z[2];
    ap[0] = z[5];
    ap[1] = n2 ? z[6] : x1;
    ap[2] = n2 ? z[7] : x2;
  } else {
    rare();
    const double wm[3] = {neg(s[0]) ? 1.0 : (iszero(s[0]) ? 0.5 : 0.0),
                          n2 ? 1.0 : (iszero(s[1]) ? 0.5 : 0.0),
                          neg(s[2]) ? 1.0 : (iszero(s[2]) ? 0.5 : 0.0)};
    const double wp[3] = {pos(s[0]) ? 1.0 : (iszero(s[0]) ? 0.5 : 0.0),
                          pos(s[1]) ? 1.0 : (iszero(s[1]) ? 0.5 : 0.0),
                          pos(s[2]) ? 1.0 : (iszero(s[2]) ? 0.5 : 0.0)};
    am[0] = z[0] * wm[0] + z[5] * wm[2];
    ap[0] = z[0] * wp[0] + z[5] * wp[2];
#pragma unroll
    for (int k = 1; k < 3; ++k) {
      am[k] = (z[k] * wm[0] + z[5 + k] * wm[2]) + z[2 + k] * wm[1];
      ap[k] = (z[k] * wp[0] + z[5 + k] * wp[2]) + z[2 + k] * wp[1];
    }
  }
  double f1[3] = {0.0, 0.0, 0.0}, f2[3] = {0.0, 0.0, 0.0}, f3[3] = {0.0, 0.0, 0.0};
  if (nodry) {
    auto wave = [&](double sp, const double* up, double za, double zb, double zc, bool mass,
                    int o, double (&f)[3]) {
      if (iszero(sp)) return;
      const double ub = up[(o + 1) * ST], uc = up[(o + 2) * ST];
      double num, zz;
      if (mass) {
        num = (up[o * ST] * za + ub * zb) + uc * zc;
        zz = (za * za + zb * zb) + zc * zc;
      } else {
        num = ub * zb + uc * zc;
        zz = zb * zb + zc * zc;
      }
      if (!pos(num) || iszero(zz)) return;  // limiter zero
      const double c = (1.0 - nu * dabs(sp)) * half_mc(num, zz);
      const double cs = neg(sp) ? dneg(c) : c;
      if (mass) f[0] = cs * za;
      f[1] = cs * zb;
      f[2] = cs * zc;
    };
    wave(s[0], pos(s[0]) ? Zm : Zp, z[0], z[1], z[2], true, 0, f1);
    wave(s[1], pos(s[1]) ? Zm : Zp, 0.0, z[3], z[4], false, 2, f2);
    wave(s[2], pos(s[2]) ? Zm : Zp, z[5], z[6], z[7], true, 5, f3);
  }
  ff[0] = f1[0] + f3[0];
  ff[1] = (f1[1] + f3[1]) + f2[1];
  ff[2] = (f1[2] + f3[2]) + f2[2];
}

// Transverse split of an increment d = (mass, momentum along the split
// direction, other momentum) in a cell with velocities w along the split
// direction and z across it and celerity c (zero when dry): eigenvectors of
// the split direction's Jacobian with speeds w - c, w, w + c.  plus/minus are
// returned in the same frame.  A part entering a dry neighbour whose bed is
// above the cell's surface is dropped; a dry cell splits nothing.  wet, wetm,
// wetp: the cell and its neighbours at -1 and +1; eta the cell's surface, bm,
// bp the neighbours' beds.
__device__ __forceinline__ void tsplit_prim(double w, double z, double c, double eta, bool wet,
                                            bool wetm, double bm, bool wetp, double bp,
                                            const double (&d)[3], double (&plus)[3],
                                            double (&minus)[3]) {
  plus[0] = plus[1] = plus[2] = 0.0;
  minus[0] = minus[1] = minus[2] = 0.0;
  if (!wet) return;
  const double l1 = w - c, l3 = w + c;
  const double c2 = twice(c);
  const double a1 = div_rn(l3 * d[0] - d[1], c2);
  const double a3 = div_rn(d[1] - l1 * d[0], c2);
  const double a2 = d[2] - z * d[0];
  const double w1 = l1 * a1, w3 = l3 * a3, w2 = w * a2;
  const double W1[3] = {w1, w1 * l1, w1 * z}, W3[3] = {w3, w3 * l3, w3 * z};
  const bool openp = wetp || !dlt(eta, bp), openm = wetm || !dlt(eta, bm);
  double p[3], q[3];
  if (neg(l1) && pos(l3)) {
    const double x = (neg(w) ? W1[2] : W3[2]) + w2;
    p[0] = W3[0]; p[1] = W3[1]; p[2] = pos(w) ? x : W3[2];
    q[0] = W1[0]; q[1] = W1[1]; q[2] = neg(w) ? x : W1[2];
  } else {
    rare();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      p[k] = (pos(l1) ? W1[k] : 0.0) + (pos(l3) ? W3[k] : 0.0);
      q[k] = (neg(l1) ? W1[k] : 0.0) + (neg(l3) ? W3[k] : 0.0);
    }
    if (pos(w)) p[2] += w2;
    if (neg(w)) q[2] += w2;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (openp) plus[k] = p[k];
    if (openm) minus[k] = q[k];
  }
}

// Exact wet test of a stored surface-deviation cell: depth = w - b (both
// FP32) compared with drytol as the FP64 value (w - b is exact in double).
// FP32 decides when the rounded difference is clear of drytol by more than
// its rounding bound; otherwise the test is redone in FP64.
// The FP64 tie-break is a separate, non-inlined function so that the
// compiler cannot evaluate it speculatively on every call (FP64 is slow on
// this part).
static __device__ __noinline__ bool wet_dev_tie(float w, float b, double drytol) {
  return ((double)w - (double)b) > drytol;
}

__device__ __forceinline__ bool wet_dev(float w, float b, double drytol,
                                        float dtf, float margin) {
  const float h = w - b;
  if (h > dtf + margin) return true;
  if (h < dtf - margin) return false;
  return wet_dev_tie(w, b, drytol);
}

// ------------------------------------------------------------------------
// The FP32 step's own forms.  That kernel is bound by issue slots, so the
// per-cell quantities come from shared memory (see the FP64 forms).  The unit
// is compiled without contraction and every fused operation is written out,
// so all kernel shapes round alike; the operations and the places where they
// fuse are those the compiler chooses for riemann / edge_fluxes.

__device__ __forceinline__ float rcpf(float x) { return seed_rcp(x); }

// ---------------------------------------------------------------- pairs
//
// Two neighbouring edges (or cells) per thread: the additions, products and
// fused products of both in one packed instruction (f32x2), which halves the
// issue slots of the arithmetic, the index work and the shared-memory
// instructions.  Each half rounds as the scalar instruction does.

typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void upk(f2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 pk1(float a) { return pk(a, a); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// A product that is rounded on its own although it feeds an addition: the
// assembler fuses mul2 and add2 (whatever their rounding modifiers), so it is
// written as a fused product with an addend nz of negative zero that the
// compiler does not know (GfGeom::negzero).
__device__ __forceinline__ f2 mulr2(f2 a, f2 b, f2 nz) { return fma2(a, b, nz); }
__device__ __forceinline__ f2 neg2(f2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f2 sub2(f2 a, f2 b) { return add2(a, neg2(b)); }
__device__ __forceinline__ f2 rcp2(f2 a) {
  float x, y;
  upk(a, x, y);
  return pk(seed_rcp(x), seed_rcp(y));
}
__device__ __forceinline__ f2 sqrt2(f2 a) {
  float x, y;
  upk(a, x, y);
  return pk(sqrtf(x), sqrtf(y));
}
__device__ __forceinline__ f2 min2(f2 a, f2 b) {
  float x, y, u, v;
  upk(a, x, y);
  upk(b, u, v);
  return pk(fminf(x, u), fminf(y, v));
}
__device__ __forceinline__ f2 max2(f2 a, f2 b) {
  float x, y, u, v;
  upk(a, x, y);
  upk(b, u, v);
  return pk(fmaxf(x, u), fmaxf(y, v));
}
// per half: c ? a : b
__device__ __forceinline__ f2 sel2(bool c0, bool c1, f2 a, f2 b) {
  float x, y, u, v;
  upk(a, x, y);
  upk(b, u, v);
  return pk(c0 ? x : u, c1 ? y : v);
}
__device__ __forceinline__ f2 ld2(const float* p) { return *reinterpret_cast<const f2*>(p); }
__device__ __forceinline__ void st2(float* p, f2 v) { *reinterpret_cast<f2*>(p) = v; }

// One side of two edges in the deviation form: stored surface and bed (minus
// eta0), normal momentum, velocities and the root of the depth (u, v and q
// are zero in a dry cell).
struct Prim32x2 {
  f2 w, b, n, u, v, q;
};

// The depth jump dh of a stationary wave, bounded for non-negative depths
// (x1, x3: what the outer waves leave over s1 and s3).
__device__ __forceinline__ float jump_bound(float dh, float s1, float s3, float x1, float x3,
                                             float hl, float hr, bool& clamped) {
  // right-going flow: the upper bound first
  const bool right = s1 >= 0.0f, sub = s1 < 0.0f && s3 > 0.0f;
  const float lo = sub ? x1 : (right ? -hl : (s3 < 0.0f ? x3 : dh));
  const float hi = sub ? x3 : (right ? (s1 > 0.0f ? x1 : dh) : hr);
  clamped = false;
  if (right && dh > hi) { dh = hi; clamped = true; }
  if (dh < lo) { dh = lo; clamped = true; }
  if (!right && dh > hi) { dh = hi; clamped = true; }
  return dh;
}

// Waves z[8] as in riemann_prim of two edges and their outer speeds s1, s3
// (the middle one is their mean); sg = sqrt(g).  The straight line is that of
// edges between wet cells whose stationary waves are inside their bounds
// (tested with a margin far above the rounding of the exact bounds); a wet/dry
// edge, and one that may be clamped, adds its blocks on the way, by selections
// for both halves at once.  (One after the other through a general solver of
// their own such edges doubled the phase's time in a front's tile: 64 patches
// of 16 x 16 with a front 16.7 us a step, 15.4 so.)
// DRY = false: both cells of every edge that counts are wet.  Returns whether
// both edges took the straight line alone, which no edge with a dry cell does.
template <bool DRY>
__device__ __forceinline__ bool riemann32x2(Prim32x2 l, Prim32x2 r, float g, float sg, f2 nz,
                                            f2 (&z)[8], f2& s1, f2& s3) {
  f2 hl = sub2(l.w, l.b), hr = sub2(r.w, r.b);
  float ql0, ql1, qr0, qr1;
  upk(l.q, ql0, ql1);
  upk(r.q, qr0, qr1);
  const bool wl0 = ql0 > 0.0f, wl1 = ql1 > 0.0f, wr0 = qr0 > 0.0f, wr1 = qr1 > 0.0f;
  const bool dry = DRY && !(wl0 && wl1 && wr0 && wr1);
  f2 dn = sub2(r.n, l.n), deta = sub2(r.w, l.w), dhs = sub2(l.b, r.b);
  bool k0 = false, k1 = false;  // per half: a wall
  if (dry) {
    // the wet side, its velocity and momentum towards the dry one
    const f2 h = sel2(wl0, wl1, hl, hr), b = sel2(wl0, wl1, l.b, r.b);
    const f2 w = sel2(wl0, wl1, l.w, r.w), q = sel2(wl0, wl1, l.q, r.q);
    const f2 u = sel2(wl0, wl1, l.u, neg2(r.u)), n = sel2(wl0, wl1, l.n, neg2(r.n));
    const f2 c = sqrt2(mul2(pk1(g), h)), sw = max2(sub2(c, u), c);
    const f2 top = add2(b, add2(h, mulr2(n, rcp2(sw), nz)));  // its HLL middle surface
    float bd0, bd1, w0, w1, t0, t1;
    upk(sel2(wl0, wl1, r.b, l.b), bd0, bd1);
    upk(w, w0, w1);
    upk(top, t0, t1);
    const bool a0 = wl0 != wr0 && bd0 > w0, a1 = wl1 != wr1 && bd1 > w1;  // bed above the water
    k0 = a0 && bd0 >= t0;
    k1 = a1 && bd1 >= t1;
    // overtopped: the dry side's step lowered to the surface
    const bool o0 = a0 && !k0, o1 = a1 && !k1;
    const f2 rise = sub2(add2(w, sel2(wl0, wl1, hr, hl)), w), fall = sub2(b, w);
    deta = sel2(o0, o1, sel2(wl0, wl1, rise, neg2(rise)), deta);
    dhs = sel2(o0, o1, sel2(wl0, wl1, fall, neg2(fall)), dhs);
    // a wall: the mirrored state on the dry side (in both halves of the
    // solution, of which the wet side's waves are kept)
    deta = sel2(k0, k1, 0ull, deta);
    dhs = sel2(k0, k1, 0ull, dhs);
    hl = sel2(k0, k1, h, sel2(wl0, wl1, hl, 0ull));
    hr = sel2(k0, k1, h, sel2(wr0, wr1, hr, 0ull));
    l.n = sel2(wl0, wl1, l.n, 0ull);
    r.n = sel2(wr0, wr1, r.n, 0ull);
    const f2 nn = neg2(n);
    dn = sel2(k0, k1, add2(nn, nn), sub2(r.n, l.n));
    l.u = sel2(k0, k1, u, l.u);
    r.u = sel2(k0, k1, neg2(u), r.u);
    l.q = sel2(k0, k1, q, l.q);
    r.q = sel2(k0, k1, q, r.q);
  }
  const f2 cl = mulr2(pk1(sg), l.q, nz), cr = mulr2(pk1(sg), r.q, nz);
  const f2 ghb = mul2(pk1(g), mul2(pk1(0.5f), add2(hl, hr)));
  const f2 uhat = mulr2(fma2(l.q, l.u, mul2(r.q, r.u)), rcp2(add2(l.q, r.q)), nz);
  const f2 chat = sqrt2(ghb);
  s1 = min2(sub2(l.u, cl), sub2(uhat, chat));
  s3 = max2(add2(r.u, cr), add2(uhat, chat));
  if (dry) {
    // one side without water: the other's speed and the front's
    const bool b0 = (wl0 && wr0) || k0, b1 = (wl1 && wr1) || k1;
    const f2 u = sel2(wl0, wl1, l.u, r.u), c = sel2(wl0, wl1, cl, cr), c2 = add2(c, c);
    s1 = sel2(b0, b1, s1, sub2(u, sel2(wl0, wl1, c, c2)));
    s3 = sel2(b0, b1, s3, add2(u, sel2(wl0, wl1, c2, c)));
  }
  const f2 den = sub2(s3, s1), rden = rcp2(den);
  const f2 ns1 = neg2(s1);
  const f2 x = sub2(fma2(s3, hr, mul2(ns1, hl)), dn);
  const f2 xm = mul2(pk1(0.9999f), x);
  const f2 ok = min2(min2(min2(sub2(xm, mul2(dhs, s1)), sub2(xm, mul2(dhs, s3))), x),
                     min2(min2(add2(dhs, hl), sub2(hr, dhs)), min2(l.q, r.q)));
  float ok0, ok1;
  upk(ok, ok0, ok1);
  f2 d1 = deta;
  const bool usual = ok0 > 0.0f && ok1 > 0.0f;
  if (!usual) {
    // the stationary wave's depth jump, bounded for non-negative depths
    const f2 hh = mulr2(mulr2(x, rden, nz), den, nz);
    const f2 b1 = mul2(hh, rcp2(s1)), b3 = mul2(hh, rcp2(s3));
    float p0, p1, q0, q1, x10, x11, x30, x31, l0, l1, r0, r1, d0, e0;
    upk(s1, p0, p1);
    upk(s3, q0, q1);
    upk(b1, x10, x11);
    upk(b3, x30, x31);
    upk(hl, l0, l1);
    upk(hr, r0, r1);
    upk(dhs, d0, e0);
    bool c0, c1;
    const float j0 = jump_bound(d0, p0, q0, x10, x30, l0, r0, c0);
    const float j1 = jump_bound(e0, p1, q1, x11, x31, l1, r1, c1);
    d1 = sel2(c0 && !(ok0 > 0.0f), c1 && !(ok1 > 0.0f), sub2(sub2(hr, hl), pk(j0, j1)), deta);
  }
  const f2 d3 = fma2(ghb, deta, fma2(r.n, r.u, neg2(mul2(l.n, l.u))));
  const f2 b1 = mul2(fma2(s3, d1, neg2(dn)), rden);
  const f2 b3 = mul2(fma2(ns1, d1, dn), rden);
  z[0] = mul2(s1, b1);
  z[1] = mulr2(mul2(s1, s1), b1, nz);
  z[2] = mulr2(l.v, z[0], nz);
  z[5] = mul2(s3, b3);
  z[6] = mulr2(mul2(s3, s3), b3, nz);
  z[7] = mulr2(r.v, z[5], nz);
  z[3] = sub2(d3, add2(z[1], z[6]));
  z[4] = sub2(fma2(r.n, r.v, neg2(mul2(l.n, l.v))), add2(z[2], z[7]));
  if (dry) {
    // nothing between two dry cells, nor behind a wall
    const bool e0 = !wl0 && !wr0, e1 = !wl1 && !wr1;
    const bool f0 = k0 || e0, f1 = k1 || e1;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      z[k] = sel2(f0 && (k >= 5 ? !wr0 : k >= 3 || !wl0), f1 && (k >= 5 ? !wr1 : k >= 3 || !wl1),
                  0ull, z[k]);
    s1 = sel2(e0, e1, 0ull, s1);
    s3 = sel2(e0, e1, 0ull, s3);
  }
  return usual;
}

// riemann32x2 of one edge with a wet and a dry cell (fields w, b, n, u, v, q).
__device__ __forceinline__ void riemann32_front(const float (&l)[6], const float (&r)[6], float g,
                                                float sg, float (&z)[8], float& s1, float& s3) {
  const bool wl = l[5] > 0.0f;
  const float hl = l[0] - l[1], hr = r[0] - r[1];
  // the wet side, its velocity and momentum towards the dry one
  const float h = wl ? hl : hr, b = wl ? l[1] : r[1], w = wl ? l[0] : r[0], q = wl ? l[5] : r[5];
  const float u = wl ? l[3] : -r[3], n = wl ? l[2] : -r[2], v = wl ? l[4] : r[4];
  const float bd = wl ? r[1] : l[1], e = wl ? hr : hl;
  const float c = sqrtf(g * h), sw = fmaxf(c - u, c);
  const bool above = bd > w, wall = above && bd >= b + (h + n * rcpf(sw)), over = above && !wall;
  // jumps towards the dry side of the surface and minus the bed
  const float jw = wall ? 0.0f : (over ? (w + e) - w : (wl ? r[0] - l[0] : l[0] - r[0]));
  const float jb = wall ? 0.0f : (over ? b - w : b - bd);
  const float deta = wl ? jw : -jw, dhs = wl ? jb : -jb;
  const float dn = wall ? -n - n : -n;
  const float cq = sg * q, c2 = 2.0f * cq, us = wl ? u : -u;
  const float ghb = g * (0.5f * (wall ? h + h : h));
  const float uhat = fmaf(q, u, -(q * u)) * rcpf(q + q), chat = sqrtf(ghb);
  s1 = wall ? fminf(u - cq, uhat - chat) : us - (wl ? cq : c2);
  s3 = wall ? fmaxf(cq - u, uhat + chat) : us + (wl ? c2 : cq);
  const float gl = wl || wall ? h : 0.0f, gr = !wl || wall ? h : 0.0f;
  const float den = s3 - s1, rden = rcpf(den);
  const float hh = ((fmaf(s3, gr, -(s1 * gl)) - dn) * rden) * den;
  bool clamped;
  const float dh = jump_bound(dhs, s1, s3, hh * rcpf(s1), hh * rcpf(s3), gl, gr, clamped);
  const float d1 = clamped ? (gr - gl) - dh : deta;
  const float nu = n * u, nv = (wl ? n : -n) * v;  // the wet side's fluxes
  const float d3 = fmaf(ghb, deta, wl ? -nu : nu);
  const float b1 = fmaf(s3, d1, -dn) * rden, b3 = fmaf(-s1, d1, dn) * rden;
  z[0] = s1 * b1;
  z[1] = (s1 * s1) * b1;
  z[2] = (wl ? v : 0.0f) * z[0];
  z[5] = s3 * b3;
  z[6] = (s3 * s3) * b3;
  z[7] = (wl ? 0.0f : v) * z[5];
  z[3] = d3 - (z[1] + z[6]);
  z[4] = (wl ? -nv : nv) - (z[2] + z[7]);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (wall && (k >= 3 || !wl) && (k < 5 || wl)) z[k] = 0.0f;
}

// Limiter coefficients of one wave of two edges: hs = half the sign of the
// speed (zero at zero speed), m = 1 - nu |s|.  The smallest normal number
// keeps a vanishing wave's ratio finite.
__device__ __forceinline__ f2 limit32x2(f2 num, f2 zz, f2 hs, f2 m, f2 nz) {
  const f2 th = mulr2(num, rcp2(add2(zz, pk1(1.17549435e-38f))), nz);
  const f2 a = mul2(pk1(0.5f), add2(pk1(1.0f), th));
  const f2 phi = max2(min2(min2(a, pk1(2.0f)), add2(th, th)), pk1(0.0f));
  return mul2(mul2(hs, m), phi);
}

// edge_fluxes for the edges at w and w + 1 (planes of pitch ST, SE the place
// of the next edge of a line); wet0, wet1: the edge takes a correction (both
// its cells are wet).  Where neither does, the limiters are left out.
template <int ST, int SE>
__device__ __forceinline__ void edge32x2(const float* w, float nu, bool wet0, bool wet1, f2 nz,
                                         f2 (&am)[3], f2 (&ap)[3], f2 (&ff)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) am[k] = ap[k] = ff[k] = 0ull;
  const f2 s1 = ld2(w + 8 * ST), s3 = ld2(w + 9 * ST);
  if ((s1 | s3) == 0ull) return;  // between dry cells
  f2 z[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) z[c] = ld2(w + c * ST);
  const f2 s2 = mul2(pk1(0.5f), add2(s1, s3));
  float a1, b1, a2, b2, a3, b3;
  upk(s1, a1, b1);
  upk(s2, a2, b2);
  upk(s3, a3, b3);
  // first wave leftwards, third rightwards, the middle one to one side; an
  // edge between dry cells beside such a one has zero waves, which may go with it
  const bool usual = ((a1 < 0.0f && a3 > 0.0f && a2 != 0.0f) || (a1 == 0.0f && a3 == 0.0f)) &&
                     ((b1 < 0.0f && b3 > 0.0f && b2 != 0.0f) || (b1 == 0.0f && b3 == 0.0f));
  if (usual) {
    const bool n0 = a2 < 0.0f, n1 = b2 < 0.0f;
    am[0] = z[0];
    ap[0] = z[5];
#pragma unroll
    for (int k = 1; k < 3; ++k) {
      const f2 x = add2(sel2(n0, n1, z[k], z[5 + k]), z[2 + k]);
      am[k] = sel2(n0, n1, x, z[k]);
      ap[k] = sel2(n0, n1, z[5 + k], x);
    }
  } else {
    auto side = [](float s) { return s < 0.0f ? 1.0f : (s == 0.0f ? 0.5f : 0.0f); };
    const f2 m1 = pk(side(a1), side(b1)), m2 = pk(side(a2), side(b2)), m3 = pk(side(a3), side(b3));
    const f2 one = pk1(1.0f);
    const f2 p1 = sub2(one, m1), p2 = sub2(one, m2), p3 = sub2(one, m3);
    am[0] = add2(mul2(m1, z[0]), mul2(m3, z[5]));
    ap[0] = add2(mul2(p1, z[0]), mul2(p3, z[5]));
#pragma unroll
    for (int k = 1; k < 3; ++k) {
      am[k] = add2(add2(mul2(m1, z[k]), mul2(m3, z[5 + k])), mul2(m2, z[2 + k]));
      ap[k] = add2(add2(mul2(p1, z[k]), mul2(p3, z[5 + k])), mul2(p2, z[2 + k]));
    }
  }
  if (!(wet0 || wet1)) return;
  f2 u[8];        // the upwind edges' waves
  f2 h1, h2, h3;  // half the signs
  if (usual) {
    const bool n0 = a2 < 0.0f, n1 = b2 < 0.0f;
    if constexpr (SE % 2 == 0) {
#pragma unroll
      for (int c = 0; c < 3; ++c) u[c] = ld2(w + c * ST + SE);
#pragma unroll
      for (int c = 5; c < 8; ++c) u[c] = ld2(w + c * ST - SE);
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float lo, hi;
        upk(z[c], lo, hi);
        u[c] = pk(hi, w[c * ST + 2]);
      }
#pragma unroll
      for (int c = 5; c < 8; ++c) {
        float lo, hi;
        upk(z[c], lo, hi);
        u[c] = pk(w[c * ST - 1], lo);
      }
    }
    h1 = pk1(-0.5f);
    h3 = pk1(0.5f);
    h2 = pk(n0 ? -0.5f : 0.5f, n1 ? -0.5f : 0.5f);
  } else {
    const int o10 = a1 > 0.0f ? -SE : SE, o11 = (b1 > 0.0f ? -SE : SE) + 1;
    const int o30 = a3 > 0.0f ? -SE : SE, o31 = (b3 > 0.0f ? -SE : SE) + 1;
#pragma unroll
    for (int c = 0; c < 3; ++c) u[c] = pk(w[c * ST + o10], w[c * ST + o11]);
#pragma unroll
    for (int c = 5; c < 8; ++c) u[c] = pk(w[c * ST + o30], w[c * ST + o31]);
    auto hsign = [](float s) { return s > 0.0f ? 0.5f : (s < 0.0f ? -0.5f : 0.0f); };
    h1 = pk(hsign(a1), hsign(b1));
    h2 = pk(hsign(a2), hsign(b2));
    h3 = pk(hsign(a3), hsign(b3));
  }
  const int o20 = a2 > 0.0f ? -SE : SE, o21 = (b2 > 0.0f ? -SE : SE) + 1;
#pragma unroll
  for (int c = 3; c < 5; ++c) u[c] = pk(w[c * ST + o20], w[c * ST + o21]);
  const f2 one = pk1(1.0f), nn = pk1(-nu);
  auto abs2 = [](f2 v) { return v & 0x7fffffff7fffffffull; };
  f2 k1 = limit32x2(fma2(u[2], z[2], fma2(u[0], z[0], mul2(u[1], z[1]))),
                    fma2(z[2], z[2], fma2(z[0], z[0], mul2(z[1], z[1]))), h1,
                    fma2(nn, abs2(s1), one), nz);
  f2 k2 = limit32x2(fma2(u[3], z[3], mul2(u[4], z[4])), fma2(z[3], z[3], mul2(z[4], z[4])), h2,
                    fma2(nn, abs2(s2), one), nz);
  f2 k3 = limit32x2(fma2(u[7], z[7], fma2(u[5], z[5], mul2(u[6], z[6]))),
                    fma2(z[7], z[7], fma2(z[5], z[5], mul2(z[6], z[6]))), h3,
                    fma2(nn, abs2(s3), one), nz);
  if (!(wet0 && wet1)) {
    k1 = sel2(wet0, wet1, k1, 0ull);
    k2 = sel2(wet0, wet1, k2, 0ull);
    k3 = sel2(wet0, wet1, k3, 0ull);
  }
  ff[0] = add2(mulr2(k1, z[0], nz), mulr2(k3, z[5], nz));
  ff[1] = add2(add2(mulr2(k1, z[1], nz), mulr2(k3, z[6], nz)), mulr2(k2, z[3], nz));
  ff[2] = add2(add2(mulr2(k1, z[2], nz), mulr2(k3, z[7], nz)), mulr2(k2, z[4], nz));
}

// tsplit_prim of two cells' increments d = (mass, along, other); w, z: velocities
// along the split direction and across it, h: depths.  A dry half's result
// is not used.
__device__ __forceinline__ void tsplit32x2(f2 w, f2 z, f2 h, float g, f2 nz, const f2 (&d)[3],
                                           f2 (&plus)[3], f2 (&minus)[3]) {
  const f2 c = sqrt2(mul2(pk1(g), h));
  const f2 l1 = sub2(w, c), l3 = add2(w, c), r2c = rcp2(add2(c, c));
  const f2 c1 = mul2(l1, mul2(fma2(l3, d[0], neg2(d[1])), r2c));
  const f2 c3 = mul2(l3, mul2(fma2(neg2(l1), d[0], d[1]), r2c));
  const f2 c2 = mul2(w, fma2(neg2(z), d[0], d[2]));
  float l1a, l1b, l3a, l3b, wa, wb;
  upk(l1, l1a, l1b);
  upk(l3, l3a, l3b);
  upk(w, wa, wb);
  const f2 p1 = sel2(l1a > 0.0f, l1b > 0.0f, c1, 0ull), q1 = sel2(l1a < 0.0f, l1b < 0.0f, c1, 0ull);
  const f2 p3 = sel2(l3a > 0.0f, l3b > 0.0f, c3, 0ull), q3 = sel2(l3a < 0.0f, l3b < 0.0f, c3, 0ull);
  const f2 p2 = sel2(wa > 0.0f, wb > 0.0f, c2, 0ull), q2 = sel2(wa < 0.0f, wb < 0.0f, c2, 0ull);
  plus[0] = add2(p1, p3);
  plus[1] = add2(mulr2(p1, l1, nz), mulr2(p3, l3, nz));
  plus[2] = add2(add2(mulr2(p1, z, nz), mulr2(p3, z, nz)), p2);
  minus[0] = add2(q1, q3);
  minus[1] = add2(mulr2(q1, l1, nz), mulr2(q3, l3, nz));
  minus[2] = add2(add2(mulr2(q1, z, nz), mulr2(q3, z, nz)), q2);
}

}  // namespace gfk
