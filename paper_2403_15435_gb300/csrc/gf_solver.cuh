// Device-side building blocks of the wave-propagation step: the augmented
// Riemann solver (Sec. 3.3), the MC limiter (Sec. 3.2) and the transverse
// eigen-split of the 2D extension (Sec. 3.2, leveque2002).  Templates on the
// real type; the FP64 translation units are compiled with -fmad=false so
// that every operation rounds as written.
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

// Transverse split of an increment d = (mass, momentum along the split
// direction, other momentum) in a cell with depth h, momenta ma (along) and
// mo (other): eigenvectors of the split direction's Jacobian with speeds
// w - c, w, w + c.  plus/minus are returned in the same frame.  A part
// entering a dry neighbour whose bed is above the cell's surface is dropped;
// a dry cell splits nothing.  Wet tests and the surface come from the caller:
// wet, wetm, wetp for the cell and its neighbours at -1 and +1, eta the
// cell's surface, bm, bp the neighbours' beds (same datum as eta).
template <typename R>
__device__ __forceinline__ void tsplit(R h, R ma, R mo, R eta, bool wet,
                                       bool wetm, R bm, bool wetp, R bp,
                                       const R (&d)[3], R g, R (&plus)[3],
                                       R (&minus)[3]) {
  plus[0] = plus[1] = plus[2] = R(0);
  minus[0] = minus[1] = minus[2] = R(0);
  if (!wet) return;
  const R w = qdiv(ma, h);
  const R z = qdiv(mo, h);
  const R c = qsqrt(g * h);
  const R a1 = qdiv((w + c) * d[0] - d[1], R(2) * c);
  const R a3 = qdiv(d[1] - (w - c) * d[0], R(2) * c);
  const R a2 = d[2] - z * d[0];
  const R l1 = w - c, l2 = w, l3 = w + c;
  const R c1 = l1 * a1, c3 = l3 * a3, c2 = l2 * a2;
  const R W1[3] = {c1, c1 * l1, c1 * z};
  const R W3[3] = {c3, c3 * l3, c3 * z};
  const R W2[3] = {R(0), R(0), c2};
  const bool openp = !(!wetp && (bp > eta));
  const bool openm = !(!wetm && (bm > eta));
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const R p1 = l1 > R(0) ? W1[k] : R(0), q1 = l1 < R(0) ? W1[k] : R(0);
    const R p3 = l3 > R(0) ? W3[k] : R(0), q3 = l3 < R(0) ? W3[k] : R(0);
    const R p2 = l2 > R(0) ? W2[k] : R(0), q2 = l2 < R(0) ? W2[k] : R(0);
    if (openp) plus[k] = (p1 + p3) + p2;
    if (openm) minus[k] = (q1 + q3) + q2;
  }
}

// ------------------------------------------------------------------------
// The FP64 step's own forms.  The FP64 pipe bounds that kernel, so whatever
// belongs to a cell (velocities, celerity, square root of the depth, surface)
// is computed once per cell instead of once per edge side, and everything but
// additions and products (comparisons, selections, scalings by two, quotients,
// roots) runs in the integer and FP32 pipes.  The operations and their order
// are those of riemann / edge_fluxes / tsplit above, so the values agree bit
// for bit up to the sign of zeros.

// One side of an edge.  A dry cell has zero u, v, c and q; h, n, t, b and eta
// are its stored values.
struct Prim {
  double h, n, t, b, eta;  // depth, normal and transverse momentum, bed, h + b
  double u, v, c, q;       // n / h, t / h, sqrt(g h), sqrt(h)
  bool wet;
};

// x rounded towards zero to FP32 (0 below its range, NaN above), without the
// FP64 pipe's conversion
__device__ __forceinline__ float trunc_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int t = (int)(hi & 0x7fffffffu) - 0x38000000;
  const float f = bitsf(__funnelshift_l(lo, (unsigned)t, 3) | (hi & 0x80000000u));
  return t < 0x00100000 ? 0.0f : (t >= 0x0fe00000 ? __int_as_float(0x7fffffff) : f);
}

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
    s1 = l.u - l.c;
    s3 = l.u + twice(l.c);
  } else {
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
  if (clamped) d1 = (r.h - l.h) - dhs;
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

// Transverse split of an increment; see tsplit.  w, z: the cell's velocities
// along the split direction and across it; c: its celerity (zero when dry).
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

// Cube root of a positive normal number: the FP32 estimate (2^-20) corrected
// by two terms of the binomial series of the exact residual ratio
// d = x / y^3 - 1, y (1 + d/3 - d^2/9), whose third term is below 2^-63.
__device__ __forceinline__ double cbrt_pos(double x) {
  const int e = (int)(dbits(x) >> 52);  // biased exponent
  if ((unsigned)(e - 4) >= 2040u) return cbrt(x);
  const int k = (e - 1023 + 1533) / 3 - 511;             // floor((e - 1023) / 3)
  const double m = bitsd(dbits(x) - ((long long)(3 * k) << 52));  // [1, 8)
  const float yf = exp2f(log2f(trunc_f32(m)) * (1.0f / 3.0f));
  const unsigned fb = __float_as_uint(yf);
  // yf to FP64 by its bits
  const double y = bitsd(((long long)((fb >> 23) + 896u) << 52) | ((long long)(fb & 0x7fffffu) << 29));
  const double y2 = y * y;  // exact: 48 bits
  const double y3 = y2 * y;
  const double r = __fma_rn(-y2, y, m);
  const double d = div_rn(r, y3);
  const double c = d * __fma_rn(d, -1.0 / 9.0, 1.0 / 3.0);
  const double t = __fma_rn(y, c, y);
  return bitsd(dbits(t) + ((long long)k << 52));
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

}  // namespace gfk
