// Device helpers: boundary-aware loads, material mixtures and the WENO5-JS
// reconstruction.  Boundary conditions are realised by ghost values computed
// inside the loads (no stored ghost layers):
//   periodic axis  -> wrap
//   wall axis      -> cell-centred fields mirror about the wall face
//                     (ghost -1-m <- cell m); even for alpha, kappa, M and
//                     Neumann T, odd for tangential velocity (no slip),
//                     2 T_w - mirror for a Dirichlet temperature side;
//                     the normal velocity is odd about the wall face and 0 on it.
#pragma once

#include <math.h>

#include "fvm_internal.h"

namespace fvm {

__device__ __forceinline__ int wrapi(int c, int n) {
  if (c < 0) {
    c += n;
    if (c < 0) c = ((c % n) + n) % n;
  } else if (c >= n) {
    c -= n;
    if (c >= n) c %= n;
  }
  return c;
}

// cell-type index along one axis; flips `s` on a wall reflection when odd
__device__ __forceinline__ int mapc(int c, int n, int bc, bool odd, int& s) {
  if (bc == PER) return wrapi(c, n);
  if (c < 0) {
    if (odd) s = -s;
    return -1 - c;
  }
  if (c >= n) {
    if (odd) s = -s;
    return 2 * n - 1 - c;
  }
  return c;
}

// face-type index along the velocity's own axis
__device__ __forceinline__ int mapf(int f, int n, int bc, int& s) {
  if (bc == PER) return wrapi(f, n);
  if (f <= 0) {
    if (f == 0) s = 0;
    else s = -s;
    return -f;
  }
  if (f >= n) {
    if (f == n) { s = 0; return 0; }
    s = -s;
    return 2 * n - f;
  }
  return f;
}

__device__ __forceinline__ long long lin(const Geo& g, int i, int j, int k) {
  return (long long)k * g.sz + (long long)j * g.sy + i;
}

// even cell field (alpha, smoothed alpha, kappa, M, properties)
template <typename R>
__device__ __forceinline__ R ld_even(const R* __restrict__ a, const Geo& g, int i, int j, int k) {
  int s = 1;
  i = mapc(i, g.n[0], g.bc[0], false, s);
  j = mapc(j, g.n[1], g.bc[1], false, s);
  k = mapc(k, g.n[2], g.bc[2], false, s);
  return __ldg(a + lin(g, i, j, k));
}

// velocity component C: face-type along C, odd cell-type along the others
template <int C, typename R>
__device__ __forceinline__ R ld_vel(const R* __restrict__ a, const Geo& g, int i, int j, int k) {
  int s = 1;
  i = (C == 0) ? mapf(i, g.n[0], g.bc[0], s) : mapc(i, g.n[0], g.bc[0], true, s);
  j = (C == 1) ? mapf(j, g.n[1], g.bc[1], s) : mapc(j, g.n[1], g.bc[1], true, s);
  k = (C == 2) ? mapf(k, g.n[2], g.bc[2], s) : mapc(k, g.n[2], g.bc[2], true, s);
  R v = __ldg(a + lin(g, i, j, k));
  return s == 1 ? v : (s == 0 ? R(0) : -v);
}

// temperature with Neumann (even) or Dirichlet (2 T_w - mirror) walls
template <typename R>
__device__ __forceinline__ R ld_T(const R* __restrict__ a, const Geo& g, const TBC& tb, int i,
                                  int j, int k) {
  int c[3] = {i, j, k};
  int m[3];
  int side = -1;
  for (int d = 0; d < 3; ++d) {
    int s = 1;
    m[d] = mapc(c[d], g.n[d], g.bc[d], false, s);
    if (d == tb.axis && g.bc[d] == WALL) {
      if (c[d] < 0 && tb.dir[0]) side = 0;
      if (c[d] >= g.n[d] && tb.dir[1]) side = 1;
    }
  }
  R v = __ldg(a + lin(g, m[0], m[1], m[2]));
  if (side >= 0) {
    double sc = (m[tb.s_axis] + 0.5) * g.h;
    double Tw = tb.T0[side] + tb.amp[side] * cos(2.0 * M_PI * sc / tb.Ls);
    v = (R)(2.0 * Tw - (double)v);
  }
  return v;
}

template <typename R>
__device__ __forceinline__ R clamp01(R a) {
  return a < R(0) ? R(0) : (a > R(1) ? R(1) : a);
}

// The FP64 pipe of an SM takes 2 lanes a clock and runs double comparisons
// too; the double kernels are bound by it, so signs and ranges are read from
// the bit pattern with integer instructions (64 times the rate).
// (NaN passes through, as in the general form; a negative zero becomes 0.)
template <>
__device__ __forceinline__ double clamp01(double a) {
  const long long b = __double_as_longlong(a);
  const double r = b >= 0x3ff0000000000000LL && b <= 0x7ff0000000000000LL ? 1.0 : a;
  return b < 0 && (unsigned long long)b <= 0xfff0000000000000ULL ? 0.0 : r;
}

// a value below 0 (a zero's sign is as good as any where this is used)
__device__ __forceinline__ bool is_negative(double a) { return __double2hiint(a) < 0; }
__device__ __forceinline__ bool is_negative(float a) { return __float_as_int(a) < 0; }

// n / d to about a unit in the last place: the hardware's approximate
// reciprocal y and the geometric series 1/d = y / (1 - e) = y (1 + e + e^2 + ...),
// e = 1 - d y, cut after three terms (the hyperpower iteration of order three;
// Altman, Pacific J. Math. 10, 1960), 4 FP64 operations instead of the about 10
// of an IEEE division.  y is good to 20 bits in its operand and in its result,
// |e| <= 3 2^-20, so that the cut leaves e^3 = 0.21 u (u = 2^-53); with the
// roundings of the series' product and of the last one 2.3 u of the value.  An
// operand outside [2^-960, 2^960] takes the division.
__device__ __forceinline__ double quotient(double n, double d) {
  const unsigned u = (unsigned)__double2hiint(d) & 0x7fffffffu;
  if (u - 0x03f00000u >= 0x78000000u) return n / d;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const double e = fma(-d, y, 1.0);
  return n * fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ float quotient(float n, float d) { return n / d; }

// float -> double, exact, with integer operations for normal numbers and zero:
// the conversion instruction takes the FP64 pipe for as long as two
// additions.  It is kept for subnormal numbers, infinities and NaN, as volatile
// assembly so that the compiler does not issue it for every value and select.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), mag = u & 0x7fffffffu;
  double d = __hiloint2double((int)((u & 0x80000000u) | ((mag >> 3) + 0x38000000u)), (int)(u << 29));
  if (mag - 0x00800000u >= 0x7f000000u) {
    d = __hiloint2double((int)(u & 0x80000000u), 0);
    if (mag != 0u) asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(f));
  }
  return d;
}

// double -> R, rounded to nearest even; to float with integer operations where
// the result is a normal number or zero (the same reason)
template <typename R>
__device__ __forceinline__ R narrow(double d);
template <>
__device__ __forceinline__ double narrow<double>(double d) { return d; }
template <>
__device__ __forceinline__ float narrow<float>(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned sign = hi & 0x80000000u, mag = hi & 0x7fffffffu;
  unsigned r = sign | ((mag - 0x38000000u) << 3) | (lo >> 29);
  const unsigned rest = lo << 3;
  if (rest > 0x80000000u || (rest == 0x80000000u && (r & 1u))) ++r;
  float f = __uint_as_float(r);
  if (mag - 0x38100000u >= 0x0fe00000u) {   // not 2^-126 <= |d| < 2^128
    f = __uint_as_float(sign);
    if ((mag | lo) != 0u) asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(d));
  }
  return f;
}

// sqrt(a) for a >= 0 to about a unit in the last place: the approximate
// reciprocal root y, whose error Newton's iteration for a^-1/2 (a y (1 + e/2), e =
// 1 - a y^2) and then Newton's iteration for the root (z + (a - z^2) / (2 z), with y
// for 1/z) square away: 5 FP64 operations instead of about 15.  With y good to d =
// 3 2^-20, z is to 3/2 d^2 + u and the result to that times d and its rounding, 1.4 u.
// Operands outside [2^-960, 2^960] take the root instruction.  A 0, which most
// cells (away from the interface) pass, is returned first: inside that branch it
// cost the 149 x 90 x 75 predictor 2.81 -> 2.93 ms.
__device__ __forceinline__ double root(double a) {
  const int hi = __double2hiint(a);
  if ((hi | __double2loint(a)) == 0) return 0.0;
  if ((unsigned)(hi - 0x03f00000) >= 0x78000000u) return sqrt(a);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double ay = a * y;
  const double e = fma(-ay, y, 1.0);
  const double z = fma(0.5 * e, ay, ay);            // a y (1 + e/2)
  return fma(fma(-z, z, a), 0.5 * y, z);
}
__device__ __forceinline__ float root(float a) { return sqrtf(a); }

// The double kernels below reorder their sums and mixtures to save FP64
// operations.  The float forms keep the order of operations they always had,
// bit for bit: they are not bound by arithmetic (the same reordering gave 3 %
// of a 256^3 step), and with a density ratio of 7900 a last-bit change of the
// predicted velocity moves the pressure beside the interface by 10^-3.

// arithmetic mixture a*p1 + (1-a)*p0 with a = clamp(alpha, 0, 1)
template <typename R>
__device__ __forceinline__ R mixp(R alpha, const double* pair) {
  R a = clamp01(alpha);
  return a * (R)pair[1] + (R(1) - a) * (R)pair[0];
}

template <typename R>
__device__ __forceinline__ R sigma_of_T(R T, const Phys& ph) {
  return (R)ph.sigma0 + (R)ph.dsdT * (T - (R)ph.T0);
}

// A pair of phase values as the double kernels mix them: lo + t d from the smaller
// value lo, t the fraction of the phase with the larger one.  Every term is
// positive, so that the mixture keeps its digits wherever the interface is; taken
// from the larger value, p0 + a (p1 - p0), the pair (7900, 1.2) kept 12 of 16 of
// them in the light phase (a relative error of 5e-13 in rho).
template <typename R>
struct Mix {
  R lo, d;
  int heavy0;   // phase [0] has the larger value
};

template <typename R>
inline Mix<R> make_mix(const double* p) {
  const int heavy0 = p[0] > p[1];
  return {(R)p[heavy0 ? 1 : 0], (R)(heavy0 ? p[0] - p[1] : p[1] - p[0]), heavy0};
}

// the fraction t of a phase fraction: a = clamp(alpha, 0, 1), or 1 - a
template <typename R>
__device__ __forceinline__ R part(R alpha, const Mix<R>& m);
template <>
__device__ __forceinline__ double part(double alpha, const Mix<double>& m) {
  double t = clamp01(alpha);
  // (volatile, so that the usual order does not pay for the subtraction)
  if (m.heavy0) asm volatile("sub.rn.f64 %0, %1, %0;" : "+d"(t) : "d"(1.0));
  return t;
}
template <>
__device__ __forceinline__ float part(float alpha, const Mix<float>&) { return clamp01(alpha); }

// Material and source constants in the working precision, so that float
// kernels carry no double arithmetic or conversions.
template <typename R>
struct PhysR {
  R rho[2], mu[2], lam[2], rcp[2];
  R sigma0, dsdT, T0;
  R g[3];
  R eps_a, eps_T, eps_u, eps_n;
  R L[3];
  R h, ih;
  R dsdc, c0, diff_c[2], eps_c;
  Mix<R> mrho, mmu, mlam, mrcp, mdiff;   // the pairs again, as the double kernels mix them
};

template <typename R>
inline PhysR<R> make_physr(const Phys& ph, const Geo& g) {
  PhysR<R> q;
  for (int k = 0; k < 2; ++k) {
    q.rho[k] = (R)ph.rho[k];
    q.mu[k] = (R)ph.mu[k];
    q.lam[k] = (R)ph.lam[k];
    q.rcp[k] = (R)ph.rcp[k];
  }
  q.sigma0 = (R)ph.sigma0;
  q.dsdT = (R)ph.dsdT;
  q.T0 = (R)ph.T0;
  for (int d = 0; d < 3; ++d) {
    q.g[d] = (R)ph.g[d];
    q.L[d] = (R)ph.L[d];
  }
  q.eps_a = (R)ph.eps_a;
  q.eps_T = (R)ph.eps_T;
  q.eps_u = (R)ph.eps_u;
  q.eps_n = (R)ph.eps_n;
  q.h = (R)g.h;
  q.ih = (R)g.ih;
  q.dsdc = (R)ph.dsdc;
  q.c0 = (R)ph.c0;
  q.diff_c[0] = (R)ph.diff_c[0];
  q.diff_c[1] = (R)ph.diff_c[1];
  q.eps_c = (R)ph.eps_c;
  q.mrho = make_mix<R>(ph.rho);
  q.mmu = make_mix<R>(ph.mu);
  q.mlam = make_mix<R>(ph.lam);
  q.mrcp = make_mix<R>(ph.rcp);
  q.mdiff = make_mix<R>(ph.diff_c);
  return q;
}

// arithmetic mixture of a pair (m: the same pair)
template <typename R>
__device__ __forceinline__ R mixr(R alpha, const R* pair, const Mix<R>& m) {
  if (sizeof(R) == 8) return m.lo + part(alpha, m) * m.d;
  R a = clamp01(alpha);
  return a * pair[1] + (R(1) - a) * pair[0];
}

template <typename R>
__device__ __forceinline__ R sigma_r(R T, const PhysR<R>& q) {
  return q.sigma0 + q.dsdT * (T - q.T0);
}

// sigma(c, T) of Eq. 5 with the solutal term
template <typename R>
__device__ __forceinline__ R sigma_rc(R T, R c, const PhysR<R>& q) {
  return q.sigma0 + q.dsdT * (T - q.T0) + q.dsdc * (c - q.c0);
}

// harmonic face mean 2 a b / (a + b), 0 where both vanish
template <typename R>
__device__ __forceinline__ R harmonic(R a, R b) {
  const R s = a + b;
  return s > R(0) ? R(2) * a * b / s : R(0);
}

// WENO5-JS value at the face right of v0 from cells v0-2 .. v0+2 (left bias),
// nonlinear weights a_k = d_k / (eps + beta_k)^2, d = (0.1, 0.6, 0.3).
//
// In double it is written as v0 plus a correction in first and second
// differences:
//   q_0 - v0 = (5 d2 - 2 d1)/6,  q_1 - v0 = (d2 + 2 d3)/6,  q_2 - v0 = (4 d3 - d4)/6,
//   12/13 (eps + beta_k) = t_k^2 + 3/13 u_k^2 + 12/13 eps = B_k,
// the weights up to a common factor 1 : 6 : 3 over B_0^2 : B_1^2 : B_2^2, brought
// over the common denominator (which grows like beta^4, far inside the double
// range) for one quotient: 40 FP64 operations instead of 61.  128^3 double, per
// stage, with the other counts of the kernels: momentum 4.27 -> 3.22 ms, scalars
// 2.89 -> 1.86, interface 1.47 -> 0.77.
//
// In float the common denominator would overflow once velocity jumps reach
// ~1e4, so float keeps the reciprocal form (which underflows gracefully
// instead) with the fast approximate division: the weights need only a few
// correct digits.
template <typename R>
__device__ __forceinline__ R weno5(R vm2, R vm1, R v0, R vp1, R vp2, R eps) {
  if (sizeof(R) == 8) {
    const R d1 = vm1 - vm2, d2 = v0 - vm1, d3 = vp1 - v0, d4 = vp2 - vp1;
    const R t0 = d2 - d1, t1 = d3 - d2, t2 = d4 - d3;
    const R u0 = R(3) * d2 - d1, u1 = d2 + d3, u2 = d4 - R(3) * d3;
    const R c = R(3.0 / 13.0), e = R(12.0 / 13.0) * eps;
    const R B0 = t0 * t0 + (c * (u0 * u0) + e);
    const R B1 = t1 * t1 + (c * (u1 * u1) + e);
    const R B2 = t2 * t2 + (c * (u2 * u2) + e);
    const R r0 = R(2) * u0 - d2, r1 = R(2) * d3 + d2, r2 = d3 - u2;
    const R P0 = B1 * B2, P1 = B0 * B2, P2 = B0 * B1;
    const R a0 = P0 * P0, a1 = P1 * P1 * R(6), a2 = P2 * P2 * R(3);
    return v0 + R(1.0 / 6.0) * quotient(a0 * r0 + a1 * r1 + a2 * r2, a0 + a1 + a2);
  }
  const R c6 = R(1) / R(6);
  R q0 = (R(2) * vm2 - R(7) * vm1 + R(11) * v0) * c6;
  R q1 = (-vm1 + R(5) * v0 + R(2) * vp1) * c6;
  R q2 = (R(2) * v0 + R(5) * vp1 - vp2) * c6;
  R t0 = vm2 - R(2) * vm1 + v0, u0 = vm2 - R(4) * vm1 + R(3) * v0;
  R t1 = vm1 - R(2) * v0 + vp1, u1 = vm1 - vp1;
  R t2 = v0 - R(2) * vp1 + vp2, u2 = R(3) * v0 - R(4) * vp1 + vp2;
  const R c1312 = R(13) / R(12);
  R b0 = c1312 * t0 * t0 + R(0.25) * u0 * u0;
  R b1 = c1312 * t1 * t1 + R(0.25) * u1 * u1;
  R b2 = c1312 * t2 * t2 + R(0.25) * u2 * u2;
  R s0 = (eps + b0) * (eps + b0);
  R s1 = (eps + b1) * (eps + b1);
  R s2 = (eps + b2) * (eps + b2);
  // the weights only need a few correct digits: fast reciprocal division
  R a0 = __fdividef(R(0.1), s0), a1 = __fdividef(R(0.6), s1), a2 = __fdividef(R(0.3), s2);
  return __fdividef(a0 * q0 + a1 * q1 + a2 * q2, a0 + a1 + a2);
}

// flux U * phi_face from the six values v[0..5] = phi at offsets -3..2 of the
// face (v[2] left of it, v[3] right of it): left-biased WENO5 when U >= 0.
// In double the cells are selected by U's sign bit, so that one
// reconstruction is evaluated and no FP64 comparison.
template <typename R>
__device__ __forceinline__ R upwind_flux(R U, const R* v, R eps) {
  if (sizeof(R) == 8) {
    const bool neg = is_negative(U);
    return U * weno5(neg ? v[5] : v[0], neg ? v[4] : v[1], neg ? v[3] : v[2], neg ? v[2] : v[3],
                     neg ? v[1] : v[4], eps);
  }
  R val = (U >= R(0)) ? weno5(v[0], v[1], v[2], v[3], v[4], eps)
                      : weno5(v[5], v[4], v[3], v[2], v[1], eps);
  return U * val;
}

}  // namespace fvm
