// Device arithmetic for helicity amplitudes: complex numbers, four-vectors,
// Dirac spinors in the chiral representation, colour-stripped vertex routines.
//
// Conventions (standard QFT; the paper fixes none): metric (+,-,-,-); chiral
// gamma matrices gamma^0 = [[0,1],[1,0]], gamma^k = [[0,s^k],[-s^k,0]], so that
//   Vslash = [[0, V0 - s.V], [V0 + s.V, 0]];
// helicity spinors (me_single.cuh) u(p,l) = (w_{-l} chi_l, w_{+l} chi_l),
//   v(p,l) = (-l w_{+l} chi_{-l}, l w_{-l} chi_{-l}), w_+- = sqrt(E +- |p|);
// polarisation vectors eps(k,l) = (-l e1 - i e2)/sqrt(2).
// Everything is templated on the arithmetic type T (float for the bulk path,
// double for the FP64 path and the rescue of unstable points).
#pragma once
#include <cuda_runtime.h>
#include <math.h>

// Amplitude arithmetic compiles for the device and, for operation counting with a
// counting scalar type, for the host.
#ifndef ME_HD
#define ME_HD __host__ __device__ __forceinline__
#endif

namespace me {

// square root for every arithmetic type used by the amplitude code
ME_HD float msqrt(float x) { return sqrtf(x); }
ME_HD double msqrt(double x) { return ::sqrt(x); }

// reciprocal square root: a float64 one is cheaper than the square root or the division it
// replaces (5.7 against 8.8 and 5.3 multiply-adds); float32 keeps correctly rounded steps
ME_HD double mrsqrt(double x) {
#ifdef __CUDA_ARCH__
  return ::rsqrt(x);
#else
  return 1.0 / ::sqrt(x);
#endif
}
template <typename T> ME_HD T mrsqrt(T x) { return T(1) / msqrt(x); }

template <typename T>
struct cx {
  T re, im;
};

template <typename T> ME_HD cx<T> operator+(cx<T> a, cx<T> b) { return {a.re + b.re, a.im + b.im}; }
template <typename T> ME_HD cx<T> operator-(cx<T> a, cx<T> b) { return {a.re - b.re, a.im - b.im}; }
template <typename T> ME_HD cx<T> operator-(cx<T> a) { return {-a.re, -a.im}; }
template <typename T> ME_HD cx<T> operator*(cx<T> a, cx<T> b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename T> ME_HD cx<T> operator*(T s, cx<T> a) { return {s * a.re, s * a.im}; }
template <typename T> ME_HD cx<T> operator*(cx<T> a, T s) { return {s * a.re, s * a.im}; }
template <typename T> ME_HD cx<T> conj(cx<T> a) { return {a.re, -a.im}; }
template <typename T> ME_HD cx<T> times_i(cx<T> a) { return {-a.im, a.re}; }
template <typename T> ME_HD T norm2(cx<T> a) { return a.re * a.re + a.im * a.im; }

// complex four-component object: a Lorentz vector with upper index, or a Dirac spinor
template <typename T>
struct c4 {
  cx<T> v[4];
};

template <typename T>
struct r4 {  // real four-vector (E, px, py, pz)
  T e, x, y, z;
};

template <typename T> ME_HD r4<T> operator+(r4<T> a, r4<T> b) { return {a.e + b.e, a.x + b.x, a.y + b.y, a.z + b.z}; }
template <typename T> ME_HD r4<T> operator-(r4<T> a, r4<T> b) { return {a.e - b.e, a.x - b.x, a.y - b.y, a.z - b.z}; }
template <typename T> ME_HD r4<T> operator-(r4<T> a) { return {-a.e, -a.x, -a.y, -a.z}; }
template <typename T> ME_HD r4<T> scale(T s, r4<T> a) { return {s * a.e, s * a.x, s * a.y, s * a.z}; }
template <typename T> ME_HD T mdot(r4<T> a, r4<T> b) { return a.e * b.e - a.x * b.x - a.y * b.y - a.z * b.z; }
template <typename U, typename T> ME_HD r4<U> cast4(r4<T> a) { return {(U)a.e, (U)a.x, (U)a.y, (U)a.z}; }

// Sums of complex products are written as one left-to-right chain of real products, so
// that the compiler fuses every product after the first into the running sum (one
// fused multiply-add per real product).  Written as sums of complex temporaries, each
// complex product would end in a separate add: on GB300 float64 runs at 1/64 of the
// float32 rate, so the float64 path pays for every such add.
template <typename T> ME_HD cx<T> cmac(cx<T> acc, cx<T> a, cx<T> b) {  // acc + a b
  return {acc.re + a.re * b.re - a.im * b.im, acc.im + a.re * b.im + a.im * b.re};
}
template <typename T> ME_HD cx<T> cmsb(cx<T> acc, cx<T> a, cx<T> b) {  // acc - a b
  return {acc.re - a.re * b.re + a.im * b.im, acc.im - a.re * b.im - a.im * b.re};
}

// complex-vector . complex-vector (Minkowski, no conjugation)
template <typename T>
ME_HD cx<T> cdot(const c4<T>& a, const c4<T>& b) {
  return cmsb(cmsb(cmsb(a.v[0] * b.v[0], a.v[1], b.v[1]), a.v[2], b.v[2]), a.v[3], b.v[3]);
}
// real-vector . complex-vector
template <typename T>
ME_HD cx<T> rdot(const r4<T>& a, const c4<T>& b) {
  return a.e * b.v[0] - a.x * b.v[1] - a.y * b.v[2] - a.z * b.v[3];
}
template <typename T>
ME_HD void cadd(c4<T>& acc, const c4<T>& x) {
#pragma unroll
  for (int i = 0; i < 4; ++i) acc.v[i] = acc.v[i] + x.v[i];
}
template <typename T>
ME_HD void csub(c4<T>& acc, const c4<T>& x) {
#pragma unroll
  for (int i = 0; i < 4; ++i) acc.v[i] = acc.v[i] - x.v[i];
}
template <typename T>
ME_HD void caxpy(c4<T>& acc, cx<T> a, const c4<T>& x) {
#pragma unroll
  for (int i = 0; i < 4; ++i) acc.v[i] = cmac(acc.v[i], a, x.v[i]);
}
// acc + s x, s real
template <typename T>
ME_HD void caxpy(c4<T>& acc, T s, const c4<T>& x) {
#pragma unroll
  for (int i = 0; i < 4; ++i) acc.v[i] = cx<T>{acc.v[i].re + s * x.v[i].re, acc.v[i].im + s * x.v[i].im};
}
template <typename T>
ME_HD c4<T> cneg(const c4<T>& x) {
  c4<T> o;
#pragma unroll
  for (int i = 0; i < 4; ++i) o.v[i] = -x.v[i];
  return o;
}
template <typename T>
ME_HD c4<T> czero() {
  c4<T> z;
#pragma unroll
  for (int i = 0; i < 4; ++i) z.v[i] = cx<T>{T(0), T(0)};
  return z;
}

// ---------------------------------------------------------------- wavefunctions
// Helicity-independent ingredients of the wavefunctions, computed once per event and
// shared by all helicities.
// Massive quark with spins along the light cone instead of the helicity axis (a sum over
// both spins does not depend on the axis): of the four components one is zero and two are
// real, with p+ = E + pz, s = sqrt(p+), m' = m / s, t = (px + i py) / s,
//   u_0 = (m', 0, s, t),  u_1 = (-t*, s, 0, m'),  v_0 = (-m', 0, s, t),  v_1 = (-t*, s, 0, -m').
// A slash against ubar takes 16 multiply-adds instead of 32, a product with v 8 instead of
// 16.  p+ is formed without cancellation as (m^2 + pt^2) / (E - pz) when pz < 0.
template <typename T>
struct wf_q {
  T s, m;
  cx<T> t;
};
template <typename T>
ME_HD wf_q<T> wf_quark(const r4<T>& p, T m) {
  const T pp = p.z >= T(0) ? p.e + p.z : (m * m + p.x * p.x + p.y * p.y) / (p.e - p.z);
  const T is = mrsqrt(pp);
  return wf_q<T>{pp * is, m * is, {p.x * is, p.y * is}};
}
// Massless: the two nonzero components (a, b) of u or v of helicity + along p, up to a phase
template <typename T>
ME_HD void chi_massless(const r4<T>& p, cx<T>& a, cx<T>& b) {
  const T pp = p.z >= T(0) ? p.e + p.z : p.e - p.z, is = mrsqrt(pp);
  const cx<T> t{p.x * is, p.y * is}, r{pp * is, T(0)};
  a = p.z >= T(0) ? r : conj(t);
  b = p.z >= T(0) ? t : r;
}
template <typename T>
ME_HD wf_q<T> scaled(const wf_q<T>& w, T f) {
  return wf_q<T>{f * w.s, f * w.m, f * w.t};
}

// Vector: (ct cp, ct sp, st, sp, cp) / sqrt(2) of the momentum direction.
template <typename T>
struct wf_v {
  T ccp, csp, st, sp, cp;
};
template <typename T>
ME_HD wf_v<T> wf_vector(const r4<T>& k) {
  const T r2 = T(0.70710678118654752440);
  const T pt2 = k.x * k.x + k.y * k.y, ika = mrsqrt(pt2 + k.z * k.z);
  const T ct = k.z * ika * r2;
  if (!(pt2 > T(0))) return wf_v<T>{ct, T(0), T(0), T(0), r2};
  const T ipt = mrsqrt(pt2), cp = k.x * ipt, sp = k.y * ipt;
  return wf_v<T>{ct * cp, ct * sp, pt2 * ipt * ika * r2, sp * r2, cp * r2};
}

// ---------------------------------------------------------------- Dirac algebra
// row spinor times Vslash (V complex, upper index)
template <typename T>
ME_HD c4<T> row_slash(const c4<T>& r, const c4<T>& V) {
  cx<T> a = V.v[0] - V.v[3], b = V.v[0] + V.v[3];
  cx<T> c = V.v[1] - times_i(V.v[2]);  // V1 - i V2
  cx<T> d = V.v[1] + times_i(V.v[2]);  // V1 + i V2
  c4<T> o;
  o.v[0] = cmac(r.v[2] * b, r.v[3], d);
  o.v[1] = cmac(r.v[2] * c, r.v[3], a);
  o.v[2] = cmsb(r.v[0] * a, r.v[1], d);
  o.v[3] = cmsb(r.v[1] * b, r.v[0], c);
  return o;
}
// Vslash in the chiral representation is fixed by four combinations of V: a = V0 - V3,
// b = V0 + V3, c = V1 - i V2, d = V1 + i V2.  A vector that is slashed against many rows
// is converted once.
template <typename T>
struct sl4 {
  cx<T> a, b, c, d;
};
template <typename T>
ME_HD sl4<T> slashed(const c4<T>& V) {
  return sl4<T>{V.v[0] - V.v[3], V.v[0] + V.v[3], V.v[1] - times_i(V.v[2]), V.v[1] + times_i(V.v[2])};
}
template <typename T>
ME_HD c4<T> row_slash(const c4<T>& r, const sl4<T>& S) {
  c4<T> o;
  o.v[0] = cmac(r.v[2] * S.b, r.v[3], S.d);
  o.v[1] = cmac(r.v[2] * S.c, r.v[3], S.a);
  o.v[2] = cmsb(r.v[0] * S.a, r.v[1], S.d);
  o.v[3] = cmsb(r.v[1] * S.b, r.v[0], S.c);
  return o;
}
// acc + r Sslash, accumulated in place
template <typename T>
ME_HD void row_slash_acc(c4<T>& acc, const c4<T>& r, const sl4<T>& S) {
  acc.v[0] = cmac(cmac(acc.v[0], r.v[2], S.b), r.v[3], S.d);
  acc.v[1] = cmac(cmac(acc.v[1], r.v[2], S.c), r.v[3], S.a);
  acc.v[2] = cmsb(cmac(acc.v[2], r.v[0], S.a), r.v[1], S.d);
  acc.v[3] = cmac(cmsb(acc.v[3], r.v[0], S.c), r.v[1], S.b);
}
template <typename T>
ME_HD void row_slash_acc(c4<T>& acc, const c4<T>& r, const c4<T>& V) {
  row_slash_acc(acc, r, slashed(V));
}
// s (Qslash + m) for rows, Q real: the combinations row_prop uses, formed once for a
// propagator that closes several rows (the scale s, a coupling times the reciprocal
// denominator, is folded in here instead of into every row)
template <typename T>
struct prop4 {
  T a, b, m;
  cx<T> c, d;
};
template <typename T>
ME_HD prop4<T> scaled_prop(const r4<T>& Q, T m, T s) {
  const T sx = s * Q.x, sy = s * Q.y;
  return prop4<T>{s * (Q.e - Q.z), s * (Q.e + Q.z), s * m, cx<T>{sx, -sy}, cx<T>{sx, sy}};
}
template <typename T>
ME_HD c4<T> row_prop(const c4<T>& r, const prop4<T>& P) {
  c4<T> o;
  o.v[0] = cmac(P.b * r.v[2] + P.m * r.v[0], r.v[3], P.d);
  o.v[1] = cmac(P.a * r.v[3] + P.m * r.v[1], r.v[2], P.c);
  o.v[2] = cmsb(P.a * r.v[0] + P.m * r.v[2], r.v[1], P.d);
  o.v[3] = cmsb(P.b * r.v[1] + P.m * r.v[3], r.v[0], P.c);
  return o;
}
// ---------------------------------------------------------------- polarisation vectors
// A transverse polarisation vector in the frame of the momenta has no time component and a
// real z component: 5 reals instead of 8.  Contractions and slashes against it skip the
// zeros, which a compiler may not (x * 0 is not 0 for every x): a slash takes 24 multiply-
// adds instead of 32, a product of two polarisations 9 instead of 16.
template <typename T>
struct pol {
  cx<T> x, y;
  T z;
};
template <typename T>
ME_HD pol<T> pol_of(const wf_v<T>& w, int lam, bool outgoing) {  // as polvec (me_single.cuh)
  const T s = outgoing ? T(-1) : T(1);
  return pol<T>{{lam > 0 ? -w.ccp : w.ccp, s * w.sp}, {lam > 0 ? -w.csp : w.csp, -s * w.cp}, lam > 0 ? w.st : -w.st};
}
// its slashed form: a = -z, b = z (real), c = x - i y, d = x + i y
template <typename T>
struct spol {
  T z;
  cx<T> c, d;
};
template <typename T>
ME_HD spol<T> slashed(const pol<T>& e) {
  return spol<T>{e.z, e.x - times_i(e.y), e.x + times_i(e.y)};
}
template <typename T> ME_HD cx<T> rmac(cx<T> acc, T s, cx<T> a) {  // acc + s a, s real
  return {acc.re + s * a.re, acc.im + s * a.im};
}
// row times eslash, and acc + row times eslash
template <typename T>
ME_HD c4<T> row_slash(const c4<T>& r, const spol<T>& S) {
  c4<T> o;
  o.v[0] = cmac(S.z * r.v[2], r.v[3], S.d);
  o.v[1] = cmac(-S.z * r.v[3], r.v[2], S.c);
  o.v[2] = cmsb(-S.z * r.v[0], r.v[1], S.d);
  o.v[3] = cmsb(S.z * r.v[1], r.v[0], S.c);
  return o;
}
template <typename T>
ME_HD void row_slash_acc(c4<T>& acc, const c4<T>& r, const spol<T>& S) {
  acc.v[0] = cmac(rmac(acc.v[0], S.z, r.v[2]), r.v[3], S.d);
  acc.v[1] = cmac(rmac(acc.v[1], -S.z, r.v[3]), r.v[2], S.c);
  acc.v[2] = cmsb(rmac(acc.v[2], -S.z, r.v[0]), r.v[1], S.d);
  acc.v[3] = cmsb(rmac(acc.v[3], S.z, r.v[1]), r.v[0], S.c);
}
// s (Qslash + m) times column, for the scaled propagator of row_prop
template <typename T>
ME_HD c4<T> col_prop(const prop4<T>& P, const c4<T>& s) {
  c4<T> o;
  o.v[0] = cmsb(P.a * s.v[2] + P.m * s.v[0], P.c, s.v[3]);
  o.v[1] = cmsb(P.b * s.v[3] + P.m * s.v[1], P.d, s.v[2]);
  o.v[2] = cmac(P.b * s.v[0] + P.m * s.v[2], P.c, s.v[1]);
  o.v[3] = cmac(P.a * s.v[1] + P.m * s.v[3], P.d, s.v[0]);
  return o;
}
// ubar of spin h times Vslash or eslash; ubar_0 = (s, t*, m', 0), ubar_1 = (0, m', -t, s)
template <typename T>
ME_HD c4<T> ubar_slash(const wf_q<T>& w, int h, const sl4<T>& S) {
  c4<T> o;
  if (h == 0) {
    o.v[0] = w.m * S.b;
    o.v[1] = w.m * S.c;
    o.v[2] = cmsb(w.s * S.a, conj(w.t), S.d);
    o.v[3] = cmac(-w.s * S.c, conj(w.t), S.b);
  } else {
    o.v[0] = cmsb(w.s * S.d, w.t, S.b);
    o.v[1] = cmsb(w.s * S.a, w.t, S.c);
    o.v[2] = -w.m * S.d;
    o.v[3] = w.m * S.b;
  }
  return o;
}
template <typename T>
ME_HD c4<T> ubar_slash(const wf_q<T>& w, int h, const spol<T>& S) {
  c4<T> o;
  if (h == 0) {
    o.v[0] = cx<T>{w.m * S.z, T(0)};
    o.v[1] = w.m * S.c;
    o.v[2] = -(conj(w.t) * S.d);
    o.v[2].re = o.v[2].re - w.s * S.z;
    o.v[3] = rmac(-w.s * S.c, S.z, conj(w.t));
  } else {
    o.v[0] = rmac(w.s * S.d, -S.z, w.t);
    o.v[1] = -(w.t * S.c);
    o.v[1].re = o.v[1].re - w.s * S.z;
    o.v[2] = -w.m * S.d;
    o.v[3] = cx<T>{w.m * S.z, T(0)};
  }
  return o;
}
// ubar Vslash added to a row
template <typename T>
ME_HD void ubar_slash_acc(c4<T>& acc, const wf_q<T>& w, int h, const sl4<T>& S) {
  if (h == 0) {
    acc.v[0] = rmac(acc.v[0], w.m, S.b);
    acc.v[1] = rmac(acc.v[1], w.m, S.c);
    acc.v[2] = cmsb(rmac(acc.v[2], w.s, S.a), conj(w.t), S.d);
    acc.v[3] = cmac(rmac(acc.v[3], -w.s, S.c), conj(w.t), S.b);
  } else {
    acc.v[0] = cmsb(rmac(acc.v[0], w.s, S.d), w.t, S.b);
    acc.v[1] = cmsb(rmac(acc.v[1], w.s, S.a), w.t, S.c);
    acc.v[2] = rmac(acc.v[2], -w.m, S.d);
    acc.v[3] = rmac(acc.v[3], w.m, S.b);
  }
}
// row . v of spin h
template <typename T>
ME_HD cx<T> dot_v(const c4<T>& r, const wf_q<T>& w, int h) {
  return h == 0 ? rmac(cmac(w.s * r.v[2], r.v[3], w.t), -w.m, r.v[0])
                : rmac(cmsb(w.s * r.v[1], r.v[0], conj(w.t)), -w.m, r.v[3]);
}
// eslash v of spin h
template <typename T>
ME_HD c4<T> slash_v(const spol<T>& S, const wf_q<T>& w, int h) {
  c4<T> o;
  if (h == 0) {
    o.v[0] = cmsb(cx<T>{-S.z * w.s, T(0)}, S.c, w.t);
    o.v[1] = rmac(S.z * w.t, -w.s, S.d);
    o.v[2] = cx<T>{-w.m * S.z, T(0)};
    o.v[3] = -w.m * S.d;
  } else {
    o.v[0] = w.m * S.c;
    o.v[1] = cx<T>{-w.m * S.z, T(0)};
    o.v[2] = rmac(w.s * S.c, -S.z, conj(w.t));
    o.v[3] = cmsb(cx<T>{-S.z * w.s, T(0)}, S.d, conj(w.t));
  }
  return o;
}
// A massless quark line of fixed helicity enters by two-component spinors: rho (the two
// nonzero components of its row) and sigma (of its column), current 2 rho sigma.  A row R of
// the heavy line contracted with it and with a column c gives 2 (X x + Y y):
//   X = R0 rho1 - R1 rho0,  Y = R2 sigma0 + R3 sigma1  (row side),
//   x = sigma1 c2 - sigma0 c3,  y = rho0 c0 + rho1 c1  (column side).
template <typename T>
struct c2 {
  cx<T> a, b;
};
template <typename T> ME_HD cx<T> line_X(const c4<T>& R, const c2<T>& rho) { return cmsb(R.v[0] * rho.b, R.v[1], rho.a); }
template <typename T> ME_HD cx<T> line_Y(const c4<T>& R, const c2<T>& sg) { return cmac(R.v[2] * sg.a, R.v[3], sg.b); }
template <typename T> ME_HD cx<T> line_x(const c4<T>& c, const c2<T>& sg) { return cmsb(sg.b * c.v[2], sg.a, c.v[3]); }
template <typename T> ME_HD cx<T> line_y(const c4<T>& c, const c2<T>& rho) { return cmac(rho.a * c.v[0], rho.b, c.v[1]); }
// the same for ubar and v of spin h
template <typename T>
ME_HD cx<T> ubar_X(const wf_q<T>& w, int h, const c2<T>& rho) {
  return h == 0 ? cmsb(w.s * rho.b, conj(w.t), rho.a) : -w.m * rho.a;
}
template <typename T>
ME_HD cx<T> ubar_Y(const wf_q<T>& w, int h, const c2<T>& sg) {
  return h == 0 ? w.m * sg.a : cmsb(w.s * sg.b, w.t, sg.a);
}
template <typename T>
ME_HD cx<T> v_x(const wf_q<T>& w, int h, const c2<T>& sg) {
  return h == 0 ? cmsb(w.s * sg.b, w.t, sg.a) : w.m * sg.a;
}
template <typename T>
ME_HD cx<T> v_y(const wf_q<T>& w, int h, const c2<T>& rho) {
  return h == 0 ? -w.m * rho.a : cmsb(w.s * rho.b, conj(w.t), rho.a);
}
template <typename T> ME_HD cx<T> cdot(const pol<T>& a, const pol<T>& b) {  // Minkowski product
  const cx<T> t = cmac(a.x * b.x, a.y, b.y);
  return cx<T>{-(t.re + a.z * b.z), -t.im};
}
template <typename T> ME_HD cx<T> cdot(const pol<T>& a, const c4<T>& b) {
  return -rmac(cmac(a.x * b.v[1], a.y, b.v[2]), a.z, b.v[3]);
}
template <typename T> ME_HD cx<T> rdot(const r4<T>& q, const pol<T>& e) {
  const cx<T> t = rmac(q.x * e.x, q.y, e.y);
  return cx<T>{-(t.re + q.z * e.z), -t.im};
}

// acc + w e
template <typename T>
ME_HD void caxpy(c4<T>& acc, cx<T> w, const pol<T>& e) {
  acc.v[1] = cmac(acc.v[1], w, e.x);
  acc.v[2] = cmac(acc.v[2], w, e.y);
  acc.v[3] = rmac(acc.v[3], e.z, w);
}

// A gluon along the z axis has e = s (0, 1, i H, 0) with s real and H = +-1, fixed by its
// helicity and direction: two reals' worth of arithmetic, and H at compile time leaves out
// one of the two chiral components as well.  (A beam gluon, in nearly every sample.)
template <typename T, int H>
struct axpol {
  T s;
};
template <typename T, int H>
struct axslash {  // H = 1: c = f, H = -1: d = f; a = b = 0 and the other of c, d
  T f;
};
template <typename T, int H> ME_HD axslash<T, H> slashed(const axpol<T, H>& e) { return axslash<T, H>{e.s + e.s}; }
template <typename T, int H> ME_HD cx<T> cdot_xy(const axpol<T, H>& e, cx<T> x, cx<T> y) {
  return H > 0 ? cx<T>{-e.s * (x.re - y.im), -e.s * (x.im + y.re)} : cx<T>{-e.s * (x.re + y.im), -e.s * (x.im - y.re)};
}
template <typename T, int H, int G> ME_HD cx<T> cdot(const axpol<T, H>& a, const axpol<T, G>& b) {
  return cx<T>{H == G ? T(0) : T(-2) * a.s * b.s, T(0)};
}
template <typename T, int H> ME_HD cx<T> cdot(const axpol<T, H>& a, const pol<T>& b) { return cdot_xy(a, b.x, b.y); }
template <typename T, int H> ME_HD cx<T> cdot(const axpol<T, H>& a, const c4<T>& b) { return cdot_xy(a, b.v[1], b.v[2]); }
template <typename T, int H> ME_HD cx<T> rdot(const r4<T>& q, const axpol<T, H>& e) {
  return cx<T>{-e.s * q.x, T(-H) * e.s * q.y};
}
template <typename T, int H>
ME_HD void caxpy(c4<T>& acc, cx<T> w, const axpol<T, H>& e) {
  const T t = T(H) * e.s;
  acc.v[1] = rmac(acc.v[1], e.s, w);
  acc.v[2] = cx<T>{acc.v[2].re - t * w.im, acc.v[2].im + t * w.re};
}
template <typename T, int H>
ME_HD void row_slash_acc(c4<T>& acc, const c4<T>& r, const axslash<T, H>& S) {
  if (H > 0) {
    acc.v[1] = rmac(acc.v[1], S.f, r.v[2]);
    acc.v[3] = rmac(acc.v[3], -S.f, r.v[0]);
  } else {
    acc.v[0] = rmac(acc.v[0], S.f, r.v[3]);
    acc.v[2] = rmac(acc.v[2], -S.f, r.v[1]);
  }
}
// ubar of spin h, the gluon's slash and the propagator after it
template <typename T>
ME_HD c4<T> gluon_line(const wf_q<T>& w, int h, const spol<T>& S, const prop4<T>& P) {
  return row_prop(ubar_slash(w, h, S), P);
}
template <typename T, int H>
ME_HD c4<T> gluon_line(const wf_q<T>& w, int h, const axslash<T, H>& S, const prop4<T>& P) {
  const cx<T> z{T(0), T(0)};
  c4<T> o;
  if (H > 0 && h == 0) {  // rows (., f m, ., -f s)
    const T r1 = S.f * w.m, r3 = -S.f * w.s;
    o.v[0] = r3 * P.d;
    o.v[1] = cx<T>{P.a * r3 + P.m * r1, T(0)};
    o.v[2] = -r1 * P.d;
    o.v[3] = cx<T>{P.b * r1 + P.m * r3, T(0)};
  } else if (H > 0) {  // (., -f t, ., 0)
    const cx<T> r1 = -S.f * w.t;
    o.v[0] = z;
    o.v[1] = P.m * r1;
    o.v[2] = -(r1 * P.d);
    o.v[3] = P.b * r1;
  } else if (h == 0) {  // (0, ., -f t*, .)
    const cx<T> r2 = -S.f * conj(w.t);
    o.v[0] = P.b * r2;
    o.v[1] = r2 * P.c;
    o.v[2] = P.m * r2;
    o.v[3] = z;
  } else {  // (f s, ., -f m, .)
    const T r0 = S.f * w.s, r2 = -S.f * w.m;
    o.v[0] = cx<T>{P.b * r2 + P.m * r0, T(0)};
    o.v[1] = r2 * P.c;
    o.v[2] = cx<T>{P.a * r0 + P.m * r2, T(0)};
    o.v[3] = -r0 * P.c;
  }
  return o;
}
// two gluons along the axis of equal H have no pair current: e1.e2 = q1.e2 = q2.e1 = 0
template <class E0, class E1> struct has_pair { static constexpr bool value = true; };
template <typename T, int H> struct has_pair<axpol<T, H>, axpol<T, H>> { static constexpr bool value = false; };

// ---------------------------------------------------------------- gluon vertices
// The three-gluon bracket of two conserved currents (Q_i . J_i = 0) with outgoing momenta,
//   s [(J1.J2)(Q2 - Q1) - 2 (Q2.J1) J2 + 2 (Q1.J2) J1],
// which is s vvv(J1, J2, -Q1, -Q2) (me_single.cuh) with the vanishing products Q1.J1 and Q2.J2 left out.
// `j12` receives J1.J2 of two polarisations (the four-gluon vertex needs it again).
template <typename T, class E1, class E2>
ME_HD c4<T> bracket(const E1& e1, const r4<T>& q1, const E2& e2, const r4<T>& q2, T s, cx<T>& j12) {
  j12 = cdot(e1, e2);
  const cx<T> w = s * j12, a = (T(-2) * s) * rdot(q2, e1), b = (T(2) * s) * rdot(q1, e2);
  const r4<T> d = q2 - q1;
  c4<T> J{{d.e * w, d.x * w, d.y * w, d.z * w}};
  caxpy(J, a, e2);
  caxpy(J, b, e1);
  return J;
}
// acc + the bracket of a polarisation and a current, with e.J given
template <typename T, class E>
ME_HD void bracket_acc(c4<T>& acc, const E& e, const r4<T>& q, const c4<T>& J, const r4<T>& Q, T s, cx<T> eJ) {
  const cx<T> w = s * eJ, a = (T(-2) * s) * rdot(Q, e), b = (T(2) * s) * rdot(q, J);
  const r4<T> d = Q - q;
  acc.v[0] = cmac(rmac(acc.v[0], d.e, w), a, J.v[0]);
  acc.v[1] = cmac(rmac(acc.v[1], d.x, w), a, J.v[1]);
  acc.v[2] = cmac(rmac(acc.v[2], d.y, w), a, J.v[2]);
  acc.v[3] = cmac(rmac(acc.v[3], d.z, w), a, J.v[3]);
  caxpy(acc, b, e);
}
template <typename T>
ME_HD void bracket_acc(c4<T>& acc, const c4<T>& J1, const r4<T>& Q1, const c4<T>& J2, const r4<T>& Q2, T s) {
  const cx<T> w = s * cdot(J1, J2), a = (T(-2) * s) * rdot(Q2, J1), b = (T(2) * s) * rdot(Q1, J2);
  const r4<T> d = Q2 - Q1;
  const T dd[4] = {d.e, d.x, d.y, d.z};
#pragma unroll
  for (int i = 0; i < 4; ++i) acc.v[i] = cmac(cmac(rmac(acc.v[i], dd[i], w), a, J2.v[i]), b, J1.v[i]);
}
// acc + 2 lr M - lm R - mr L: the colour-ordered four-gluon vertex of three polarisations
// or currents with the products lr = L.R, lm = L.M, mr = M.R (times the coupling) given
template <typename T, class L, class M, class R>
ME_HD void quartic_acc(c4<T>& acc, const L& l, const M& m, const R& r, cx<T> lr, cx<T> lm, cx<T> mr) {
  caxpy(acc, T(2) * lr, m);
  caxpy(acc, -lm, r);
  caxpy(acc, -mr, l);
}

}  // namespace me
