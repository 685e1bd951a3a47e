// Helicity amplitudes one at a time (host check, me_blockcheck.cu).
//
// The kernels evaluate helicity blocks and closed forms (me_procs.cuh).  The routines here take a single
// helicity configuration with helicity spinors and plain vertices -- colour-ordered
// recursion for t tbar + gluons, Feynman diagrams for the quark processes -- on the same
// per-event kinematics, and share none of the blocks' shortcuts.
#pragma once
#include "me_procs.cuh"

namespace me {

template <typename T>
ME_HD void cscale(c4<T>& x, T a) {
#pragma unroll
  for (int i = 0; i < 4; ++i) x.v[i] = a * x.v[i];
}

// two-component helicity eigenstate chi_lam along p/|p|; |p|+pz is formed without
// cancellation as pt^2/(|p|-pz) when pz < 0.
template <typename T>
ME_HD void chi(const r4<T>& p, int lam, cx<T>& c0, cx<T>& c1) {
  T pt2 = p.x * p.x + p.y * p.y;
  T pa = msqrt(pt2 + p.z * p.z);
  T s = (p.z >= T(0)) ? pa + p.z : pt2 / (pa - p.z);
  if (s > T(0)) {
    T rden = T(1) / msqrt(T(2) * pa * s);
    if (lam > 0) {
      c0 = cx<T>{s * rden, T(0)};
      c1 = cx<T>{p.x * rden, p.y * rden};
    } else {
      c0 = cx<T>{-p.x * rden, p.y * rden};
      c1 = cx<T>{s * rden, T(0)};
    }
  } else {  // exactly along -z
    if (lam > 0) {
      c0 = cx<T>{T(0), T(0)};
      c1 = cx<T>{T(1), T(0)};
    } else {
      c0 = cx<T>{T(-1), T(0)};
      c1 = cx<T>{T(0), T(0)};
    }
  }
}

template <typename T>
ME_HD void omegas(const r4<T>& p, T m, T& wp, T& wm) {
  T pa = msqrt(p.x * p.x + p.y * p.y + p.z * p.z);
  wp = msqrt(p.e + pa);
  wm = (m == T(0)) ? T(0) : m / wp;
}

template <typename T>
ME_HD c4<T> spinor_u(const r4<T>& p, T m, int lam) {
  T wp, wm;
  omegas(p, m, wp, wm);
  cx<T> a, b;
  chi(p, lam, a, b);
  T top = lam > 0 ? wm : wp, bot = lam > 0 ? wp : wm;
  return c4<T>{{top * a, top * b, bot * a, bot * b}};
}

template <typename T>
ME_HD c4<T> spinor_v(const r4<T>& p, T m, int lam) {
  T wp, wm;
  omegas(p, m, wp, wm);
  cx<T> a, b;
  chi(p, -lam, a, b);
  T top = lam > 0 ? -wp : wm;   // -lam * w_{+lam}
  T bot = lam > 0 ? wm : -wp;   //  lam * w_{-lam}
  return c4<T>{{top * a, top * b, bot * a, bot * b}};
}

// Dirac adjoint psi^dagger gamma^0 (chiral rep: swap blocks, conjugate)
template <typename T>
ME_HD c4<T> dbar(const c4<T>& s) {
  return c4<T>{{conj(s.v[2]), conj(s.v[3]), conj(s.v[0]), conj(s.v[1])}};
}

template <typename T>
ME_HD c4<T> polvec(const r4<T>& k, int lam, bool outgoing) {
  T pt2 = k.x * k.x + k.y * k.y;
  T pt = msqrt(pt2);
  T ka = msqrt(pt2 + k.z * k.z);
  T ct = k.z / ka, st = pt / ka;
  T cp = T(1), sp = T(0);
  if (pt > T(0)) {
    cp = k.x / pt;
    sp = k.y / pt;
  }
  const T r2 = T(0.70710678118654752440);
  // eps = (-lam e1 - i e2)/sqrt(2), e1 = (0, ct cp, ct sp, -st), e2 = (0, -sp, cp, 0)
  T l = (T)lam;
  c4<T> e;
  e.v[0] = cx<T>{T(0), T(0)};
  e.v[1] = cx<T>{-l * ct * cp * r2, sp * r2};
  e.v[2] = cx<T>{-l * ct * sp * r2, -cp * r2};
  e.v[3] = cx<T>{l * st * r2, T(0)};
  if (outgoing) {
#pragma unroll
    for (int i = 1; i < 4; ++i) e.v[i] = conj(e.v[i]);
  }
  return e;
}

// Vslash times column spinor
template <typename T>
ME_HD c4<T> slash_col(const c4<T>& V, const c4<T>& s) {
  cx<T> a = V.v[0] - V.v[3], b = V.v[0] + V.v[3];
  cx<T> c = V.v[1] - times_i(V.v[2]);
  cx<T> d = V.v[1] + times_i(V.v[2]);
  c4<T> o;
  o.v[0] = cmsb(a * s.v[2], c, s.v[3]);
  o.v[1] = cmsb(b * s.v[3], d, s.v[2]);
  o.v[2] = cmac(b * s.v[0], c, s.v[1]);
  o.v[3] = cmac(d * s.v[0], a, s.v[1]);
  return o;
}
// row spinor times (Qslash + m), Q real
template <typename T>
ME_HD c4<T> row_prop(const c4<T>& r, const r4<T>& Q, T m) {
  T a = Q.e - Q.z, b = Q.e + Q.z;
  cx<T> c = cx<T>{Q.x, -Q.y}, d = cx<T>{Q.x, Q.y};
  c4<T> o;
  o.v[0] = cmac(b * r.v[2] + m * r.v[0], r.v[3], d);
  o.v[1] = cmac(a * r.v[3] + m * r.v[1], r.v[2], c);
  o.v[2] = cmsb(a * r.v[0] + m * r.v[2], r.v[1], d);
  o.v[3] = cmsb(b * r.v[1] + m * r.v[3], r.v[0], c);
  return o;
}
// (-Qslash + m) times column spinor, Q real
template <typename T>
ME_HD c4<T> col_prop(const r4<T>& Q, T m, const c4<T>& s) {
  T a = Q.e - Q.z, b = Q.e + Q.z;
  cx<T> c = cx<T>{Q.x, -Q.y}, d = cx<T>{Q.x, Q.y};
  c4<T> o;
  o.v[0] = cmac(m * s.v[0] - a * s.v[2], c, s.v[3]);
  o.v[1] = cmac(m * s.v[1] - b * s.v[3], d, s.v[2]);
  o.v[2] = cmsb(m * s.v[2] - b * s.v[0], c, s.v[1]);
  o.v[3] = cmsb(m * s.v[3] - a * s.v[1], d, s.v[0]);
  return o;
}
// vector current J^mu = r gamma^mu s
template <typename T>
ME_HD c4<T> vcurrent(const c4<T>& r, const c4<T>& s) {
  c4<T> J;
  J.v[0] = cmac(cmac(cmac(r.v[0] * s.v[2], r.v[1], s.v[3]), r.v[2], s.v[0]), r.v[3], s.v[1]);
  J.v[1] = cmsb(cmsb(cmac(r.v[0] * s.v[3], r.v[1], s.v[2]), r.v[2], s.v[1]), r.v[3], s.v[0]);
  J.v[2] = times_i(cmac(cmsb(cmsb(r.v[1] * s.v[2], r.v[0], s.v[3]), r.v[3], s.v[0]), r.v[2], s.v[1]));
  J.v[3] = cmac(cmsb(cmsb(r.v[0] * s.v[2], r.v[1], s.v[3]), r.v[2], s.v[0]), r.v[3], s.v[1]);
  return J;
}
template <typename T>
ME_HD cx<T> spdot(const c4<T>& r, const c4<T>& s) {
  return cmac(cmac(cmac(r.v[0] * s.v[0], r.v[1], s.v[1]), r.v[2], s.v[2]), r.v[3], s.v[3]);
}

// three-gluon Lorentz structure contracted with J1_mu J2_nu, momenta k1,k2,k3 incoming:
// W^rho = (J1.J2)(k1-k2)^rho + J2^rho (k2-k3).J1 + J1^rho (k3-k1).J2
template <typename T>
ME_HD c4<T> vvv(const c4<T>& J1, const c4<T>& J2, const r4<T>& k1, const r4<T>& k2) {
  r4<T> k3 = -(k1 + k2);
  cx<T> j12 = cdot(J1, J2);
  cx<T> a = rdot(k2 - k3, J1);
  cx<T> b = rdot(k3 - k1, J2);
  r4<T> d = k1 - k2;
  c4<T> W;
  W.v[0] = cmac(cmac(d.e * j12, a, J2.v[0]), b, J1.v[0]);
  W.v[1] = cmac(cmac(d.x * j12, a, J2.v[1]), b, J1.v[1]);
  W.v[2] = cmac(cmac(d.y * j12, a, J2.v[2]), b, J1.v[2]);
  W.v[3] = cmac(cmac(d.z * j12, a, J2.v[3]), b, J1.v[3]);
  return W;
}
// s W(J1, J2), and acc + s W(J1, J2): the scale goes into the three scalar coefficients
template <typename T>
ME_HD c4<T> vvv(const c4<T>& J1, const c4<T>& J2, const r4<T>& k1, const r4<T>& k2, T s) {
  r4<T> k3 = -(k1 + k2);
  const cx<T> j12 = s * cdot(J1, J2);
  const cx<T> a = s * rdot(k2 - k3, J1);
  const cx<T> b = s * rdot(k3 - k1, J2);
  r4<T> d = k1 - k2;
  c4<T> W;
  W.v[0] = cmac(cmac(d.e * j12, a, J2.v[0]), b, J1.v[0]);
  W.v[1] = cmac(cmac(d.x * j12, a, J2.v[1]), b, J1.v[1]);
  W.v[2] = cmac(cmac(d.y * j12, a, J2.v[2]), b, J1.v[2]);
  W.v[3] = cmac(cmac(d.z * j12, a, J2.v[3]), b, J1.v[3]);
  return W;
}
// colour-ordered four-gluon structure: 2(L.R) M - (L.M) R - (M.R) L
template <typename T>
ME_HD c4<T> vvvv_ordered(const c4<T>& L, const c4<T>& M, const c4<T>& R) {
  cx<T> lr = cdot(L, R), lm = cdot(L, M), mr = cdot(M, R);
  cx<T> two_lr = lr + lr;
  c4<T> o;
#pragma unroll
  for (int i = 0; i < 4; ++i) o.v[i] = cmsb(cmsb(two_lr * M.v[i], lm, R.v[i]), mr, L.v[i]);
  return o;
}

// ---------------------------------------------------------------- amplitudes
__host__ __device__ constexpr int factorial(int n) { return n <= 1 ? 1 : n * factorial(n - 1); }

// permutation number `idx` (lexicographic) of {0..n-1}
ME_HD void nth_perm(int n, int idx, int* out) {
  int pool[4] = {0, 1, 2, 3};
  int m = n;
  for (int i = 0; i < n; ++i) {
    int f = factorial(m - 1);
    int k = idx / f;
    idx -= k * f;
    out[i] = pool[k];
    for (int j = k; j < m - 1; ++j) pool[j] = pool[j + 1];
    --m;
  }
}

// Generic colour-ordered recursion (used for 4 gluons): for every ordering, contiguous
// gluon currents J[i][j] and the top line U[k]; denominators from the per-event table.
template <typename T, int NG>
ME_HD void amp_ttng(const KinTT<T, NG>& K, int hel, const Couplings& cp, cx<T>* A) {
  constexpr int NF = factorial(NG);
  const T g = gs_of<T>(cp);
  const T mt = mt_of<T>(cp);
  c4<T> eps[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    const int l = i < 2 ? i : i + 2;
    eps[i] = polvec(K.pl[l], hel_of(hel, l), l >= 2);
  }
  const c4<T> ub = dbar(spinor_u(K.pl[2], mt, hel_of(hel, 2)));
  const c4<T> vb = spinor_v(K.pl[3], mt, hel_of(hel, 3));
  for (int f = 0; f < NF; ++f) {
    int s[NG];
    nth_perm(NG, f, s);
    c4<T> J[NG][NG];
    r4<T> Q[NG][NG];
    int M[NG][NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      J[i][i] = eps[s[i]];
      Q[i][i] = K.q[s[i]];
      M[i][i] = 1 << s[i];
    }
#pragma unroll
    for (int len = 2; len <= NG; ++len) {
#pragma unroll
      for (int i = 0; i + len - 1 < NG; ++i) {
        const int j = i + len - 1;
        Q[i][j] = Q[i][j - 1] + K.q[s[j]];
        M[i][j] = M[i][j - 1] | (1 << s[j]);
        const T inv = K.ig[M[i][j]];
        c4<T> acc = czero<T>();
#pragma unroll
        for (int k = i; k < j; ++k) cadd(acc, vvv(J[i][k], J[k + 1][j], -Q[i][k], -Q[k + 1][j]));
        cscale(acc, -g * inv);
        if (len >= 3) {
          c4<T> acc4 = czero<T>();
#pragma unroll
          for (int k = i; k < j - 1; ++k)
#pragma unroll
            for (int l = k + 1; l < j; ++l) cadd(acc4, vvvv_ordered(J[i][k], J[k + 1][l], J[l + 1][j]));
          caxpy(acc, cx<T>{g * g * inv, T(0)}, acc4);
        }
        J[i][j] = acc;
      }
    }
    c4<T> U[NG];
    U[0] = ub;
    r4<T> Qu = K.pl[2];
#pragma unroll
    for (int k = 1; k < NG; ++k) {
      Qu = Qu + K.q[s[k - 1]];
      c4<T> acc = czero<T>();
#pragma unroll
      for (int j = 0; j < k; ++j) cadd(acc, row_slash(U[j], J[j][k - 1]));
      c4<T> pr = row_prop(acc, Qu, mt);
      cscale(pr, -g * K.iq[M[0][k - 1]]);
      U[k] = pr;
    }
    cx<T> a = cx<T>{T(0), T(0)};
#pragma unroll
    for (int j = 0; j < NG; ++j) a = a + spdot(row_slash(U[j], J[j][NG - 1]), vb);
    A[f] = times_i(a) * g;
  }
}

// t tbar + 2 or 3 gluons with every sub-current computed once per helicity.
// Colour-ordered currents obey the reflection identity J(s reversed) = (-1)^(k+1) J(s)
// for k gluons (V3 is antisymmetric in its two legs, the ordered V4 symmetric in its
// outer legs), so J(yx) = -J(xy) and J(zyx) = J(xyz); the quark currents U(x), U(xy)
// and the amplitudes of all orderings then reuse them.  Orderings are numbered
// lexicographically as in amp_ttng, so the colour basis is the same.
template <typename T>
ME_HD void amp_tt2_fast(const KinTT<T, 2>& K, int hel, const Couplings& cp, cx<T>* A) {
  const T g = gs_of<T>(cp), mt = mt_of<T>(cp);
  const r4<T> k0 = K.q[0], k1 = K.q[1], kt = K.pl[2];
  const c4<T> e0 = polvec(K.pl[0], hel_of(hel, 0), false);
  const c4<T> e1 = polvec(K.pl[1], hel_of(hel, 1), false);
  const c4<T> ub = dbar(spinor_u(kt, mt, hel_of(hel, 2)));
  const c4<T> vb = spinor_v(K.pl[3], mt, hel_of(hel, 3));
  c4<T> J01 = vvv(e0, e1, -k0, -k1);
  cscale(J01, -g * K.ig[3]);
  const cx<T> s01 = spdot(row_slash(ub, J01), vb);
  c4<T> U0 = row_prop(row_slash(ub, e0), kt + k0, mt);
  cscale(U0, -g * K.iq[1]);
  c4<T> U1 = row_prop(row_slash(ub, e1), kt + k1, mt);
  cscale(U1, -g * K.iq[2]);
  // A(01) = ig[ub J01 v + U0 e1 v],  A(10) = ig[-ub J01 v + U1 e0 v]
  A[0] = times_i(s01 + spdot(row_slash(U0, e1), vb)) * g;
  A[1] = times_i(spdot(row_slash(U1, e0), vb) - s01) * g;
}

template <typename T>
ME_HD void amp_tt3_fast(const KinTT<T, 3>& K, int hel, const Couplings& cp, cx<T>* A) {
  const T g = gs_of<T>(cp), mt = mt_of<T>(cp);
  const r4<T> k0 = K.q[0], k1 = K.q[1], k2 = K.q[2], kt = K.pl[2];
  const c4<T> e0 = polvec(K.pl[0], hel_of(hel, 0), false);
  const c4<T> e1 = polvec(K.pl[1], hel_of(hel, 1), false);
  const c4<T> e2 = polvec(K.pl[4], hel_of(hel, 4), true);
  const c4<T> ub = dbar(spinor_u(kt, mt, hel_of(hel, 2)));
  const c4<T> vb = spinor_v(K.pl[3], mt, hel_of(hel, 3));
  // pair currents J(xy), x<y; J(yx) = -J(xy)
  c4<T> J01 = vvv(e0, e1, -k0, -k1);
  cscale(J01, -g * K.ig[3]);
  c4<T> J02 = vvv(e0, e2, -k0, -k2);
  cscale(J02, -g * K.ig[5]);
  c4<T> J12 = vvv(e1, e2, -k1, -k2);
  cscale(J12, -g * K.ig[6]);
  // three-gluon currents F(abc) = F(cba): -(g/Q^2)[V3(a, bc) + V3(ab, c)] + (g^2/Q^2) V4(a,b,c)
  const T c3 = -g * K.ig[7], c4g = g * g * K.ig[7];
  cx<T> a[6];
  {
    c4<T> F = vvv(e0, J12, -k0, -(k1 + k2));
    cadd(F, vvv(J01, e2, -(k0 + k1), -k2));
    cscale(F, c3);
    caxpy(F, cx<T>{c4g, T(0)}, vvvv_ordered(e0, e1, e2));
    a[0] = a[5] = spdot(row_slash(ub, F), vb);  // 012, 210
  }
  {
    c4<T> mJ12 = J12;
    cscale(mJ12, T(-1));
    c4<T> F = vvv(e0, mJ12, -k0, -(k1 + k2));
    cadd(F, vvv(J02, e1, -(k0 + k2), -k1));
    cscale(F, c3);
    caxpy(F, cx<T>{c4g, T(0)}, vvvv_ordered(e0, e2, e1));
    a[1] = a[3] = spdot(row_slash(ub, F), vb);  // 021, 120
  }
  {
    c4<T> mJ01 = J01;
    cscale(mJ01, T(-1));
    c4<T> F = vvv(e1, J02, -k1, -(k0 + k2));
    cadd(F, vvv(mJ01, e2, -(k0 + k1), -k2));
    cscale(F, c3);
    caxpy(F, cx<T>{c4g, T(0)}, vvvv_ordered(e1, e0, e2));
    a[2] = a[4] = spdot(row_slash(ub, F), vb);  // 102, 201
  }
  // orderings grouped by the gluon next to the top: U(x), then U(x y) = U(x) e_y + ubar J(xy)
  {  // x = 0: orderings 012 (a0), 021 (a1)
    c4<T> U = row_prop(row_slash(ub, e0), kt + k0, mt);
    cscale(U, -g * K.iq[1]);
    const cx<T> t = spdot(row_slash(U, J12), vb);
    a[0] = a[0] + t;
    a[1] = a[1] - t;
    c4<T> r = row_slash(U, e1);
    cadd(r, row_slash(ub, J01));
    c4<T> W = row_prop(r, kt + k0 + k1, mt);
    cscale(W, -g * K.iq[3]);
    a[0] = a[0] + spdot(row_slash(W, e2), vb);
    r = row_slash(U, e2);
    cadd(r, row_slash(ub, J02));
    W = row_prop(r, kt + k0 + k2, mt);
    cscale(W, -g * K.iq[5]);
    a[1] = a[1] + spdot(row_slash(W, e1), vb);
  }
  {  // x = 1: orderings 102 (a2), 120 (a3)
    c4<T> U = row_prop(row_slash(ub, e1), kt + k1, mt);
    cscale(U, -g * K.iq[2]);
    const cx<T> t = spdot(row_slash(U, J02), vb);
    a[2] = a[2] + t;
    a[3] = a[3] - t;
    c4<T> r = row_slash(U, e0);
    c4<T> b = row_slash(ub, J01);
    cscale(b, T(-1));
    cadd(r, b);
    c4<T> W = row_prop(r, kt + k0 + k1, mt);
    cscale(W, -g * K.iq[3]);
    a[2] = a[2] + spdot(row_slash(W, e2), vb);
    r = row_slash(U, e2);
    cadd(r, row_slash(ub, J12));
    W = row_prop(r, kt + k1 + k2, mt);
    cscale(W, -g * K.iq[6]);
    a[3] = a[3] + spdot(row_slash(W, e0), vb);
  }
  {  // x = 2: orderings 201 (a4), 210 (a5)
    c4<T> U = row_prop(row_slash(ub, e2), kt + k2, mt);
    cscale(U, -g * K.iq[4]);
    const cx<T> t = spdot(row_slash(U, J01), vb);
    a[4] = a[4] + t;
    a[5] = a[5] - t;
    c4<T> r = row_slash(U, e0);
    c4<T> b = row_slash(ub, J02);
    cscale(b, T(-1));
    cadd(r, b);
    c4<T> W = row_prop(r, kt + k0 + k2, mt);
    cscale(W, -g * K.iq[5]);
    a[4] = a[4] + spdot(row_slash(W, e1), vb);
    r = row_slash(U, e1);
    b = row_slash(ub, J12);
    cscale(b, T(-1));
    cadd(r, b);
    W = row_prop(r, kt + k1 + k2, mt);
    cscale(W, -g * K.iq[6]);
    a[5] = a[5] + spdot(row_slash(W, e0), vb);
  }
#pragma unroll
  for (int f = 0; f < 6; ++f) A[f] = times_i(a[f]) * g;
}

template <typename T>
ME_HD c4<T> lepton_current(const KinEE<T>& K, int hel, const Couplings& cp) {
  // vbar(e+) gamma^mu u(e-) with the photon propagator: (e Q_e / s) vbar gamma u
  c4<T> vb = dbar(spinor_v(K.pl[0], T(0), hel_of(hel, 0)));
  c4<T> u = spinor_u(K.pl[1], T(0), hel_of(hel, 1));
  c4<T> L = vcurrent(vb, u);
  cscale(L, -ee_of<T>(cp) * K.is);
  return L;
}

template <typename T>
ME_HD void amp_ee_uu(const KinEE<T>& K, int hel, const Couplings& cp, cx<T>* A) {
  c4<T> L = lepton_current<T>(K, hel, cp);
  c4<T> ub = dbar(spinor_u(K.pl[2], T(0), hel_of(hel, 2)));
  c4<T> v = spinor_v(K.pl[3], T(0), hel_of(hel, 3));
  const T equ = (T)(cp.ee * (2.0 / 3.0));
  A[0] = times_i(spdot(row_slash(ub, L), v)) * equ;
}

template <typename T>
ME_HD void amp_ee_uug(const KinEE<T>& K, int hel, const Couplings& cp, cx<T>* A) {
  c4<T> L = lepton_current<T>(K, hel, cp);
  c4<T> ub = dbar(spinor_u(K.pl[2], T(0), hel_of(hel, 2)));
  c4<T> v = spinor_v(K.pl[3], T(0), hel_of(hel, 3));
  c4<T> eps = polvec(K.pl[4], hel_of(hel, 4), true);
  const T g = gs_of<T>(cp);
  const T equ = (T)(cp.ee * (2.0 / 3.0));
  // gluon on the quark side: ubar (i g eps) i(Q1slash)/Q1^2, Q1 = p_u + p_g
  c4<T> u1 = row_prop(row_slash(ub, eps), K.pl[2] + K.pl[4], T(0));
  cscale(u1, -g * K.i1);
  // gluon on the antiquark side: i(-Q2slash)/Q2^2 (i g eps) v, Q2 = p_ubar + p_g
  c4<T> v1 = col_prop(K.pl[3] + K.pl[4], T(0), slash_col(eps, v));
  cscale(v1, -g * K.i2);
  cx<T> a = spdot(row_slash(u1, L), v) + spdot(row_slash(ub, L), v1);
  A[0] = times_i(a) * equ;
}

template <typename T>
ME_HD c4<T> light_current(const c4<T>& vbar_ub, const c4<T>& u_u, T inv, T g) {
  // (g/Q^2) vbar gamma u  (vertex i g gamma, propagator -i/Q^2)
  c4<T> J = vcurrent(vbar_ub, u_u);
  cscale(J, g * inv);
  return J;
}

template <typename T>
ME_HD void amp_uu_tt(const KinUU<T>& K, int hel, const Couplings& cp, cx<T>* A) {
  const T g = gs_of<T>(cp), mt = mt_of<T>(cp);
  c4<T> uu = spinor_u(K.pl[0], T(0), hel_of(hel, 0));
  c4<T> vbu = dbar(spinor_v(K.pl[1], T(0), hel_of(hel, 1)));
  c4<T> ub = dbar(spinor_u(K.pl[2], mt, hel_of(hel, 2)));
  c4<T> vt = spinor_v(K.pl[3], mt, hel_of(hel, 3));
  c4<T> Ju = light_current(vbu, uu, K.is, g);
  cx<T> d = times_i(spdot(row_slash(ub, Ju), vt)) * g;
  A[0] = d * T(0.5);
  A[1] = d * (T)(-1.0 / 6.0);
}

template <typename T>
ME_HD void amp_uu_ttg(const KinUU<T>& K, int hel, const Couplings& cp, cx<T>* A) {
  const T g = gs_of<T>(cp), mt = mt_of<T>(cp);
  c4<T> uu = spinor_u(K.pl[0], T(0), hel_of(hel, 0));
  c4<T> vbu = dbar(spinor_v(K.pl[1], T(0), hel_of(hel, 1)));
  c4<T> ub = dbar(spinor_u(K.pl[2], mt, hel_of(hel, 2)));
  c4<T> vt = spinor_v(K.pl[3], mt, hel_of(hel, 3));
  c4<T> eps = polvec(K.pl[4], hel_of(hel, 4), true);
  const r4<T>* q = K.q;
  // u-line current without emission
  c4<T> Ju = light_current(vbu, uu, K.is, g);
  // D1: gluon off the top: ubar (ig eps) S_F(q2+q4) (ig Ju) v
  c4<T> r1 = row_prop(row_slash(ub, eps), q[2] + q[4], mt);
  cscale(r1, -g * K.ia);
  cx<T> D1 = times_i(spdot(row_slash(r1, Ju), vt)) * g;
  // D2: gluon off the antitop: ubar (ig Ju) S_F(-(q3+q4)) (ig eps) v
  c4<T> c1 = col_prop(q[3] + q[4], mt, slash_col(eps, vt));
  cscale(c1, -g * K.ib);
  cx<T> D2 = times_i(spdot(row_slash(ub, Ju), c1)) * g;
  // D3: gluon off the incoming antiquark (row side of the light line)
  c4<T> r3 = row_prop(row_slash(vbu, eps), q[1] + q[4], T(0));
  cscale(r3, -g * K.ic);
  c4<T> J3 = light_current(r3, uu, K.is3, g);
  cx<T> D3 = times_i(spdot(row_slash(ub, J3), vt)) * g;
  // D4: gluon off the incoming quark (column side)
  c4<T> c4u = col_prop(q[0] + q[4], T(0), slash_col(eps, uu));
  cscale(c4u, -g * K.id);
  c4<T> J4 = light_current(vbu, c4u, K.is3, g);
  cx<T> D4 = times_i(spdot(row_slash(ub, J4), vt)) * g;
  // D5: three-gluon vertex joining the light current, the heavy current and the gluon
  c4<T> Jt = vcurrent(ub, vt);
  cscale(Jt, g * K.it);
  c4<T> W = vvv(Ju, Jt, -(q[0] + q[1]), -(q[2] + q[3]));
  cx<T> D5 = cdot(W, eps) * g;
  const T h = T(0.5), hn = (T)(-1.0 / 6.0);
  cx<T> iD5 = times_i(D5);
  A[0] = (D1 + D4) * h - iD5 * h;
  A[1] = (D2 + D3) * h + iD5 * h;
  A[2] = (D1 + D2) * hn;
  A[3] = (D3 + D4) * hn;
}

// partial amplitudes of one helicity
template <int PID, typename T>
ME_HD void amplitude(const Kin<PID, T>& K, int hel, const Couplings& cp, cx<T>* A) {
  if constexpr (PID == P_EE_UU) amp_ee_uu<T>(K, hel, cp, A);
  else if constexpr (PID == P_EE_UUG) amp_ee_uug<T>(K, hel, cp, A);
  else if constexpr (PID == P_GG_TT) amp_tt2_fast<T>(K, hel, cp, A);
  else if constexpr (PID == P_GG_TTG) amp_tt3_fast<T>(K, hel, cp, A);
  else if constexpr (PID == P_GG_TTGG) amp_ttng<T, 4>(K, hel, cp, A);
  else if constexpr (PID == P_UU_TT) amp_uu_tt<T>(K, hel, cp, A);
  else amp_uu_ttg<T>(K, hel, cp, A);
}

// The live blocks of the processes whose kernels have closed forms, from single helicities
template <int PID, typename T, class F>
ME_HD void single_block(const Kin<PID, T>& K, int hb, const Couplings& cp, F&& consume) {
  for (int r = 0; r < 4; ++r) {
    if constexpr (PID == P_EE_UU || PID == P_EE_UUG) {
      if (r == 0 || r == 3) continue;  // u, ubar with equal helicities: zero
    }
    cx<T> A[Proc<PID>::NFLOW];
    amplitude<PID, T>(K, hb | (r << 2), cp, A);
    consume(r, A);
  }
}

}  // namespace me
