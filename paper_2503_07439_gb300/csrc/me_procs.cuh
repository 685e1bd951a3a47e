// Per-process colour-decomposed helicity amplitudes (device).
//
// Each block routine returns, for one helicity configuration after another, the partial
// amplitudes J_c of the process in its colour-flow basis, so that the colour-summed squared
// amplitude is J^dagger C J (Sec. 2.1, Eq. (born): |sum of diagrams|^2; Sec. 4.2:
// Born, real and counterterms are all tree-level amplitudes).
//
//  * t tbar + n gluons (gg->tt, gg->ttg, gg->ttgg): colour-ordered Berends-Giele
//    recursion.  Full amplitude M = sum_sigma (T^{a_s1} ... T^{a_sn})_{i_t j_tbar} A(sigma);
//    colour-ordered rules derived from the Feynman rules with [T^a,T^b] = i f^abc T^c:
//      gluon current  J(LR)  = -(g/Q^2) V3(J_L, J_R; -Q_L, -Q_R)
//                     J(LMR) = +(g^2/Q^2) [2(J_L.J_R) J_M - (J_L.J_M) J_R - (J_M.J_R) J_L]
//      quark line     U(s_1..s_k) = sum_j U(s_1..s_j) (i g Jslash(s_{j+1}..s_k)) i(Qslash+m)/(Q^2-m^2)
//      amplitude      A(s) = sum_j U(s_1..s_j) (i g Jslash(s_{j+1}..s_n)) v(tbar).
//  * e+e- -> u ubar (g): photon current from the leptons inserted on the quark line.
//  * u ubar -> t tbar (g): explicit diagrams, colour by Fierz onto a 2- (4-) element basis.
// Momenta: all-outgoing (q = -p for incoming legs).  Everything that does not depend
// on the helicities -- momenta in T and the reciprocal propagator denominators, whose
// invariants are formed in float64 to avoid cancellation -- is prepared once per event
// (prepare<PID,T>) and shared by all helicities; spinors and currents are in T.  The 2 -> 2 processes
// and e+e- -> u ubar g have closed forms; me_single.cuh has every process one helicity at a time, for
// the host check.
#pragma once
#include <type_traits>

#include "me_math.cuh"

namespace me {

enum ProcId : int {
  P_EE_UU = 0,
  P_EE_UUG = 1,
  P_GG_TT = 2,
  P_GG_TTG = 3,
  P_GG_TTGG = 4,
  P_UU_TT = 5,
  P_UU_TTG = 6,
  P_COUNT = 7
};

template <int PID> struct Proc;
template <> struct Proc<P_EE_UU> { static constexpr int NEXT = 4, NHEL = 16, NFLOW = 1; };
template <> struct Proc<P_EE_UUG> { static constexpr int NEXT = 5, NHEL = 32, NFLOW = 1; };
template <> struct Proc<P_GG_TT> { static constexpr int NEXT = 4, NHEL = 16, NFLOW = 2, NG = 2; };
template <> struct Proc<P_GG_TTG> { static constexpr int NEXT = 5, NHEL = 32, NFLOW = 6, NG = 3; };
template <> struct Proc<P_GG_TTGG> { static constexpr int NEXT = 6, NHEL = 64, NFLOW = 24, NG = 4; };
template <> struct Proc<P_UU_TT> { static constexpr int NEXT = 4, NHEL = 16, NFLOW = 2; };
template <> struct Proc<P_UU_TTG> { static constexpr int NEXT = 5, NHEL = 32, NFLOW = 4; };

// The couplings and the top mass; the float32 copies spare the float32 kernels a float64
// conversion (as dear as a float64 multiply-add) per thread and use.
struct Couplings {
  double gs;   // strong coupling g_s
  double ee;   // electromagnetic coupling e
  double mt;   // top mass
  float gsf, eef, mtf;
  Couplings() = default;
  __host__ __device__ Couplings(double g, double e, double m)
      : gs(g), ee(e), mt(m), gsf((float)g), eef((float)e), mtf((float)m) {}
};
// The same with both couplings at 1.  A tree amplitude is a fixed product of couplings times a
// function of the momenta, so the kernels evaluate the function and multiply its square by
// the couplings in float64 (tree_coupling): a float32 coupling, off by up to 3e-8, would
// shift every matrix element by up to eight times that, and the subtraction would not
// cancel the shift against the float64 counterterms.
ME_HD Couplings unit_couplings(const Couplings& c) {
  Couplings u = c;
  u.gs = u.ee = 1.0;
  u.gsf = u.eef = 1.0f;
  return u;
}
template <typename T> ME_HD T gs_of(const Couplings& c) { return (T)c.gs; }
template <> ME_HD float gs_of<float>(const Couplings& c) { return c.gsf; }
template <typename T> ME_HD T ee_of(const Couplings& c) { return (T)c.ee; }
template <> ME_HD float ee_of<float>(const Couplings& c) { return c.eef; }
template <typename T> ME_HD T mt_of(const Couplings& c) { return (T)c.mt; }
template <> ME_HD float mt_of<float>(const Couplings& c) { return c.mtf; }

// the couplings of a process's tree |M|^2
ME_HD double tree_coupling(int pid, const Couplings& c) {
  const double g2 = c.gs * c.gs, e4 = c.ee * c.ee * c.ee * c.ee;
  switch (pid) {
    case P_EE_UU: return e4;
    case P_EE_UUG: return e4 * g2;
    case P_GG_TT:
    case P_UU_TT: return g2 * g2;
    case P_GG_TTGG: return g2 * g2 * g2 * g2;
    default: return g2 * g2 * g2;
  }
}

ME_HD int hel_of(int hel, int leg) { return ((hel >> leg) & 1) ? 1 : -1; }

// ----------------------------------------------------------------------------
// Per-event kinematics of t tbar + NG gluons.  Gluon g (0..NG-1) is leg 0, 1, 4, 5.
// ig[S] = 1/Q_S^2 for a gluon subset S (bit mask, |S| >= 2), iq[S] = 1/((p_t+Q_S)^2-m^2).
template <typename T, int NG>
struct KinTT {
  r4<T> pl[6];          // physical external momenta (wavefunctions)
  r4<T> q[NG];          // outgoing gluon momenta
  T ig[1 << NG];
  T iq[1 << NG];
  wf_v<T> wg[NG];       // polarisation ingredients of the gluons (legs 0, 1, 4, 5)
  wf_q<T> wt, wtb;      // spinor ingredients of the top and, times g_s, of the antitop
  bool axis;            // beams exactly along +z (leg 0) and -z (leg 1)
};

ME_HD bool zero_bits(double x) {  // x == 0, off the float64 pipe
#ifdef __CUDA_ARCH__
  return (__double_as_longlong(x) << 1) == 0;
#else
  return x == 0.0;
#endif
}

template <typename T, int NG>
ME_HD KinTT<T, NG> prep_tt(const r4<double>* p, const Couplings& cp) {
  KinTT<T, NG> K;
  const int NEXT = NG + 2;
  for (int l = 0; l < NEXT; ++l) K.pl[l] = cast4<T>(p[l]);
  K.axis = zero_bits(p[0].x) && zero_bits(p[0].y) && zero_bits(p[1].x) && zero_bits(p[1].y) && K.pl[0].z > T(0) &&
           T(0) > K.pl[1].z;
  r4<double> q[NG];
  for (int i = 0; i < NG; ++i) {
    const int l = i < 2 ? i : i + 2;
    q[i] = l < 2 ? -p[l] : p[l];
    K.q[i] = l < 2 ? -K.pl[l] : K.pl[l];
    K.wg[i] = wf_vector(K.pl[l]);
  }
  K.wt = wf_quark(K.pl[2], mt_of<T>(cp));
  K.wtb = scaled(wf_quark(K.pl[3], mt_of<T>(cp)), gs_of<T>(cp));
  // The gluons are massless and the top on shell, so every subset invariant is a sum of
  // pairwise products (float64):  Q_S^2 = 2 sum_{i<j in S} q_i.q_j,
  // (p_t + Q_S)^2 - m^2 = 2 sum_{i in S} p_t.q_i + Q_S^2.
  double qq[NG][NG], tq[NG];
  for (int i = 0; i < NG; ++i) {
    tq[i] = mdot(p[2], q[i]);
    for (int j = i + 1; j < NG; ++j) qq[i][j] = mdot(q[i], q[j]);
  }
  for (int S = 1; S < (1 << NG); ++S) {
    double s2 = 0.0, st = 0.0;
    int cnt = 0;
    for (int i = 0; i < NG; ++i)
      if (S >> i & 1) {
        st += tq[i];
        ++cnt;
        for (int j = i + 1; j < NG; ++j)
          if (S >> j & 1) s2 += qq[i][j];
      }
    K.ig[S] = cnt >= 2 ? T(1) / (T)(2.0 * s2) : T(0);
    K.iq[S] = cnt <= NG - 1 ? T(1) / (T)(2.0 * (st + s2)) : T(0);
  }
  K.ig[0] = K.iq[0] = T(0);
  return K;
}

// ----------------------------------------------------------------------------
// Helicity blocks.  A block is one helicity configuration hb of every leg except the
// heavy pair (legs 2 and 3; their bits in hb are zero) together with the four (t, tbar)
// helicities hb | (r << 2), r = 0..3.  For t tbar + gluons the gluon currents depend on
// the gluon helicities only and the quark-line rows ubar(t) ... on the top helicity
// only, so a block builds the gluon currents once, the rows once per top helicity, and
// closes each row with both antitop spinors: the partial amplitudes of the four
// single-helicity evaluations, with the shared pieces computed once.
// consume(r, A) receives the partial amplitudes of heavy spins r.
//
// The blocks are bound by the float64 pipe where they run in float64 (2 lane operations per
// SM and cycle) and by instruction issue in float32, so what counts is the number of
// operations.  Five-real polarisations (pol), light-cone quark spins (wf_q), brackets of
// conserved currents without their vanishing terms, products e.J computed once and each
// gluon-pair bracket used by both currents it enters take a general g g -> t tbar g block from
// 7349 to 4737 operations and a g g -> t tbar g g block from 66751 to 49460 (28044 with the products,
// currents and colour sums shared as in tt4_block and s4_colour_sum); beams on the z axis
// take the former to about 3300.  GB300: 2^20 subtracted g g -> t tbar g points 5.55 -> 2.20 ms,
// 30011 in float64 1.385 -> 0.552 ms (counterterms and rescue included).

// g g -> t tbar g: the three-gluon currents F(012) = F(210), F(021) = F(120),
// F(102) = F(201) and the pair currents J(xy) are built once per block; per top spin the
// row R_s of ordering s collects ubar F(s), U(x) J(yz) and W(xy) e_z.
// consume(r, A) receives the partial amplitudes of heavy spins r without the factor i g.
// E0, E1: polarisations of the beam gluons, pol or axpol (on the axis the block takes about 1600
// multiply-adds instead of 2500).  spins: the top spins evaluated, bit ht.
template <typename T, class E0, class E1, class F>
ME_HD void tt3_block(const KinTT<T, 3>& K, const E0& e0, const E1& e1, const pol<T>& e2, const Couplings& cp, unsigned spins,
                     F&& consume) {
  constexpr bool PAIR = has_pair<E0, E1>::value;
  const T g = gs_of<T>(cp), mt = mt_of<T>(cp);
  const r4<T> k0 = K.q[0], k1 = K.q[1], k2 = K.q[2], kt = K.pl[2];
  const r4<T> k01 = k0 + k1, k02 = k0 + k2, k12 = k1 + k2;
  cx<T> e01, e02, e12;
  const c4<T> J01 = bracket(e0, k0, e1, k1, -g * K.ig[3], e01);
  const c4<T> J02 = bracket(e0, k0, e2, k2, -g * K.ig[5], e02);
  const c4<T> J12 = bracket(e1, k1, e2, k2, -g * K.ig[6], e12);
  const T c3 = -g * K.ig[7], c4g = g * g * K.ig[7];
  e01 = c4g * e01;
  e02 = c4g * e02;
  e12 = c4g * e12;
  // each bracket of a gluon with a pair current enters two of the three currents:
  // J(a|bc) = -J(a|cb)
  c4<T> F0 = czero<T>(), F2 = czero<T>(), B = czero<T>();
  bracket_acc(F0, e0, k0, J12, k12, c3, cdot(e0, J12));
  c4<T> F1 = cneg(F0);
  if constexpr (PAIR) {
    bracket_acc(B, e2, k2, J01, k01, c3, cdot(e2, J01));  // J(2|01)
    csub(F0, B);
    cadd(F2, B);
    B = czero<T>();
  }
  bracket_acc(B, e1, k1, J02, k02, c3, cdot(e1, J02));  // J(1|02)
  csub(F1, B);
  cadd(F2, B);
  if constexpr (PAIR) {
    quartic_acc(F0, e0, e1, e2, e02, e01, e12);
    quartic_acc(F1, e0, e2, e1, e01, e02, e12);
    quartic_acc(F2, e1, e0, e2, e12, e01, e02);
  } else {  // e01 = 0
    caxpy(F0, T(2) * e02, e1);
    caxpy(F0, -e12, e0);
    caxpy(F1, -e02, e1);
    caxpy(F1, -e12, e0);
    caxpy(F2, T(2) * e12, e0);
    caxpy(F2, -e02, e1);
  }
  const auto se0 = slashed(e0);
  const auto se1 = slashed(e1);
  const spol<T> se2 = slashed(e2);
  const sl4<T> sJ01 = slashed(J01), sJ02 = slashed(J02), sJ12 = slashed(J12);
  const sl4<T> sF0 = slashed(F0), sF1 = slashed(F1), sF2 = slashed(F2);
  const r4<T> Q0 = kt + k0, Q1 = kt + k1, Q2 = kt + k2;
  const prop4<T> P0 = scaled_prop(Q0, mt, -g * K.iq[1]), P1 = scaled_prop(Q1, mt, -g * K.iq[2]),
                 P2 = scaled_prop(Q2, mt, -g * K.iq[4]);
  const prop4<T> P01 = scaled_prop(kt + k01, mt, -g * K.iq[3]), P02 = scaled_prop(kt + k02, mt, -g * K.iq[5]),
                 P12 = scaled_prop(kt + k12, mt, -g * K.iq[6]);
#pragma unroll
  for (int ht = 0; ht < 2; ++ht) {
    if (!(spins >> ht & 1u)) continue;
    c4<T> R[6];
    R[0] = ubar_slash(K.wt, ht, sF0);  // orderings 012, 021, 102, 120, 201, 210
    R[1] = ubar_slash(K.wt, ht, sF1);
    R[2] = ubar_slash(K.wt, ht, sF2);
    R[3] = R[1];
    R[4] = R[2];
    R[5] = R[0];
    const c4<T> S02 = ubar_slash(K.wt, ht, sJ02), S12 = ubar_slash(K.wt, ht, sJ12);
    c4<T> S01 = czero<T>();
    if constexpr (PAIR) S01 = ubar_slash(K.wt, ht, sJ01);
    {  // first gluon 0: orderings 012, 021
      const c4<T> U = gluon_line(K.wt, ht, se0, P0);
      const c4<T> t = row_slash(U, sJ12);
      cadd(R[0], t);
      csub(R[1], t);
      c4<T> r = S01;
      row_slash_acc(r, U, se1);
      row_slash_acc(R[0], row_prop(r, P01), se2);
      r = S02;
      row_slash_acc(r, U, se2);
      row_slash_acc(R[1], row_prop(r, P02), se1);
    }
    {  // first gluon 1: orderings 102, 120
      const c4<T> U = gluon_line(K.wt, ht, se1, P1);
      const c4<T> t = row_slash(U, sJ02);
      cadd(R[2], t);
      csub(R[3], t);
      c4<T> r = cneg(S01);
      row_slash_acc(r, U, se0);
      row_slash_acc(R[2], row_prop(r, P01), se2);
      r = S12;
      row_slash_acc(r, U, se2);
      row_slash_acc(R[3], row_prop(r, P12), se0);
    }
    {  // first gluon 2: orderings 201, 210
      const c4<T> U = gluon_line(K.wt, ht, se2, P2);
      if constexpr (PAIR) {
        const c4<T> t = row_slash(U, sJ01);
        cadd(R[4], t);
        csub(R[5], t);
      }
      c4<T> r = cneg(S02);
      row_slash_acc(r, U, se0);
      row_slash_acc(R[4], row_prop(r, P02), se1);
      r = cneg(S12);
      row_slash_acc(r, U, se1);
      row_slash_acc(R[5], row_prop(r, P12), se0);
    }
#pragma unroll
    for (int hv = 0; hv < 2; ++hv) {
      cx<T> A[6];
#pragma unroll
      for (int f = 0; f < 6; ++f) A[f] = dot_v(R[f], K.wtb, hv);
      consume(ht | (hv << 1), A);
    }
  }
}

template <typename T, class F>
ME_HD void amp_tt3_block(const KinTT<T, 3>& K, int hb, const Couplings& cp, unsigned spins, F&& consume) {
  const pol<T> e2 = pol_of(K.wg[2], hel_of(hb, 4), true);
  if (K.axis) {
    // leg 0 (helicity + in every block) is -(0, 1, i, 0) / sqrt 2, leg 1 the same for
    // helicity - and (0, 1, -i, 0) / sqrt 2 for +
    const T r2 = T(0.70710678118654752440);
    const axpol<T, 1> e0{-r2};
    if (hel_of(hb, 1) < 0) tt3_block(K, e0, axpol<T, 1>{-r2}, e2, cp, spins, consume);
    else tt3_block(K, e0, axpol<T, -1>{r2}, e2, cp, spins, consume);
  } else {
    tt3_block(K, pol_of(K.wg[0], hel_of(hb, 0), false), pol_of(K.wg[1], hel_of(hb, 1), false), e2, cp, spins,
              consume);
  }
}

// ----------------------------------------------------------------------------
// e+(0) e-(1) -> u(2) ubar(3) [g(4)].  Photon exchange; charges Q_e = -1, Q_u = 2/3.
template <typename T>
struct KinEE {
  r4<T> pl[5];
  T is;      // 1/s of the photon
  T i1, i2;  // 1/(p_u+k)^2, 1/(p_ubar+k)^2 (real emission)
  T d[4];    // p0.p2, p0.p3, p1.p2, p1.p3 (real emission)
  T n1, n2;  // i1, i2 as they enter |M|^2 (ee_uug_block)
};

template <typename T, int NEXT>
ME_HD KinEE<T> prep_ee(const r4<double>* p) {
  KinEE<T> K;
  for (int l = 0; l < NEXT; ++l) K.pl[l] = cast4<T>(p[l]);
  const r4<double> Q = p[0] + p[1];
  K.is = T(1) / (T)mdot(Q, Q);
  K.i1 = K.i2 = T(0);
  if (NEXT == 5) {
    const r4<double> Q1 = p[2] + p[4], Q2 = p[3] + p[4];
    K.i1 = T(1) / (T)mdot(Q1, Q1);
    K.i2 = T(1) / (T)mdot(Q2, Q2);
    for (int i = 0; i < 4; ++i) K.d[i] = (T)mdot(p[i >> 1], p[2 + (i & 1)]);
    K.n1 = K.i1;
    K.n2 = K.i2;
    if constexpr (!std::is_same<T, float>::value) {
      cx<T> a[3], c[3];
      for (int l = 0; l < 3; ++l) chi_massless(K.pl[2 + l], a[l], c[l]);
      K.n1 = K.i1 * K.i1 * norm2(cmsb(a[0] * c[2], c[0], a[2]));
      K.n2 = K.i2 * K.i2 * norm2(cmsb(a[1] * c[2], c[1], a[2]));
    }
  }
  return K;
}

// e+e- -> u ubar g, one helicity block (gluon helicity fixed, both quark helicities) at unit
// couplings, colour-summed.  Every nonzero helicity amplitude is maximally helicity
// violating, |A|^2 = 8 (p_l.p_q)^2 / ((p0.p1) (p2.p4) (p3.p4)) up to couplings and charges,
// with l the lepton and q the quark of one helicity (Berends et al. 1981): block 0 (gluon
// helicity -) pairs the quarks with e-, block 1 with e+.
// A Feynman amplitude has 1 / (2 p2.p4) from a propagator, formed by cancellation from the
// momenta, and a numerator that goes like the angle, formed from the spinors: where the gluon
// is nearly collinear the two round differently.  In float64 the block keeps that form,
// |<24>|^2 / (2 p2.p4)^2 for 1 / (2 p2.p4), so that it stays the float64 value of the
// amplitude, to which float64 results are held where their inputs fix them; float32 takes the
// closed form as it is (99 % of the errors within 2.1e-7 instead of 6.9e-7).  65,536 subtracted points: 286 us with the helicity amplitudes, 187 us here.
// The products with 1 / (2 p2.p4) and 1 / (2 p3.p4) come first, as ratios without a dimension:
// the three reciprocal invariants alone, of order s^-3, would leave float32 from sqrt(s) = 1e7 on.
template <typename T>
ME_HD T ee_uug_block(const KinEE<T>& K, int b) {
  const T x = K.d[2 - 2 * b], y = K.d[3 - 2 * b];
  return T(512.0 / 9.0) * K.is * ((x * K.n1) * (x * K.n2) + (y * K.n1) * (y * K.n2));
}

// ----------------------------------------------------------------------------
// u(0) ubar(1) -> t(2) tbar(3) [g(4)].  Colour basis (i=t, j=tbar, k=u, l=ubar):
//   Born: e1 = d_ik d_lj, e2 = d_ij d_lk;  (T^b)_ij (T^b)_lk = (e1 - e2/N)/2.
//   Real: e1 = T^a_ik d_lj, e2 = d_ik T^a_lj, e3 = T^a_ij d_lk, e4 = d_ij T^a_lk.
template <typename T>
struct KinUU {
  r4<T> pl[5];
  r4<T> q[5];  // outgoing momenta
  T is;        // 1/(q0+q1)^2
  T ia, ib;    // top / antitop propagators with the gluon
  T ic, id;    // light-quark propagators with the gluon
  T is3, it;   // 1/(q0+q1+q4)^2, 1/(q2+q3)^2
  wf_q<T> wt, wtb;  // real emission: spinor ingredients of the top and the antitop,
  wf_v<T> wg;       // the gluon's polarisation,
  c2<T> rho, sg;    // and the light line: vbar(ubar, -) and u(u, +)
};

template <typename T, int NEXT>
ME_HD KinUU<T> prep_uu(const r4<double>* p, const Couplings& cp) {
  KinUU<T> K;
  r4<double> q[5];
  for (int l = 0; l < NEXT; ++l) {
    K.pl[l] = cast4<T>(p[l]);
    q[l] = l < 2 ? -p[l] : p[l];
    K.q[l] = l < 2 ? -K.pl[l] : K.pl[l];
  }
  K.ia = K.ib = K.ic = K.id = K.is3 = K.it = T(0);
  if constexpr (NEXT == 5 && std::is_same<T, float>::value) {
    // on-shell legs: every denominator from five products (float64)
    const double d01 = mdot(q[0], q[1]), d04 = mdot(q[0], q[4]), d14 = mdot(q[1], q[4]);
    K.is = T(0.5) / (T)d01;
    K.ia = T(0.5) / (T)mdot(q[2], q[4]);
    K.ib = T(0.5) / (T)mdot(q[3], q[4]);
    K.ic = T(0.5) / (T)d14;
    K.id = T(0.5) / (T)d04;
    K.is3 = K.it = T(0.5) / (T)(d01 + d04 + d14);
  } else {
    const double m2 = cp.mt * cp.mt;
    const r4<double> s01 = q[0] + q[1];
    K.is = T(1) / (T)mdot(s01, s01);
    if (NEXT == 5) {
      const r4<double> a = q[2] + q[4], b = q[3] + q[4], c = q[1] + q[4], d = q[0] + q[4];
      const r4<double> s3 = s01 + q[4], t = q[2] + q[3];
      K.ia = T(1) / (T)(mdot(a, a) - m2);
      K.ib = T(1) / (T)(mdot(b, b) - m2);
      K.ic = T(1) / (T)mdot(c, c);
      K.id = T(1) / (T)mdot(d, d);
      K.is3 = T(1) / (T)mdot(s3, s3);
      K.it = T(1) / (T)mdot(t, t);
    }
  }
  if (NEXT == 5) {
    K.wt = wf_quark(K.pl[2], mt_of<T>(cp));
    K.wtb = wf_quark(K.pl[3], mt_of<T>(cp));
    K.wg = wf_vector(K.pl[4]);
    chi_massless(K.pl[1], K.rho.a, K.rho.b);
    K.rho.a = conj(K.rho.a);
    K.rho.b = conj(K.rho.b);
    chi_massless(K.pl[0], K.sg.a, K.sg.b);
  }
  return K;
}

// u ubar -> t tbar g, one helicity block: the light line's helicities and the gluon's fixed,
// the four heavy spins open.  The light line enters by its spinors (line_X ... line_y):
//   d1, d2  gluon off the top, the antitop: heavy line with (rho, sigma),
//   d3, d4  gluon off the incoming ubar, u: (rho', sigma), (rho, sigma'),
//   w       three-gluon vertex, linear in the heavy current T: with both currents conserved,
//           2 [(k.e)(J.T) + (q4.J)(e.T) - (J.e)(q4.T)], k = p0 + p1.
// Flows (no factor i): A = (d1 + d4 - w)/2, (d2 + d3 + w)/2, -(d1 + d2)/6, -(d3 + d4)/6.
// 1500 operations per block against 7343 for four single helicities; 600,011 subtracted
// u ubar -> t tbar g points with cuts, whose float64 rescue is bound by the float64 pipe:
// 2088 -> 1271 us.
template <typename T, class F>
ME_HD void amp_uu_block(const KinUU<T>& K, int hb, const Couplings& cp, F&& consume) {
  const T g = gs_of<T>(cp), mt = mt_of<T>(cp);
  const pol<T> e = pol_of(K.wg, hel_of(hb, 4), true);
  const spol<T> se = slashed(e);
  const r4<T>* q = K.q;
  const c2<T> rho = K.rho, sg = K.sg;
  c2<T> rp, sp;  // rho', sigma': the emission's slash, then the massless propagator
  {
    const r4<T> Q = q[1] + q[4];
    const cx<T> o2 = cmsb(-se.z * rho.a, rho.b, se.d), o3 = cmsb(se.z * rho.b, rho.a, se.c);
    const T f = -g * K.ic, a = f * (Q.e - Q.z), b = f * (Q.e + Q.z);
    const cx<T> c{f * Q.x, -f * Q.y};
    rp.a = cmac(b * o2, o3, conj(c));
    rp.b = cmac(a * o3, o2, c);
  }
  {
    const r4<T> Q = q[0] + q[4];
    const cx<T> o0 = cmsb(-se.z * sg.a, se.c, sg.b), o1 = cmsb(se.z * sg.b, se.d, sg.a);
    const T f = g * K.id, a = f * (Q.e - Q.z), b = f * (Q.e + Q.z);
    const cx<T> c{f * Q.x, -f * Q.y};
    sp.a = cmac(b * o0, c, o1);
    sp.b = cmac(a * o1, conj(c), o0);
  }
  const T fu = T(2) * g * g * K.is, f3 = T(2) * g * g * K.is3, fw = T(2) * g * fu, it = K.it, ih = T(0.5) * it;
  // the light current (without its factor 2) slashed, and the vertex's vector times 1 / (q2 + q3)^2,
  // Z = (q4.J) e - (J.e) q4 (1 / (q2 + q3)^2 times the other propagator, of order s^-2, would
  // leave float32 from sqrt(s) = 1e10 on)
  const cx<T> ja = rho.b * sg.b, jb = rho.a * sg.a, jc = rho.b * sg.a, jd = rho.a * sg.b;
  const T qa = q[4].e - q[4].z, qb = q[4].e + q[4].z;
  const cx<T> qc{q[4].x, -q[4].y};
  const cx<T> qJ = ih * cmsb(cmsb(rmac(qa * jb, qb, ja), qc, jd), conj(qc), jc);
  const cx<T> eJ = ih * cmsb(cmsb(se.z * (ja - jb), se.c, jd), se.d, jc);
  const sl4<T> Z{rmac(-se.z * qJ, -qa, eJ), rmac(se.z * qJ, -qb, eJ), cmsb(qJ * se.c, eJ, qc),
                 cmsb(qJ * se.d, eJ, conj(qc))};
  const cx<T> ke = it * rdot(K.pl[0] + K.pl[1], e);
  const prop4<T> P1 = scaled_prop(q[2] + q[4], mt, -g * K.ia), P2 = scaled_prop(-(q[3] + q[4]), mt, -g * K.ib);
  cx<T> xs[2], xsp[2], yr[2], yrp[2], cx1[2], cy1[2];
#pragma unroll
  for (int hv = 0; hv < 2; ++hv) {
    const c4<T> c1 = col_prop(P2, slash_v(se, K.wtb, hv));
    cx1[hv] = line_x(c1, sg);
    cy1[hv] = line_y(c1, rho);
    xs[hv] = v_x(K.wtb, hv, sg);
    xsp[hv] = v_x(K.wtb, hv, sp);
    yr[hv] = v_y(K.wtb, hv, rho);
    yrp[hv] = v_y(K.wtb, hv, rp);
  }
#pragma unroll
  for (int ht = 0; ht < 2; ++ht) {
    const c4<T> r1 = row_prop(ubar_slash(K.wt, ht, se), P1);
    const cx<T> X1 = line_X(r1, rho), Y1 = line_Y(r1, sg);
    const cx<T> X = ubar_X(K.wt, ht, rho), Xp = ubar_X(K.wt, ht, rp);
    const cx<T> Y = ubar_Y(K.wt, ht, sg), Yp = ubar_Y(K.wt, ht, sp);
    const c4<T> z = ubar_slash(K.wt, ht, Z);
#pragma unroll
    for (int hv = 0; hv < 2; ++hv) {
      const cx<T> d1 = fu * cmac(X1 * xs[hv], Y1, yr[hv]), d2 = fu * cmac(X * cx1[hv], Y, cy1[hv]);
      const cx<T> d3 = f3 * cmac(Xp * xs[hv], Y, yrp[hv]), d4 = f3 * cmac(X * xsp[hv], Yp, yr[hv]);
      const cx<T> w = fw * cmac(dot_v(z, K.wtb, hv), ke, cmac(X * xs[hv], Y, yr[hv]));
      const T h = T(0.5), hn = (T)(-1.0 / 6.0);
      const cx<T> A[4] = {h * (d1 + d4 - w), h * (d2 + d3 + w), hn * (d1 + d2), hn * (d3 + d4)};
      consume(ht | (hv << 1), A);
    }
  }
}

// ----------------------------------------------------------------------------
template <int PID, typename T> struct KinOf;
template <typename T> struct KinOf<P_EE_UU, T> { using type = KinEE<T>; };
template <typename T> struct KinOf<P_EE_UUG, T> { using type = KinEE<T>; };
template <typename T> struct KinOf<P_GG_TT, T> { using type = KinTT<T, 2>; };
template <typename T> struct KinOf<P_GG_TTG, T> { using type = KinTT<T, 3>; };
template <typename T> struct KinOf<P_GG_TTGG, T> { using type = KinTT<T, 4>; };
template <typename T> struct KinOf<P_UU_TT, T> { using type = KinUU<T>; };
template <typename T> struct KinOf<P_UU_TTG, T> { using type = KinUU<T>; };
template <int PID, typename T> using Kin = typename KinOf<PID, T>::type;

// helicity-independent per-event kinematics
template <int PID, typename T>
ME_HD Kin<PID, T> prepare(const r4<double>* p, const Couplings& cp) {
  if constexpr (PID == P_EE_UU) return prep_ee<T, 4>(p);
  else if constexpr (PID == P_EE_UUG) return prep_ee<T, 5>(p);
  else if constexpr (PID == P_GG_TT) return prep_tt<T, 2>(p, cp);
  else if constexpr (PID == P_GG_TTG) return prep_tt<T, 3>(p, cp);
  else if constexpr (PID == P_GG_TTGG) return prep_tt<T, 4>(p, cp);
  else if constexpr (PID == P_UU_TT) return prep_uu<T, 4>(p, cp);
  else return prep_uu<T, 5>(p, cp);
}

// The four gluons of a block: beam gluons of type E0, E1 (pol or axpol), outgoing ones pol.  The
// gluon index is a constant wherever these are called in unrolled code.
template <typename T, class E0, class E1>
struct FourGluons {
  E0 e0;
  E1 e1;
  pol<T> e2, e3;
  ME_HD cx<T> dot(int i, const c4<T>& J) const {
    return i == 0 ? cdot(e0, J) : i == 1 ? cdot(e1, J) : i == 2 ? cdot(e2, J) : cdot(e3, J);
  }
  ME_HD void add(c4<T>& acc, cx<T> w, int i) const {
    if (i == 0) caxpy(acc, w, e0);
    else if (i == 1) caxpy(acc, w, e1);
    else if (i == 2) caxpy(acc, w, e2);
    else caxpy(acc, w, e3);
  }
  ME_HD void current(c4<T>& acc, int i, const r4<T>& q, const c4<T>& J, const r4<T>& Q, T s, cx<T> eJ) const {
    if (i == 0) bracket_acc(acc, e0, q, J, Q, s, eJ);
    else if (i == 1) bracket_acc(acc, e1, q, J, Q, s, eJ);
    else if (i == 2) bracket_acc(acc, e2, q, J, Q, s, eJ);
    else bracket_acc(acc, e3, q, J, Q, s, eJ);
  }
  ME_HD c4<T> pair(int x, int y, const r4<T>* q, T s, cx<T>& xy) const {  // x < y
    return x == 0 ? (y == 1 ? bracket(e0, q[0], e1, q[1], s, xy) : y == 2 ? bracket(e0, q[0], e2, q[2], s, xy)
                                                                          : bracket(e0, q[0], e3, q[3], s, xy))
           : x == 1 ? (y == 2 ? bracket(e1, q[1], e2, q[2], s, xy) : bracket(e1, q[1], e3, q[3], s, xy))
                    : bracket(e2, q[2], e3, q[3], s, xy);
  }
  ME_HD void row(c4<T>& acc, const c4<T>& r, int i) const {
    if (i == 0) row_slash_acc(acc, r, slashed(e0));
    else if (i == 1) row_slash_acc(acc, r, slashed(e1));
    else if (i == 2) row_slash_acc(acc, r, slashed(e2));
    else row_slash_acc(acc, r, slashed(e3));
  }
  ME_HD c4<T> line(const wf_q<T>& w, int h, int i, const prop4<T>& P) const {
    return i == 0 ? gluon_line(w, h, slashed(e0), P) : i == 1 ? gluon_line(w, h, slashed(e1), P)
           : i == 2 ? gluon_line(w, h, slashed(e2), P) : gluon_line(w, h, slashed(e3), P);
  }
};

// g g -> t tbar g g.  The ordered gluon currents are built once per block with the
// reflection identities: 6 pairs J(xy), x < y; 12 triples J(xyz) (one of each
// reversed pair), for each left-out gluon from three brackets and J(xyz) + J(yxz) + J(xzy) = 0;
// 6 quadruples J(0xyz), which give the others by sums.  Per top spin, the quark line
// is extended ordering by ordering, U(w) -> U(wx) -> U(wxy), and the row of ordering
// wxyz is ubar J(wxyz) + U(w) J(xyz) + U(wx) J(yz) + U(wxy) e_z; a product of U(w) or U(wx)
// with a current serves the ordering that has it reversed too.  Orderings are
// numbered lexicographically, as in amp_ttng.
template <typename T, class G, class F>
ME_HD void tt4_block(const KinTT<T, 4>& K, const G& e, const Couplings& cp, F&& consume) {
  const T g = gs_of<T>(cp), mt = mt_of<T>(cp);
  const r4<T>* q = K.q;
  // pair currents, index pidx(x, y) for x < y, and the products e_i . e_j, e_i . J(xy)
  c4<T> J2[6];
  cx<T> ee[6], eJ[4][6];
  auto pidx = [](int x, int y) { return x == 0 ? y - 1 : (x == 1 ? y + 1 : 5); };
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = x + 1; y < 4; ++y) {
      J2[pidx(x, y)] = e.pair(x, y, q, -g * K.ig[(1 << x) | (1 << y)], ee[pidx(x, y)]);
    }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = x + 1; y < 4; ++y)
        if (i != x && i != y) eJ[i][pidx(x, y)] = e.dot(i, J2[pidx(x, y)]);
  auto e2 = [&](int x, int y) { return ee[x < y ? pidx(x, y) : pidx(y, x)]; };
  auto ej = [&](int i, int x, int y) {  // e_i . J(xy), J(yx) = -J(xy)
    return x < y ? eJ[i][pidx(x, y)] : -eJ[i][pidx(y, x)];
  };
  auto j2 = [&](int x, int y) {  // ordered pair current
    return x < y ? J2[pidx(x, y)] : cneg(J2[pidx(y, x)]);
  };
  // triple currents J(xyz) for x < z (J(zyx) = J(xyz)); index tidx = 3 * (missing gluon) + (middle slot)
  c4<T> J3[12];
  auto tidx = [](int x, int y, int z) {
    const int miss = 6 - x - y - z;
    // the three gluons of the triple in increasing order a < b < c; middle y in {a, b, c}
    const int a = miss == 0 ? 1 : 0;
    const int c = miss == 3 ? 2 : 3;
    return 3 * miss + (y == a ? 0 : (y == c ? 2 : 1));
  };
#pragma unroll
  for (int w = 0; w < 4; ++w) {  // x < y < z: the gluons other than w
    const int x = w == 0 ? 1 : 0, y = w <= 1 ? 2 : 1, z = w <= 2 ? 3 : 2;
    const T c3 = -g * K.ig[15 ^ (1 << w)], c4g = g * g * K.ig[15 ^ (1 << w)];
    const cx<T> exy = c4g * e2(x, y), eyz = c4g * e2(y, z), exz = c4g * e2(x, z);
    c4<T> Jy = czero<T>(), Jx = czero<T>(), B = czero<T>();
    e.current(Jy, x, q[x], J2[pidx(y, z)], q[y] + q[z], c3, ej(x, y, z));  // x (yz)
    e.current(Jx, y, q[y], J2[pidx(x, z)], q[x] + q[z], c3, ej(y, x, z));  // y (xz)
    e.current(B, z, q[z], J2[pidx(x, y)], q[x] + q[y], c3, ej(z, x, y));   // z (xy)
    csub(Jy, B);
    cadd(Jx, B);
    e.add(Jy, T(2) * exz, y);
    e.add(Jy, -exy, z);
    e.add(Jy, -eyz, x);
    e.add(Jx, T(2) * eyz, x);
    e.add(Jx, -exy, z);
    e.add(Jx, -exz, y);
    J3[tidx(x, y, z)] = Jy;
    J3[tidx(y, x, z)] = Jx;
    cadd(Jx, Jy);
    J3[tidx(x, z, y)] = cneg(Jx);
  }
  auto j3 = [&](int x, int y, int z) { return J3[tidx(x, y, z)]; };
  // quadruple currents J(0xyz)
  c4<T> J4[6];
  auto q0 = [](int x, int y) { return 2 * (x - 1) + (y > (x == 1 ? 2 : 1) ? 1 : 0); };
#pragma unroll
  for (int x = 1; x < 4; ++x)
#pragma unroll
    for (int y = 1; y < 4; ++y) {
      if (y == x) continue;
      const int w = 0, z = 6 - x - y;
      const T c3 = -g * K.ig[15], c4g = g * g * K.ig[15];
      const r4<T> qwx = q[w] + q[x], qyz = q[y] + q[z];
      const c4<T> Jxyz = j3(x, y, z), Jwxy = j3(w, x, y), Jwx = j2(w, x), Jxy = j2(x, y), Jyz = j2(y, z);
      c4<T> J = czero<T>();
      e.current(J, w, q[w], Jxyz, q[x] + qyz, c3, e.dot(w, Jxyz));
      bracket_acc(J, Jwx, qwx, Jyz, qyz, c3);
      e.current(J, z, q[z], Jwxy, qwx + q[y], -c3, e.dot(z, Jwxy));
      // 2 (L.R) M - (L.M) R - (M.R) L for (e_w, e_x, J_yz), (e_w, J_xy, e_z), (J_wx, e_y, e_z),
      // collected by vector
      e.add(J, c4g * (T(2) * ej(w, y, z)), x);
      e.add(J, c4g * (T(2) * ej(z, w, x)), y);
      e.add(J, -c4g * (ej(x, y, z) + ej(z, x, y)), w);
      e.add(J, -c4g * (ej(w, x, y) + ej(y, w, x)), z);
      caxpy(J, -c4g * e2(w, x), Jyz);
      caxpy(J, T(2) * c4g * e2(w, z), Jxy);
      caxpy(J, -c4g * e2(y, z), Jwx);
      J4[q0(x, y)] = J;
    }
  // the others by reflection and decoupling: 0 second in x 0 y z, with J(x 0 y z) + J(0 x y z)
  // + J(0 y x z) + J(0 y z x) = 0
  auto quad = [&](int w, int x, int y) {
    const int z = 6 - w - x - y;
    if (w == 0) return J4[q0(x, y)];
    if (z == 0) return cneg(J4[q0(y, x)]);
    const bool second = x == 0;
    const int a = second ? w : z, b = second ? y : x, c = second ? z : w;
    c4<T> J = J4[q0(a, b)];
    cadd(J, J4[q0(b, a)]);
    cadd(J, J4[q0(b, c)]);
    return second ? cneg(J) : J;
  };
  const r4<T> kt = K.pl[2];
#pragma unroll 1
  for (int ht = 0; ht < 2; ++ht) {
    cx<T> A[2][24];
    int f = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const c4<T> U1 = e.line(K.wt, ht, w, scaled_prop(kt + q[w], mt, -g * K.iq[1 << w]));
      // U(w) J(xy), x < y, and U(w) J(xyz) by its middle gluon y
      c4<T> P[6], Q[4];
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = x + 1; y < 4; ++y)
          if (x != w && y != w) {
            P[pidx(x, y)] = row_slash(U1, slashed(J2[pidx(x, y)]));
            Q[6 - w - x - y] = row_slash(U1, slashed(j3(x, 6 - w - x - y, y)));
          }
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        if (x == w) continue;
        c4<T> r2 = ubar_slash(K.wt, ht, slashed(j2(w, x)));
        e.row(r2, U1, x);
        const c4<T> U2 = row_prop(r2, scaled_prop(kt + q[w] + q[x], mt, -g * K.iq[(1 << w) | (1 << x)]));
        c4<T> D = czero<T>();  // U(wx) J(yz), y < z
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          if (y == w || y == x) continue;
          const int z = 6 - w - x - y;
          if (y < z) D = row_slash(U2, slashed(J2[pidx(y, z)]));
          c4<T> r3 = x < y ? P[pidx(x, y)] : cneg(P[pidx(y, x)]);
          ubar_slash_acc(r3, K.wt, ht, slashed(j3(w, x, y)));
          e.row(r3, U2, y);
          const c4<T> U3 =
              row_prop(r3, scaled_prop(kt + q[w] + q[x] + q[y], mt, -g * K.iq[(1 << w) | (1 << x) | (1 << y)]));
          c4<T> R = Q[y];
          if (y < z) cadd(R, D);
          else csub(R, D);
          ubar_slash_acc(R, K.wt, ht, slashed(quad(w, x, y)));
          e.row(R, U3, z);
#pragma unroll
          for (int hv = 0; hv < 2; ++hv) A[hv][f] = dot_v(R, K.wtb, hv);
          ++f;
        }
      }
    }
#pragma unroll
    for (int hv = 0; hv < 2; ++hv) consume(ht | (hv << 1), A[hv]);
  }
}
template <typename T, class F>
ME_HD void amp_tt4_block(const KinTT<T, 4>& K, int hb, const Couplings& cp, F&& consume) {
  const pol<T> e2 = pol_of(K.wg[2], hel_of(hb, 4), true), e3 = pol_of(K.wg[3], hel_of(hb, 5), true);
  if (K.axis) {  // as amp_tt3_block
    const T r2 = T(0.70710678118654752440);
    using A = axpol<T, 1>;
    using B = axpol<T, -1>;
    if (hel_of(hb, 1) < 0) tt4_block(K, FourGluons<T, A, A>{{-r2}, {-r2}, e2, e3}, cp, consume);
    else tt4_block(K, FourGluons<T, A, B>{{-r2}, {r2}, e2, e3}, cp, consume);
  } else {
    tt4_block(K, FourGluons<T, pol<T>, pol<T>>{pol_of(K.wg[0], hel_of(hb, 0), false), pol_of(K.wg[1], hel_of(hb, 1), false), e2, e3},
              cp, consume);
  }
}

// Colour sum of the 24 orderings of four gluons.  Relabelling the gluons changes no colour
// factor, and l -> l ^ v, v = 0 .. 3, is a group of relabellings: in the sums
//   S_k[a] = sum_v (-1)^|k & v| J(ordering v, v ^ x, v ^ y, v ^ z),
// a numbering the arrangements xyz of 1, 2, 3 lexicographically, the matrix falls into one
// 6 x 6 block for each k.  Nor does reversing an ordering, which takes S_k[a] to
// (-1)^|k & z| S_k[a]: for k > 0 the two arrangements with sign + couple only to each other
// and the four with - to each other.  That leaves 21 + 3 (3 + 10) coefficients (off-diagonal
// ones doubled) and 264 operations, where the triangle of the 24 x 24 matrix takes 648.
constexpr int S4_COEF = 60;
// gluon i = 0, 1, 2 of arrangement a
__host__ __device__ constexpr int s4_at(int a, int i) {
  const int x = 1 + (a >> 1), lo = x == 1 ? 2 : 1, hi = x == 3 ? 2 : 3;
  return i == 0 ? x : (i == 1) == ((a & 1) == 0) ? lo : hi;
}
// flow number (lexicographic) of the ordering v, v ^ x, v ^ y, v ^ z of arrangement a
__host__ __device__ constexpr int s4_flow(int v, int a) {
  const int w[4] = {v, v ^ s4_at(a, 0), v ^ s4_at(a, 1), v ^ s4_at(a, 2)};
  int f = 0;
  for (int i = 0; i < 3; ++i) {
    int smaller = 0;
    for (int j = i + 1; j < 4; ++j) smaller += w[j] < w[i];
    f = f * (4 - i) + smaller;
  }
  return f;
}
// 0 if (-1)^|k & z| of arrangement a is +, 1 if -
__host__ __device__ constexpr int s4_parity(int k, int a) {
  const int z = k & s4_at(a, 2);
  return (z ^ (z >> 1)) & 1;
}
// J(v, a): the amplitude of the ordering v, v ^ x, v ^ y, v ^ z
template <typename T, class A>
ME_HD T s4_colour_sum(const T* coef, const A& J) {
  cx<T> S[4][6];
#pragma unroll
  for (int a = 0; a < 6; ++a) {
    const cx<T> j0 = J(0, a), j1 = J(1, a), j2 = J(2, a), j3 = J(3, a);
    const cx<T> p = j0 + j1, m = j0 - j1, q = j2 + j3, r = j2 - j3;
    S[0][a] = p + q;
    S[1][a] = m + r;
    S[2][a] = p - q;
    S[3][a] = m - r;
  }
  T s = T(0);
  int i = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      cx<T> z{T(0), T(0)};
#pragma unroll
      for (int b = a; b < 6; ++b)
        if (s4_parity(k, a) == s4_parity(k, b)) z = rmac(z, coef[i++], S[k][b]);
      s += S[k][a].re * z.re + S[k][a].im * z.im;
    }
  return s;
}
// the coefficients from the 24 x 24 matrix C; false if C lacks the symmetry
inline bool s4_coefficients(const double* C, double* coef) {
  auto c = [&](int v, int a, int u, int b) { return C[s4_flow(v, a) * 24 + s4_flow(u, b)]; };
  int i = 0;
  for (int k = 0; k < 4; ++k)
    for (int a = 0; a < 6; ++a)
      for (int b = a; b < 6; ++b) {
        double t = 0;
        for (int u = 0; u < 4; ++u) {
          for (int v = 0; v < 4; ++v)
            if (std::abs(c(v, a, v ^ u, b) - c(0, a, u, b)) > 1e-12) return false;
          const int q = k & u;
          t += ((q ^ (q >> 1)) & 1) ? -c(0, a, u, b) : c(0, a, u, b);
        }
        if (s4_parity(k, a) == s4_parity(k, b)) coef[i++] = (a == b ? 0.25 : 0.5) * t;
        else if (std::abs(t) > 1e-12) return false;
      }
  return i == S4_COEF;
}

// Helicity blocks of one member of each flipped pair (leg 0 at +): NHEL / 8 blocks;
// block b sets legs 1, 4, 5 from the bits of b.
template <int PID> __host__ __device__ constexpr int n_blocks() { return Proc<PID>::NHEL / 8; }
ME_HD int block_hel(int b) { return 1 | ((b & 1) << 1) | ((b >> 1) << 4); }

// A massless fermion pair coupled through a vector current has opposite helicities
// (chirality is conserved at the vertex; the wrong-chirality spinor components are
// exactly zero): with legs 0, 1 such a pair (e+e-, u ubar), the blocks with leg 1 at +
// vanish identically and are skipped, and for e+e- -> u ubar (g) the heavy-pair slots
// (legs 2, 3 = u, ubar) with equal helicities vanish too.
template <int PID> __host__ __device__ constexpr bool massless_initial_pair() {
  return PID == P_EE_UU || PID == P_EE_UUG || PID == P_UU_TT || PID == P_UU_TTG;
}
template <int PID> __host__ __device__ constexpr int n_live_blocks() {
  return massless_initial_pair<PID>() ? n_blocks<PID>() / 2 : n_blocks<PID>();
}
template <int PID> ME_HD int live_block_hel(int i) { return block_hel(massless_initial_pair<PID>() ? 2 * i : i); }

// Partial amplitudes of the four helicities hb | (r << 2), of g g -> t tbar g those whose top spin
// r & 1 is among `spins`.  (e+e- -> u ubar g has ee_uug_block, the 2 -> 2 processes closed_sum.)
template <int PID, typename T, class F>
ME_HD void amplitude_block(const Kin<PID, T>& K, int hb, const Couplings& cp, F&& consume, unsigned spins = 3u) {
  static_assert(PID == P_GG_TTG || PID == P_GG_TTGG || PID == P_UU_TTG, "processes with block routines");
  if constexpr (PID == P_GG_TTG) amp_tt3_block<T>(K, hb, cp, spins, consume);
  else if constexpr (PID == P_GG_TTGG) amp_tt4_block<T>(K, hb, cp, consume);
  else amp_uu_block<T>(K, hb, cp, consume);
}

// ----------------------------------------------------------------------------
// Helicity- and colour-summed 2 -> 2 Borns in closed form.  With the massless beams p0, p1,
// the quark p2 of mass m, tau_i = (p_i.p2) / (p0.p1) and rho = 4 m^2 / s:
//   u ubar -> t tbar:  sum = 16 g^4 (tau_0^2 + tau_1^2 + rho / 2)   (one colour structure),
//   e+e- -> u ubar:    sum = 24 e^4 Q_u^2 (tau_0^2 + tau_1^2),
//   g g -> t tbar (Combridge 1979, by colour flow): the two orderings obey
//     tau_0 A(01) = tau_1 A(10) =: X with sum |X|^2 = 8 g^4 tau_0 tau_1 F,
//     F = tau_0^2 + tau_1^2 + rho - rho^2 / (4 tau_0 tau_1),
//   so for any symmetric colour matrix M
//     sum J^T M J = 8 g^4 F (M_00 tau_1 / tau_0 + 2 M_01 + M_11 tau_0 / tau_1);
//   with one gluon polarised along a transverse unit vector e (either gluon: the value is
//   symmetric), sum |X|^2 = 4 g^4 (tau_0 tau_1 F + rho (2 (e.p2)^2 / s - q)),
//   q = tau_0 tau_1 - rho / 4 = pt^2 / s.
// They take some 30 operations where the helicity amplitudes take 1400 to 3000, and stay
// accurate at small tau; all terms but rho^2 are positive.
template <typename T>
struct Inv22 {
  T c, t0, t1, rho;  // p0.p1, tau_0, tau_1, rho
};
template <typename T>
ME_HD Inv22<T> inv22(const r4<double>* p, T m) {  // the products in float64
  Inv22<T> k;
  k.c = (T)mdot(p[0], p[1]);
  const T ic = T(1) / k.c;
  k.t0 = (T)mdot(p[0], p[2]) * ic;
  k.t1 = (T)mdot(p[1], p[2]) * ic;
  k.rho = T(2) * m * m * ic;
  return k;
}
// u ubar -> t tbar and e+e- -> u ubar: the sum over everything but the couplings and colour
template <typename T>
ME_HD T born_qq(const Inv22<T>& k) {
  return k.t0 * k.t0 + k.t1 * k.t1 + T(0.5) * k.rho;
}
// g g -> t tbar: sum J^T M J = f (M_00 r0 + 2 M_01 + M_11 r1)
template <typename T>
struct BornGG {
  T f, r0, r1;
};
template <typename T>
ME_HD BornGG<T> born_gg(const Inv22<T>& k, const Couplings& cp) {
  const T i01 = T(1) / (k.t0 * k.t1), a = k.t0 * k.t0, b = k.t1 * k.t1;
  const T g2 = gs_of<T>(cp) * gs_of<T>(cp);
  const T F = a + b + k.rho * (T(1) - T(0.25) * k.rho * i01);
  return BornGG<T>{T(8) * g2 * g2 * F, b * i01, a * i01};
}
constexpr double GG_C00 = 16.0 / 3.0, GG_C01 = -2.0 / 3.0;  // colour matrix of g g -> t tbar
template <typename T>
ME_HD T born_gg_colour(const BornGG<T>& b) {  // M = C
  return b.f * (T(GG_C00) * (b.r0 + b.r1) + T(2.0 * GG_C01));
}
// the same with one gluon polarised along e, ep2 = (e.p2)^2 / (p0.p1) (either gluon)
template <typename T>
ME_HD T born_gg_polarised(const Inv22<T>& k, const BornGG<T>& b, T ep2, const Couplings& cp) {
  const T g2 = gs_of<T>(cp) * gs_of<T>(cp), t01 = k.t0 * k.t1;
  const T col = T(0.5 * GG_C00) * (b.r0 + b.r1) + T(GG_C01);
  return col * (b.f + T(8) * g2 * g2 * k.rho * (ep2 - (t01 - T(0.25) * k.rho)) / t01);
}
// (sum J^T M J) / f for a symmetric matrix M (row-major 2 x 2)
template <typename T>
ME_HD T born_gg_form(const BornGG<T>& b, const T* M) {
  return M[0] * b.r0 + T(2) * M[1] + M[3] * b.r1;
}
// u ubar -> t tbar with the matrix M: its amplitude in the basis (d_ik d_lj, d_ij d_lk) is
// proportional to (1/2, -1/6), `sum` is the plain Born / 2
template <typename T>
ME_HD T born_uu_matrix(T sum, const T* M) {
  return sum * (T(0.25) * M[0] - T(1.0 / 12.0) * (M[1] + M[2]) + T(1.0 / 36.0) * M[3]);
}

// Processes whose whole tree is one of these
template <int PID> __host__ __device__ constexpr bool closed_tree() {
  return PID == P_EE_UU || PID == P_GG_TT || PID == P_UU_TT;
}
// The on-shell momentum that the helicity spinors of (E, p) stand for: E + |p| and the
// direction are kept, E - |p| becomes m^2 / (E + |p|).
ME_HD r4<double> on_shell(const r4<double>& p, double m) {
  const double a = msqrt(p.x * p.x + p.y * p.y + p.z * p.z), wp = p.e + a, wm = m * m / wp;
  const double f = a > 0.0 ? 0.5 * (wp - wm) / a : 0.0;
  return r4<double>{0.5 * (wp + wm), f * p.x, f * p.y, f * p.z};
}
// |M|^2 of one of them, summed over helicities and colours.  The quark pairs use the traces
// of both lines, [(p0.p2)(p1.p3) + (p0.p3)(p1.p2) + m^2 p0.p1] / (p0.p1)^2 for born_qq, which
// hold for momenta that do not add up exactly, as the sum over helicity amplitudes does; in
// float64 the final momenta are put on shell as its spinors are (a generator that boosts
// strongly leaves both off by 1e-11 here and there).
template <int PID, typename T>
ME_HD T closed_sum(const r4<double>* p, const Couplings& cp) {
  if constexpr (PID == P_GG_TT) {
    return born_gg_colour(born_gg(inv22<T>(p, mt_of<T>(cp)), cp));
  } else {
    const T m = PID == P_EE_UU ? T(0) : mt_of<T>(cp);
    const T c = (T)mdot(p[0], p[1]), ic = T(1) / c;
    r4<double> p2 = p[2], p3 = p[3];
    if constexpr (!std::is_same<T, float>::value) {
      p2 = on_shell(p2, PID == P_EE_UU ? 0.0 : cp.mt);
      p3 = on_shell(p3, PID == P_EE_UU ? 0.0 : cp.mt);
    }
    const T a = (T)mdot(p[0], p2) * ic, b = (T)mdot(p[1], p3) * ic;
    const T d = (T)mdot(p[0], p3) * ic, e = (T)mdot(p[1], p2) * ic;
    const T q = a * b + d * e + m * m * ic;
    if constexpr (PID == P_EE_UU) {
      const T e2 = ee_of<T>(cp) * ee_of<T>(cp);
      return T(24.0 * 4.0 / 9.0) * e2 * e2 * q;
    } else {
      const T g2 = gs_of<T>(cp) * gs_of<T>(cp);
      return T(16) * g2 * g2 * q;
    }
  }
}

}  // namespace me
