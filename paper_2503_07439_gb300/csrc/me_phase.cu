// Flat phase-space points generated on the device: the multi-event input (Sec. 4.4,
// step 1) produced where the matrix elements consume it, instead of on the host.
//
//  * Counter-based random numbers: Philox4x32-10 (Salmon, Moraes, Dror and Shaw, "Parallel
//    random numbers: as easy as 1, 2, 3", SC'11), written here from that definition.
//    Counter (point index lo, point index hi, stream, block), key (seed lo, seed hi).
//    Block b of point i gives the uniforms 2b and 2b+1 as 53-bit doubles in (0, 1):
//    ((w0 >> 5) 2^26 + (w1 >> 6) + 1/2) 2^-53 from the word pairs (w0, w1), (w2, w3).
//  * RAMBO (Kleiss, Stirling and Ellis, Comput. Phys. Commun. 40 (1986) 359): massless
//    momenta from isotropic directions with energies -log(u u'), boosted and scaled to the
//    centre-of-mass energy; constant weight (2 pi)^(4-3n) (pi/2)^(n-1) s^(n-2)/((n-1)!(n-2)!).
//    For massive particles the published rescaling k = (sqrt(m^2 + x^2 |p|^2), x p), x from
//    energy conservation by Newton iteration, with the weight factor
//    (sum |k| / sqrt s)^(2n-3) prod(|k|/E) sqrt(s) / sum(|k|^2/E).
// The two incoming beams are massless along +z and -z.  One thread per point.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>

#include "../../include/me.h"
#include "me_internal.h"

namespace {

__device__ __forceinline__ void philox_round(uint32_t c[4], uint32_t k0, uint32_t k1) {
  const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
  const uint32_t hi0 = __umulhi(M0, c[0]), lo0 = M0 * c[0];
  const uint32_t hi1 = __umulhi(M1, c[2]), lo1 = M1 * c[2];
  const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
  c[0] = n0;
  c[1] = lo1;
  c[2] = n2;
  c[3] = lo0;
}

__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
  const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += W0;
      k1 += W1;
    }
    philox_round(c, k0, k1);
  }
}

// ((w0 >> 5) 2^26 + (w1 >> 6) + 1/2) 2^-53.  The 53-bit integer is put together in the
// mantissas of two doubles (2^84 + hi 2^32 and 2^52 + lo) and scaled in the exponent: three
// float64 additions instead of two conversions, a multiply-add, an addition and a
// multiplication, the same bits.
__device__ __forceinline__ double u01(uint32_t w0, uint32_t w1) {
  const uint32_t a = w0 >> 5, b = w1 >> 6;
  const uint32_t hi = a >> 6, lo = (a << 26) | b;
  const double x = __hiloint2double(0x45300000, (int)hi), y = __hiloint2double(0x43300000, (int)lo);
  const double k = __dadd_rn(__dadd_rn(__dadd_rn(x, -(19342813113834066795298816.0 + 4503599627370496.0)), y), 0.5);
  return __hiloint2double(__double2hiint(k) - (53 << 20), __double2loint(k));
}

struct Masses {
  double m[4];
};

// RAMBO point from 4 NOUT uniforms: final momenta k[j][0..3] and the weight.  Float64 runs at
// 1/64 of the float32 rate and a division or square root costs five to nine multiply-adds,
// so reciprocals are shared, square roots come from reciprocal ones, angles from sincospi,
// and the mass rescaling is solved in float32 first (its result is within 1e-6, two float64
// Newton steps then end at float64 rounding).
template <int NOUT>
__device__ __forceinline__ void rambo_point(const double* u, double rs, const double* masses, double w_massless,
                                            double k[][4], double& w_out) {
  // massless momenta
  double q[NOUT][4], Q[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int j = 0; j < NOUT; ++j) {
    const double c = 2.0 * u[4 * j] - 1.0;
    const double s = sqrt(1.0 - c * c);
    const double q0 = -log(u[4 * j + 2] * u[4 * j + 3]), qs = q0 * s;
    double sf, cf;
    sincospi(2.0 * u[4 * j + 1], &sf, &cf);
    q[j][0] = q0;
    q[j][1] = qs * cf;
    q[j][2] = qs * sf;
    q[j][3] = q0 * c;
#pragma unroll
    for (int a = 0; a < 4; ++a) Q[a] += q[j][a];
  }
  const double iM = rsqrt(Q[0] * Q[0] - Q[1] * Q[1] - Q[2] * Q[2] - Q[3] * Q[3]);
  const double b[3] = {-Q[1] * iM, -Q[2] * iM, -Q[3] * iM};
  const double x = rs * iM, g = Q[0] * iM, a = 1.0 / (1.0 + g);
#pragma unroll
  for (int j = 0; j < NOUT; ++j) {
    const double bq = b[0] * q[j][1] + b[1] * q[j][2] + b[2] * q[j][3];
    const double f = q[j][0] + a * bq;
    k[j][0] = x * (g * q[j][0] + bq);
#pragma unroll
    for (int d = 0; d < 3; ++d) k[j][1 + d] = x * (q[j][1 + d] + b[d] * f);
  }
  // massive rescaling
  double w = w_massless, msum = 0.0;
  bool massive = false;
#pragma unroll
  for (int j = 0; j < NOUT; ++j) {
    msum += masses[j];
    massive |= masses[j] != 0.0;
  }
  if (massive) {
    const double irs = 1.0 / rs;
    double xs;
    {
      float pf[NOUT], mf[NOUT];
      const float r = (float)(msum * irs);
#pragma unroll
      for (int j = 0; j < NOUT; ++j) {
        pf[j] = (float)(k[j][0] * irs);
        mf[j] = (float)(masses[j] * irs);
      }
      float xf = sqrtf(fmaxf(0.0f, 1.0f - r * r));
      for (int it = 0; it < 12; ++it) {
        float fs = -1.0f, df = 0.0f;
#pragma unroll
        for (int j = 0; j < NOUT; ++j) {
          const float t = xf * pf[j], e = sqrtf(mf[j] * mf[j] + t * t);
          fs += e;
          df += e > 0.0f ? t * pf[j] / e : 0.0f;
        }
        const float dx = fs / df;
        xf -= dx;
        if (!(fabsf(dx) > 1e-6f * xf)) break;
      }
      // near threshold float32 may not settle: start from the massless guess there
      xs = xf > 0.0f && xf <= 1.0f ? (double)xf : sqrt(fmax(0.0, 1.0 - (msum * irs) * (msum * irs)));
    }
    for (int it = 0; it < 60; ++it) {
      double fs = -rs, df = 0.0;
#pragma unroll
      for (int j = 0; j < NOUT; ++j) {
        if (masses[j] != 0.0) {
          const double t = xs * k[j][0], e2 = masses[j] * masses[j] + t * t, ie = rsqrt(e2);
          fs += e2 * ie;
          df += t * k[j][0] * ie;
        } else {
          fs += xs * k[j][0];
          df += k[j][0];
        }
      }
      const double dx = fs / df;
      xs -= dx;
      // Newton converges quadratically: after a step below 1e-9 of xs, xs is exact to rounding
      if (!(fabs(dx) > 1e-9 * xs)) break;
    }
    double sk = 0.0, prod = 1.0, sk2e = 0.0;
#pragma unroll
    for (int j = 0; j < NOUT; ++j) {
      const double ka = xs * k[j][0];
      sk += ka;
      if (masses[j] != 0.0) {
        const double e2 = masses[j] * masses[j] + ka * ka, ie = rsqrt(e2);
        k[j][0] = e2 * ie;
        prod *= ka * ie;
        sk2e += ka * ka * ie;
      } else {
        k[j][0] = ka;
        sk2e += ka;
      }
#pragma unroll
      for (int d = 1; d < 4; ++d) k[j][d] *= xs;
    }
    const double y = sk * irs;
    double pw = y;  // (sum |k| / sqrt s)^(2n-3)
#pragma unroll
    for (int e = 1; e < 2 * NOUT - 3; ++e) pw *= y;
    w *= pw * prod * rs / sk2e;
  }
  w_out = w;
}

template <int NOUT>
__global__ void k_rambo(uint64_t seed, uint32_t stream, long long first, double rs, Masses ms, double w_massless, long n,
                        double* __restrict__ p, double* __restrict__ wgt) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  constexpr int NEXT = NOUT + 2;
  const unsigned long long idx = (unsigned long long)(first + i);
  const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFull), k1 = (uint32_t)(seed >> 32);
  double u[4 * NOUT];
#pragma unroll
  for (int b = 0; b < 2 * NOUT; ++b) {
    uint32_t c[4] = {(uint32_t)(idx & 0xFFFFFFFFull), (uint32_t)(idx >> 32), stream, (uint32_t)b};
    philox4x32_10(c, k0, k1);
    u[2 * b] = u01(c[0], c[1]);
    u[2 * b + 1] = u01(c[2], c[3]);
  }
  double k[NOUT][4], w;
  rambo_point<NOUT>(u, rs, ms.m, w_massless, k, w);
  // beams, then the outgoing momenta: p[comp][leg][n]
  const double hb = 0.5 * rs;
  const double beams[2][4] = {{hb, 0.0, 0.0, hb}, {hb, 0.0, 0.0, -hb}};
#pragma unroll
  for (int comp = 0; comp < 4; ++comp) {
    p[(comp * NEXT + 0) * n + i] = beams[0][comp];
    p[(comp * NEXT + 1) * n + i] = beams[1][comp];
#pragma unroll
    for (int j = 0; j < NOUT; ++j) p[(comp * NEXT + 2 + j) * n + i] = k[j][comp];
  }
  if (wgt) wgt[i] = w;
}

// ---------------------------------------------------------------- points in FKS variables
// Real-emission points from a multichannel density whose channels are the variables of the
// two FKS sectors plus flat phase space (RAMBO).  u0 picks the channel: flat with share
// kAlphaFlat, else one sector (equal shares).  A sector channel is flat in the emitted
// gluon's energy fraction xi (flat three-body phase space has density ~ xi there) and
// samples its cosine to the sector's reference direction as y_j = 1 - 2 v^2, v uniform in
// (v_min, 1), 2 v_min^2 = kYCut (density g(y) = 1 / (4 v (1 - v_min)) ~ 1/sqrt(1 - y)),
// azimuth and Born direction uniform.  The weight is the phase-space measure over the sum
// of all channel densities at the point, 1 / (a_flat / w_RAMBO + sum_j a_j h_j): bounded
// by w_RAMBO / a_flat where the sector channels are thin, and no sector channel comes
// closer than kYCut to a collinear limit (the flat channel covers that region).
// Uniforms: u0..u17 of point i from Philox blocks 0..8 at counter (i lo, i hi, stream,
// block); the flat channel's RAMBO takes u6..u17.
constexpr double kAlphaFlat = 0.25;
constexpr double kYCut = 1e-6;

constexpr double kVMin = 7.0710678118654752440e-4;  // sqrt(kYCut / 2)

__device__ __forceinline__ double coll_density(double y) {
  const double omy = 1.0 - y;
  if (!(omy >= kYCut)) return 0.0;
  return (0.25 / (1.0 - kVMin)) * rsqrt(0.5 * omy);
}

__device__ __forceinline__ void boost_vel(const double p[4], const double b[3], double out[4]) {
  const double b2 = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
  const double g = rsqrt(1.0 - b2);
  const double bp = b[0] * p[1] + b[1] * p[2] + b[2] * p[3];
  const double g2 = g * g / (1.0 + g);  // (g - 1) / b^2
  out[0] = g * (p[0] + bp);
#pragma unroll
  for (int d = 0; d < 3; ++d) out[1 + d] = p[1 + d] + (g2 * bp + g * p[0]) * b[d];
}

// Initial-state sectors of 2 -> Q Qbar g (beams j = 0 along +z, 1 along -z, Q mass
// `mass`): xi = xi_max u1, v from u2, phi = 2 pi u3, the pair's rest-frame direction
// (2 u4 - 1, 2 pi u5); the pair recoils against the gluon with mass^2 s (1 - xi).
// dPhi_3 = dPhi_2(s) xi K dxi dy dphi, K = s beta(s(1-xi)) / (64 pi^3 beta(s)):
// channel density h_j = 4 g(y_j) / (xi_max beta(s) xi K).
// Final-state sectors of massless 2 -> 3 (partner leg 2 or 3, along (2 u1 - 1, 2 pi u2)):
// xi = u3, v from u4, phi = 2 pi u5 about the partner; the partner's energy
// sqrt(s)(1-xi)/(2 - xi(1-y_j)) leaves the third parton massless; channel density
// h_j = 4 g(y_j) / (xi K_j), K_j = s (1 - xi) / (16 pi^3 (2 - xi (1 - y_j))^2).
//
// The flat channel's RAMBO and the sectors' maps are different code, each some 300 to 500
// float64 instructions, and the channel is random: with a point per lane every warp would run
// both.  Each block therefore sorts its points by channel first (a scan over u0's decisions in
// shared memory), so that one of its warps at most runs both.  500,009 g g -> t tbar g
// points: 1181 us before (float64 pipe 88 % busy), 466 us with eight warps in a block.
// While blocks of four warps fit on the SMs one each (19,456 points), every scheduler's float64
// pipe has a single warp, and a call takes one warp's serial chain: 8192 points 24.6 us for
// e+e- -> u ubar g and 31 us for g g -> t tbar g.  With eight warps two share each pipe: 32.8 and
// 43 us (30.7 and 49 us without the sort).
constexpr int FKS_WIDE = 256, FKS_NARROW = 128;
constexpr int64_t FKS_NARROW_POINTS = 152 * FKS_NARROW;

template <bool ISR, int FKS_THREADS>
__global__ void __launch_bounds__(FKS_THREADS) k_fks_points(uint64_t seed, uint32_t stream, long long first, double rs,
                                                            double mass, double w3_massless, long n,
                                                            double* __restrict__ p, double* __restrict__ wgt) {
  __shared__ unsigned short order[FKS_THREADS];
  __shared__ int warp_flat[FKS_THREADS / 32];
  const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFull), k1 = (uint32_t)(seed >> 32);
  const long base = (long)blockIdx.x * FKS_THREADS;
  const double a_f = kAlphaFlat, a_s = 0.5 * (1.0 - kAlphaFlat);
  auto uniforms = [&](unsigned long long idx, uint32_t blk, double* u) {
    uint32_t c[4] = {(uint32_t)(idx & 0xFFFFFFFFull), (uint32_t)(idx >> 32), stream, blk};
    philox4x32_10(c, k0, k1);
    u[0] = u01(c[0], c[1]);
    u[1] = u01(c[2], c[3]);
  };
  {
    double u[2];
    uniforms((unsigned long long)(first + base + threadIdx.x), 0, u);
    const bool f = u[0] < a_f;
    const unsigned bal = __ballot_sync(0xffffffffu, f);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_flat[warp] = __popc(bal);
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < FKS_THREADS / 32; ++w) {
      before += w < warp ? warp_flat[w] : 0;
      all += warp_flat[w];
    }
    const int rank = before + __popc(bal & ((1u << lane) - 1u));  // flat points before this one
    order[f ? rank : all + (int)threadIdx.x - rank] = (unsigned short)threadIdx.x;
    __syncthreads();
  }
  const long i = base + order[threadIdx.x];
  if (i >= n) return;
  const unsigned long long idx = (unsigned long long)(first + i);
  double u[6];
  uniforms(idx, 0, u);
  const double s = rs * rs;
  const bool flat = u[0] < a_f;
  const int sec = u[0] < a_f + a_s ? 0 : 1;
  const double masses[3] = {ISR ? mass : 0.0, ISR ? mass : 0.0, 0.0};
  double q[5][4];  // legs: beams, then 2, 3, 4 (gluon)
  const double hb = 0.5 * rs;
  q[0][0] = hb; q[0][1] = 0.0; q[0][2] = 0.0; q[0][3] = hb;
  q[1][0] = hb; q[1][1] = 0.0; q[1][2] = 0.0; q[1][3] = -hb;
  if (flat) {
    double v[12];
#pragma unroll
    for (int b = 0; b < 6; ++b) uniforms(idx, 3 + b, v + 2 * b);
    double k[3][4], wr;
    rambo_point<3>(v, rs, masses, w3_massless, k, wr);
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) q[2 + j][c] = k[j][c];
  } else {
    uniforms(idx, 1, u + 2);
    uniforms(idx, 2, u + 4);
    const double v = kVMin + (1.0 - kVMin) * u[ISR ? 2 : 4];
    const double yj = 1.0 - 2.0 * v * v;
    if (ISR) {
      const double ximax = 1.0 - 4.0 * mass * mass / s;
      const double xi = ximax * u[1];
      const double y = sec == 0 ? yj : -yj;
      double sf, cf, sp2, cp2;
      sincospi(2.0 * u[3], &sf, &cf);
      const double ek = 0.5 * rs * xi;
      const double et = ek * sqrt(fmax(0.0, (1.0 - y) * (1.0 + y)));
      q[4][0] = ek;
      q[4][1] = et * cf;
      q[4][2] = et * sf;
      q[4][3] = ek * y;
      const double Q0 = rs - ek, M2 = Q0 * Q0 - ek * ek;
      const double cp = 2.0 * u[4] - 1.0;
      // p* sin(theta) and p* cos(theta) of the pair's rest frame
      const double ps2 = fmax(0.0, 0.25 * M2 - mass * mass), pstar = sqrt(ps2);
      const double pt = pstar * sqrt(fmax(0.0, (1.0 - cp) * (1.0 + cp)));
      sincospi(2.0 * u[5], &sp2, &cp2);
      const double e = 0.5 * sqrt(M2);
      const double p3[4] = {e, pt * cp2, pt * sp2, pstar * cp};
      const double p4[4] = {e, -p3[1], -p3[2], -p3[3]};
      const double iQ0 = 1.0 / Q0;
      const double bvec[3] = {-q[4][1] * iQ0, -q[4][2] * iQ0, -q[4][3] * iQ0};
      boost_vel(p3, bvec, q[2]);
      boost_vel(p4, bvec, q[3]);
    } else {
      const double cdir = 2.0 * u[1] - 1.0, xi = u[3];
      double spd, cpd, sf, cf;
      sincospi(2.0 * u[2], &spd, &cpd);
      sincospi(2.0 * u[5], &sf, &cf);
      const double sd = sqrt(fmax(0.0, (1.0 - cdir) * (1.0 + cdir)));
      const double nj[3] = {sd * cpd, sd * spd, cdir};
      double ea[3] = {-cdir * nj[0], -cdir * nj[1], 1.0 - cdir * nj[2]};  // z - (z.nj) nj
      const double ia = rsqrt(ea[0] * ea[0] + ea[1] * ea[1] + ea[2] * ea[2]);
#pragma unroll
      for (int d = 0; d < 3; ++d) ea[d] *= ia;
      const double eb[3] = {nj[1] * ea[2] - nj[2] * ea[1], nj[2] * ea[0] - nj[0] * ea[2], nj[0] * ea[1] - nj[1] * ea[0]};
      const double sr = sqrt(fmax(0.0, (1.0 - yj) * (1.0 + yj)));
      const double ei = 0.5 * rs * xi, ej = rs * (1.0 - xi) / (2.0 - xi * (1.0 - yj));
      double pj[4] = {ej, 0.0, 0.0, 0.0}, po[4] = {rs - ej - ei, 0.0, 0.0, 0.0};
      q[4][0] = ei;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double ni = yj * nj[d] + sr * (cf * ea[d] + sf * eb[d]);
        pj[1 + d] = ej * nj[d];
        q[4][1 + d] = ei * ni;
        po[1 + d] = -(pj[1 + d] + q[4][1 + d]);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        q[2][c] = sec == 0 ? pj[c] : po[c];
        q[3][c] = sec == 0 ? po[c] : pj[c];
      }
    }
  }
  // every channel's density at this point, from its momenta
  const double irs = 1.0 / rs, xi_pt = 2.0 * q[4][0] * irs;
  const double ig = rsqrt(q[4][1] * q[4][1] + q[4][2] * q[4][2] + q[4][3] * q[4][3]);
  double h;
  if (ISR) {
    // a_f / w_RAMBO (rambo_point's weight as a function of the momenta; the gluon is massless)
    const double a2 = q[2][1] * q[2][1] + q[2][2] * q[2][2] + q[2][3] * q[2][3];
    const double a3 = q[3][1] * q[3][1] + q[3][2] * q[3][2] + q[3][3] * q[3][3];
    const double i2 = rsqrt(fmax(a2, 1e-300)), i3 = rsqrt(fmax(a3, 1e-300)), kg = q[4][0];
    const double y = (a2 * i2 + a3 * i3 + kg) * irs, e23 = q[2][0] * q[3][0];
    const double sk2e = a2 * q[3][0] + a3 * q[2][0] + kg * e23;  // sum(|k|^2 / E) E2 E3
    const double m2 = 4.0 * mass * mass / s;
    const double cz = q[4][3] * ig;
    // h_j = 4 g(y_j) / (xi_max beta(s) xi K), K = s beta(s (1 - xi)) / (64 pi^3 beta(s))
    const double b2 = fmax(0.0, 1.0 - m2 / (1.0 - xi_pt));
    const double c0 = a_s * 4.0 * 64.0 * M_PI * M_PI * M_PI / ((1.0 - m2) * s);
    h = a_f * sk2e * i2 * i3 / (w3_massless * y * y * y * rs) +
        c0 * (coll_density(cz) + coll_density(-cz)) * rsqrt(b2) / xi_pt;
  } else {
    h = a_f / w3_massless;
    const double omx = 1.0 - xi_pt, ix = 1.0 / (xi_pt * omx);
#pragma unroll
    for (int j = 2; j <= 3; ++j) {
      const double ik = rsqrt(q[j][1] * q[j][1] + q[j][2] * q[j][2] + q[j][3] * q[j][3]);
      const double y = (q[4][1] * q[j][1] + q[4][2] * q[j][2] + q[4][3] * q[j][3]) * ig * ik;
      const double d = 2.0 - xi_pt * (1.0 - y);
      h += a_s * 4.0 * 16.0 * M_PI * M_PI * M_PI / s * coll_density(y) * d * d * ix;
    }
  }
#pragma unroll
  for (int comp = 0; comp < 4; ++comp)
#pragma unroll
    for (int l = 0; l < 5; ++l) p[(comp * 5 + l) * n + i] = q[l][comp];
  if (wgt) wgt[i] = 1.0 / h;
}

// ---------------------------------------------------------------- unweighting
// Hit-or-miss unweighting of signed weights: point i is kept iff u_i w_max < |w_i|, with
// u_i the first uniform of Philox4x32-10 at counter (point lo, point hi, stream, 0);
// a kept point carries sign(w_i) max(w_max, |w_i|), so that the expected event weight
// is w_i.  The kept indices are written in increasing order: one pass decides every point,
// leaves a bit per point and a count per block, and its last block scans the counts; the
// second pass reads the bits and writes the kept points.
//
// The decision is u w_max < |w| in float64, but float64 instructions run at 1/64 of the
// float32 rate, so it is taken in float32 first, from the leading bits of u and |w|, and in
// float64 only where the two sides are within 1e-6 relative or 1e-8 (the leading 27 bits of
// u) of each other, or not ordinary numbers: the same decisions.  A call
// takes its workspace from those that the handle keeps (allocating and freeing it from the pool
// took most of a call).  2^20 weights against their maximum, the events filled in by the caller: 365 us
// before, 105 us.
constexpr int UW_THREADS = 256;
constexpr int UW_ITEMS = 8;                       // points per thread
constexpr int UW_TILE = UW_THREADS * UW_ITEMS;    // points per block
constexpr int UW_WORDS = UW_TILE / 32;            // mask words per block
constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;

// Results of the last block, in mapped host memory.
struct UwResult {
  unsigned long long max_bits, n_over, n_kept;
};
// Device counters, zero between calls.
struct UwCounters {
  unsigned long long max_bits, n_over;
  unsigned ticket, pad;
};

struct UwArgs {
  const double* w;
  long n;
  double wmax;    // <= 0: the batch maximum of |w| (its bits in ctr->max_bits)
  uint64_t seed;
  uint32_t stream;
  long long first;
  UwCounters* ctr;
  int* counts;     // [blocks]: kept points, then their exclusive scan
  unsigned* bits;  // [n / 32]
};

__device__ __forceinline__ double uw_wmax(const UwArgs& a) {
  return a.wmax > 0.0 ? a.wmax : __longlong_as_double((long long)a.ctr->max_bits);
}
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
// float32 value of a non-negative double's bits, truncated; NaN outside the float32 normals
__device__ __forceinline__ float float_of_bits(unsigned long long b) {
  const int e = (int)(b >> 52) - 896;
  if (b == 0) return 0.0f;
  return e > 0 && e < 255 ? __uint_as_float((unsigned)(b >> 29) - (896u << 23)) : __uint_as_float(0x7fffffffu);
}

// maximum of |w| (NaN skipped): the bit patterns of non-negative doubles order like the
// numbers, so an integer maximum gives it, in any order of the blocks
__global__ void __launch_bounds__(UW_THREADS) k_uw_absmax(const double* __restrict__ w, long n,
                                                          unsigned long long* __restrict__ out) {
  __shared__ unsigned long long sm[UW_THREADS / 32];
  unsigned long long m = 0;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const unsigned long long b = abs_bits(w[i]);
    if (b <= kInfBits && b > m) m = b;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, m, o);
    m = y > m ? y : m;
  }
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < UW_THREADS / 32 ? sm[threadIdx.x] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, m, o);
      m = y > m ? y : m;
    }
    if (threadIdx.x == 0 && m) atomicMax(out, m);
  }
}

// inclusive scan of one int per thread over the block; returns it, *total the block's sum
__device__ __forceinline__ int block_scan(int v, int* sm, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();  // sm may still be read by the previous scan
  if (lane == 31) sm[warp] = x;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int k = 0; k < UW_THREADS / 32; ++k) {
    before += k < warp ? sm[k] : 0;
    all += sm[k];
  }
  *total = all;
  return before + x;
}

__global__ void __launch_bounds__(UW_THREADS) k_uw_decide(UwArgs a, UwResult* __restrict__ res) {
  __shared__ int sm[UW_THREADS / 32];
  __shared__ bool final_block;
  const double wmax = uw_wmax(a);
  const unsigned long long mb = abs_bits(wmax);
  const float fm = float_of_bits(mb), im = 1.0f / fm;  // inf for a maximum of 0: decided in float64
  const uint32_t k0 = (uint32_t)(a.seed & 0xFFFFFFFFull), k1 = (uint32_t)(a.seed >> 32);
  const int lane = threadIdx.x & 31;
  int kept = 0, over = 0;  // of the warp, on every lane
#pragma unroll 2
  for (int t = 0; t < UW_ITEMS; ++t) {
    const long i = (long)blockIdx.x * UW_TILE + t * UW_THREADS + threadIdx.x;
    bool keep = false, ov = false;
    if (i < a.n) {
      const double w = a.w[i];
      const unsigned long long b = abs_bits(w);
      ov = b > mb && b <= kInfBits;
      const unsigned long long idx = (unsigned long long)(a.first + i);
      uint32_t c[4] = {(uint32_t)(idx & 0xFFFFFFFFull), (uint32_t)(idx >> 32), a.stream, 0u};
      philox4x32_10(c, k0, k1);
      const float r = float_of_bits(b) * im, u = __uint2float_rn(c[0] >> 5) * 7.450580597e-9f;
      const float d = u - r;
      keep = d < 0.0f;
      if (!(fabsf(d) > 1e-6f * (u + r) + 1e-8f)) keep = u01(c[0], c[1]) * wmax < fabs(w);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, keep), bov = __ballot_sync(0xffffffffu, ov);
    kept += __popc(bal);
    over += __popc(bov);
    if (lane == 0 && (i & ~31L) < a.n) a.bits[i >> 5] = bal;
  }
  int total, total_over;
  block_scan(lane == 0 ? kept : 0, sm, &total);
  block_scan(lane == 0 ? over : 0, sm, &total_over);
  if (threadIdx.x == 0) {
    __stcg(a.counts + blockIdx.x, total);
    if (total_over) atomicAdd(&a.ctr->n_over, (unsigned long long)total_over);
    __threadfence();
    final_block = atomicAdd(&a.ctr->ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!final_block) return;
  __threadfence();
  // exclusive scan of the counts in place, by this block alone
  long long carry = 0;
  for (unsigned base = 0; base < gridDim.x; base += UW_THREADS * UW_ITEMS) {
    int v[UW_ITEMS], sum = 0;
#pragma unroll
    for (int t = 0; t < UW_ITEMS; ++t) {
      const unsigned i = base + threadIdx.x * UW_ITEMS + t;
      v[t] = i < gridDim.x ? __ldcg(a.counts + i) : 0;
      sum += v[t];
    }
    int all;
    long long at = carry + block_scan(sum, sm, &all) - sum;
#pragma unroll
    for (int t = 0; t < UW_ITEMS; ++t) {
      const unsigned i = base + threadIdx.x * UW_ITEMS + t;
      if (i < gridDim.x) a.counts[i] = (int)at;
      at += v[t];
    }
    carry += all;
  }
  if (threadIdx.x == 0) {
    res->max_bits = mb;
    res->n_over = atomicAdd(&a.ctr->n_over, 0ull);
    res->n_kept = (unsigned long long)carry;
    __threadfence_system();
  }
}

// Each warp places the kept points of UW_ITEMS neighbouring words: the popcounts of the block's
// words are scanned by every warp, and the weights of its words load before the first store.
// The overweight test compares bits (a kept weight is no NaN), which stays off the float64 pipe.
__global__ void __launch_bounds__(UW_THREADS) k_uw_write(UwArgs a, int* __restrict__ kept, double* __restrict__ kept_w) {
  static_assert(UW_WORDS == 64 && UW_WORDS == UW_ITEMS * (UW_THREADS / 32), "two words per lane, UW_ITEMS per warp");
  const int lane = threadIdx.x & 31, first = (threadIdx.x >> 5) * UW_ITEMS;
  const long w0 = (long)blockIdx.x * UW_WORDS, nw = (a.n + 31) / 32;
  const unsigned lo = w0 + 2 * lane < nw ? a.bits[w0 + 2 * lane] : 0u;
  const unsigned hi = w0 + 2 * lane + 1 < nw ? a.bits[w0 + 2 * lane + 1] : 0u;
  const int own = __popc(lo) + __popc(hi);
  int incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const double wmax = uw_wmax(a);
  const unsigned long long mb = abs_bits(wmax);
  int pos = a.counts[blockIdx.x] + __shfl_sync(0xffffffffu, incl - own, first / 2);
  double w[UW_ITEMS];
  unsigned m[UW_ITEMS];
#pragma unroll
  for (int k = 0; k < UW_ITEMS; ++k) {
    m[k] = __shfl_sync(0xffffffffu, k & 1 ? hi : lo, (first + k) / 2);
    w[k] = kept_w && (m[k] >> lane & 1u) ? a.w[(w0 + first + k) * 32 + lane] : 0.0;
  }
#pragma unroll
  for (int k = 0; k < UW_ITEMS; ++k) {
    if (m[k] >> lane & 1u) {
      const int at = pos + __popc(m[k] & ((1u << lane) - 1u));
      kept[at] = (int)((w0 + first + k) * 32 + lane);
      if (kept_w) kept_w[at] = abs_bits(w[k]) > mb ? w[k] : copysign(wmax, w[k]);
    }
    pos += __popc(m[k]);
  }
}

bool on_device(const void* ptr) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, ptr) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" int me_generate_flat(me_handle* h, uint64_t seed, uint32_t stream, int64_t first_point, double sqrt_s,
                                int64_t n, double* momenta, double* ps_weights) {
  if (!h) return me_internal_fail(ME_ERR_ARG, "me_generate_flat: NULL handle");
  if (n < 0 || n > (int64_t)INT32_MAX || first_point < 0 || !(sqrt_s > 0.0))
    return me_internal_fail(ME_ERR_ARG, "me_generate_flat: bad n, first_point or sqrt_s");
  if (n == 0) return ME_OK;
  if (!momenta || !on_device(momenta) || (ps_weights && !on_device(ps_weights)))
    return me_internal_fail(ME_ERR_ARG, "me_generate_flat: momenta and ps_weights must be device memory");
  double masses[4];
  int nout = 0;
  cudaStream_t st = nullptr;
  const int rc = me_internal_final_masses(h, masses, &nout, &st);
  if (rc != ME_OK) return rc;
  double msum = 0.0;
  for (int j = 0; j < nout; ++j) msum += masses[j];
  if (!(msum < sqrt_s)) return me_internal_fail(ME_ERR_ARG, "me_generate_flat: sqrt_s below the final-state masses");
  // constant massless weight (2 pi)^(4-3n) (pi/2)^(n-1) s^(n-2) / ((n-1)! (n-2)!)
  const double s = sqrt_s * sqrt_s;
  double fact = 1.0;
  for (int j = 2; j <= nout - 1; ++j) fact *= j;
  double fact2 = 1.0;
  for (int j = 2; j <= nout - 2; ++j) fact2 *= j;
  const double w0 = std::pow(2.0 * M_PI, 4 - 3 * nout) * std::pow(0.5 * M_PI, nout - 1) * std::pow(s, nout - 2) /
                    (fact * fact2);
  Masses ms{};
  for (int j = 0; j < nout; ++j) ms.m[j] = masses[j];
  const int threads = 128;
  const unsigned blocks = (unsigned)((n + threads - 1) / threads);
  switch (nout) {
    case 2: k_rambo<2><<<blocks, threads, 0, st>>>(seed, stream, first_point, sqrt_s, ms, w0, n, momenta, ps_weights); break;
    case 3: k_rambo<3><<<blocks, threads, 0, st>>>(seed, stream, first_point, sqrt_s, ms, w0, n, momenta, ps_weights); break;
    case 4: k_rambo<4><<<blocks, threads, 0, st>>>(seed, stream, first_point, sqrt_s, ms, w0, n, momenta, ps_weights); break;
    default: return me_internal_fail(ME_ERR_PROCESS, "me_generate_flat: unsupported multiplicity");
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return me_internal_fail(ME_ERR_CUDA, (std::string("me_generate_flat: ") + cudaGetErrorString(e)).c_str());
  return ME_OK;
}

extern "C" int me_generate_fks(me_handle* h, uint64_t seed, uint32_t stream, int64_t first_point, double sqrt_s,
                               int64_t n, double* momenta, double* ps_weights) {
  if (!h) return me_internal_fail(ME_ERR_ARG, "me_generate_fks: NULL handle");
  const int pid = me_internal_handle_process(h);
  const bool isr = pid == me_internal_process_id("gg_ttg") || pid == me_internal_process_id("uu_ttg");
  if (!isr && pid != me_internal_process_id("ee_uug"))
    return me_internal_fail(ME_ERR_PROCESS, "me_generate_fks: process has no FKS sectors");
  if (n < 0 || n > (int64_t)INT32_MAX || first_point < 0 || !(sqrt_s > 0.0))
    return me_internal_fail(ME_ERR_ARG, "me_generate_fks: bad n, first_point or sqrt_s");
  if (n == 0) return ME_OK;
  if (!momenta || !on_device(momenta) || (ps_weights && !on_device(ps_weights)))
    return me_internal_fail(ME_ERR_ARG, "me_generate_fks: momenta and ps_weights must be device memory");
  double masses[4];
  int nout = 0;
  cudaStream_t st = nullptr;
  const int rc = me_internal_final_masses(h, masses, &nout, &st);
  if (rc != ME_OK) return rc;
  const double mass = masses[0];
  if (!(2.0 * mass < sqrt_s)) return me_internal_fail(ME_ERR_ARG, "me_generate_fks: sqrt_s below the final-state masses");
  // massless three-body volume (2 pi)^(4-3n) (pi/2)^(n-1) s^(n-2) / ((n-1)! (n-2)!) = s / (256 pi^3)
  const double w3 = sqrt_s * sqrt_s / (256.0 * M_PI * M_PI * M_PI);
  const bool narrow = n <= FKS_NARROW_POINTS;
  const int threads = narrow ? FKS_NARROW : FKS_WIDE;
  const unsigned blocks = (unsigned)((n + threads - 1) / threads);
  auto launch = [&](auto kernel) {
    kernel<<<blocks, threads, 0, st>>>(seed, stream, first_point, sqrt_s, mass, w3, n, momenta, ps_weights);
  };
  if (narrow) launch(isr ? k_fks_points<true, FKS_NARROW> : k_fks_points<false, FKS_NARROW>);
  else launch(isr ? k_fks_points<true, FKS_WIDE> : k_fks_points<false, FKS_WIDE>);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return me_internal_fail(ME_ERR_CUDA, (std::string("me_generate_fks: ") + cudaGetErrorString(e)).c_str());
  return ME_OK;
}

extern "C" int me_unweight(me_handle* h, const double* weights, int64_t n, double w_max, uint64_t seed, uint32_t stream,
                           int64_t first_point, int32_t* kept, double* kept_weights, int64_t* n_kept, double* w_max_used,
                           int64_t* n_over) {
  if (!h || !n_kept) return me_internal_fail(ME_ERR_ARG, "me_unweight: NULL handle or n_kept");
  if (n < 0 || n > (int64_t)INT32_MAX || first_point < 0 || !(w_max == w_max))
    return me_internal_fail(ME_ERR_ARG, "me_unweight: bad n, first_point or w_max");
  *n_kept = 0;
  if (n_over) *n_over = 0;
  if (w_max_used) *w_max_used = w_max > 0.0 ? w_max : 0.0;
  if (n == 0) return ME_OK;
  if (!weights || !kept || !on_device(weights) || !on_device(kept) || (kept_weights && !on_device(kept_weights)))
    return me_internal_fail(ME_ERR_ARG, "me_unweight: weights, kept and kept_weights must be device memory");
  double masses[4];
  int nout = 0;
  cudaStream_t st = nullptr;
  const int rc = me_internal_final_masses(h, masses, &nout, &st);  // the handle's device and stream
  if (rc != ME_OK) return rc;
  // allocation and the wait below are allowed while another thread captures a stream, in any mode
  struct Relaxed {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    Relaxed() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~Relaxed() { cudaThreadExchangeStreamCaptureMode(&mode); }
  } relaxed;
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &capturing) != cudaSuccess || capturing != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return me_internal_fail(ME_ERR_CUDA, "me_unweight: the handle's stream is being captured");
  }
  // workspace: counters, per-block counts, one bit per point, and the result in mapped host memory
  const long nb = (long)((n + UW_TILE - 1) / UW_TILE), nw = (long)((n + 31) / 32);
  const size_t counts_at = 64, bits_at = counts_at + ((size_t)nb * sizeof(int) + 63) / 64 * 64;
  Workspace space{};
  const int rcw = me_internal_workspace_take(h, bits_at + (size_t)nw * sizeof(unsigned), st, &space);
  if (rcw != ME_OK) return rcw;
  char* ws = (char*)space.dev;
  UwArgs a{weights, (long)n, w_max, seed, stream, (long long)first_point, (UwCounters*)ws, (int*)(ws + counts_at),
           (unsigned*)(ws + bits_at)};
  cudaError_t e = cudaMemsetAsync(ws, 0, sizeof(UwCounters), st);
  if (e == cudaSuccess && !(w_max > 0.0)) {
    const unsigned g = (unsigned)std::min<long>(nb, 1216);  // 8 blocks on each of 152 SMs
    k_uw_absmax<<<g, UW_THREADS, 0, st>>>(weights, (long)n, &a.ctr->max_bits);
  }
  if (e == cudaSuccess) {
    k_uw_decide<<<(unsigned)nb, UW_THREADS, 0, st>>>(a, (UwResult*)space.host_dev);
    k_uw_write<<<(unsigned)nb, UW_THREADS, 0, st>>>(a, kept, kept_weights);
    e = cudaGetLastError();
  }
  const cudaError_t es = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = es;
  const UwResult res = *(const UwResult*)space.host;
  me_internal_workspace_give(h, space, st);
  if (e != cudaSuccess)
    return me_internal_fail(ME_ERR_CUDA, (std::string("me_unweight: ") + cudaGetErrorString(e)).c_str());
  *n_kept = (int64_t)res.n_kept;
  if (n_over) *n_over = (int64_t)res.n_over;
  if (w_max_used) {
    double wm = w_max;
    if (!(w_max > 0.0)) std::memcpy(&wm, &res.max_bits, sizeof wm);
    *w_max_used = wm;
  }
  return ME_OK;
}
