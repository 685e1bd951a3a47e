// Kernels of the event-parallel NLO hot path (templates; instantiated in me_inst_*.cu).
//
// Layout: momenta are structure-of-arrays float64 p[comp][leg][n] (comp = E,px,py,pz),
// so that consecutive events are consecutive addresses; weights are float64 w[n].
// A group of LPE consecutive lanes handles one event: the lanes split the helicity
// blocks (and, for the subtracted real, the Born-kinematics tasks) and reduce with warp
// shuffles.  Helicity sums run over one member of each pair (h, -h) -- the
// configurations with leg 0 at + -- and are doubled: flipping every helicity leaves the
// colour-summed squared amplitude (and every colour/spin-correlated one) unchanged for
// these tree amplitudes with real couplings (pinned against the oracle).  A helicity
// block (me_procs.cuh) is one configuration of the other legs with the four helicities
// of the heavy pair, evaluated with shared gluon currents and quark-line rows; the 2 -> 2
// trees are closed forms (their invariants in float64), and so are the counterterms' Borns, in
// float64 throughout.  Born, real, soft and
// collinear terms are evaluated for every point and masked afterwards (Sec. 4.3, Algorithm 2),
// so a warp never diverges on cuts, or through the per-term queues below.
#pragma once
#include <algorithm>
#include <atomic>

#include "me_procs.cuh"

// minimum resident 128-thread blocks per SM requested from the register allocator: 2
// gives the subtracted-real kernels up to 255 registers (8 warps per SM, fewer spills);
// measured against 3 (168 registers, 12 warps): 9.56 against 9.64 ms per c2 step
#ifndef ME_MINB
#define ME_MINB 2
#endif

namespace me {

constexpr int MAX_FLOW = 24;
constexpr int N_PAIRS = 10;  // unordered pairs (k<=l) of the 4 coloured legs of a 2->2 Born

// Device-resident process constants (written once per device at set-up):
// colour matrices (row-major NFLOW x NFLOW) and the 2->2 Born
// colour correlators C^{kl} (pair order (0,0),(0,1),..,(3,3); [0] gg->tt, [1] uu->tt).
// U holds the upper triangle of the symmetric C with the off-diagonal entries doubled
// (U_aa = C_aa, U_ab = 2 C_ab for b > a, zero below), so that
// J^dagger C J = sum_a Re(J_a^* sum_{b >= a} U_ab J_b).
struct ColourTables {
  double C[P_COUNT][MAX_FLOW * MAX_FLOW];
  double U[P_COUNT][MAX_FLOW * MAX_FLOW];
  float Uf[P_COUNT][MAX_FLOW * MAX_FLOW];
  double Ccorr[2][N_PAIRS][4];
  double S4[S4_COEF];  // g g -> t tbar g g (s4_colour_sum)
  float S4f[S4_COEF];
  double Cqq[N_PAIRS];  // u ubar -> t tbar, contracted with its one colour structure (born_uu_matrix)
};

// Cuts of one configuration (Algorithm 2's passCuts, applied to each term at its own
// kinematics).  Each decision is an integer result taken in float64 with the operations
// in a fixed order and no contraction, so that any implementation doing the same
// operations on the same momenta decides alike:
//   CUT_PT      both heavy quarks (legs 2, 3):  px*px + py*py >= pt2_min
//   CUT_Y       both heavy quarks:  E + |pz| <= ey2 * (E - |pz|),  ey2 = exp(2 y_max)
//   CUT_AXIS    e+e-: the most energetic final parton m (first of equal energies):
//               pz*pz <= cos2_max * ((px*px + py*py) + pz*pz)  (thrust axis along p_m)
//   CUT_THRUST  e+e-: 2 E_m <= thrust_max * (E_0 + E_1)  (thrust T = 2 E_m / sqrt(s))
enum : unsigned { CUT_PT = 1u, CUT_Y = 2u, CUT_AXIS = 4u, CUT_THRUST = 8u };
struct Cuts {
  unsigned mask;  // 0: no cut
  double pt2_min, ey2, cos2_max, thrust_max;
};

struct KParams {
  Couplings cp;
  double tree_scale;    // |M|^2 at unit couplings -> weight: couplings / (initial spin x colour average and
                        // identical-particle factor), x the n-body NLO factor
  double real_scale;    // half helicity sum of a real block at unit couplings -> |M|^2
  double born_scale;    // couplings of the underlying Born / its average
  double xi_cut, delta; // FKS plus-distribution cut-offs
  double xi_thr, y_thr; // points with xi < xi_thr or 1-y < y_thr go to the FP64 path
  double tol_eps;       // tol / me_eps: target accuracy of a weight over the assumed error of a
                        // bulk-precision matrix element
  int flag_unstable;    // 1: append unstable points to the rescue list
  int item_rescue;      // with flag_unstable: records and float64 items instead of the point list
  Cuts cut;             // cuts of every term (mask 0: none)
  const ColourTables* tab;
};

template <typename T> ME_HD const T* s4tab(const ColourTables* t);
template <> ME_HD const double* s4tab<double>(const ColourTables* t) { return t->S4; }
template <> ME_HD const float* s4tab<float>(const ColourTables* t) { return t->S4f; }
template <typename T> ME_HD const T* utab(const ColourTables* t, int pid);
template <> ME_HD const double* utab<double>(const ColourTables* t, int pid) { return t->U[pid]; }
template <> ME_HD const float* utab<float>(const ColourTables* t, int pid) { return t->Uf[pid]; }

template <int PID, typename T>
ME_HD T colour_sum(const ColourTables* tab, const cx<T>* J) {
  constexpr int NF = Proc<PID>::NFLOW;
  if constexpr (PID == P_GG_TTGG)
    return s4_colour_sum(s4tab<T>(tab), [&](int v, int a) { return J[s4_flow(v, a)]; });
  T s = T(0);
  // triangular form: NF (NF + 1) + 2 NF multiply-adds instead of 2 NF^2 + 2 NF
  const T* __restrict__ Um = utab<T>(tab, PID);
#pragma unroll
  for (int a = 0; a < NF; ++a) {
    const T d = Um[a * NF + a];
    T zr = d * J[a].re, zi = d * J[a].im;
#pragma unroll
    for (int b = a + 1; b < NF; ++b) {
      const T c = Um[a * NF + b];
      zr += c * J[b].re;
      zi += c * J[b].im;
    }
    s += J[a].re * zr + J[a].im * zi;
  }
  return s;
}

// Live block b (K at unit couplings), summed over the four heavy-pair helicities and colours
template <int PID, typename T, typename KP>
ME_HD T block_sum(const Kin<PID, T>& K, int b, const KP& kp) {
  if constexpr (PID == P_EE_UUG) {
    return ee_uug_block(K, b);
  } else {
    T acc = T(0);
    amplitude_block<PID, T>(K, live_block_hel<PID>(b), unit_couplings(kp.cp),
                            [&](int, const cx<T>* J) { acc += colour_sum<PID, T>(kp.tab, J); });
    return acc;
  }
}

template <int LPE, typename T>
__device__ __forceinline__ T group_sum(T v, unsigned mask) {
#pragma unroll
  for (int o = LPE / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o, LPE);
  return v;
}

template <int LPE>
__device__ __forceinline__ unsigned group_mask() {
  if constexpr (LPE == 32) {
    return 0xffffffffu;
  } else {
    const unsigned lane = threadIdx.x & 31u;
    return ((1u << LPE) - 1u) << (lane & ~(unsigned)(LPE - 1));
  }
}

// legs 0 .. LEGS - 1 of an event with NEXT legs
template <int NEXT, int LEGS>
__device__ __forceinline__ void load_legs(const double* __restrict__ p, long n, long i, r4<double>* k) {
#pragma unroll
  for (int l = 0; l < LEGS; ++l) {
    k[l].e = __ldg(p + (0L * NEXT + l) * n + i);
    k[l].x = __ldg(p + (1L * NEXT + l) * n + i);
    k[l].y = __ldg(p + (2L * NEXT + l) * n + i);
    k[l].z = __ldg(p + (3L * NEXT + l) * n + i);
  }
}
template <int NEXT>
__device__ __forceinline__ void load_event(const double* __restrict__ p, long n, long i, r4<double>* k) {
  load_legs<NEXT, NEXT>(p, n, i, k);
}

// ---------------------------------------------------------------- cuts
__device__ __forceinline__ bool heavy_pass(const r4<double>& q, const Cuts& c) {
  bool ok = true;
  if (c.mask & CUT_PT) ok = ok && __dadd_rn(__dmul_rn(q.x, q.x), __dmul_rn(q.y, q.y)) >= c.pt2_min;
  if (c.mask & CUT_Y) {
    const double a = fabs(q.z);
    ok = ok && __dadd_rn(q.e, a) <= __dmul_rn(c.ey2, __dsub_rn(q.e, a));
  }
  return ok;
}

// passCuts of a configuration k of process PID (or of a Born counter-event of it)
template <int PID>
__device__ __forceinline__ bool pass_cuts(const r4<double>* k, const Cuts& c) {
  if constexpr (PID == P_EE_UU || PID == P_EE_UUG) {
    r4<double> m = k[2];
#pragma unroll
    for (int i = 3; i < Proc<PID>::NEXT; ++i)
      if (k[i].e > m.e) m = k[i];
    bool ok = true;
    if (c.mask & CUT_AXIS) {
      const double t = __dadd_rn(__dmul_rn(m.x, m.x), __dmul_rn(m.y, m.y));
      const double z2 = __dmul_rn(m.z, m.z);
      ok = ok && z2 <= __dmul_rn(c.cos2_max, __dadd_rn(t, z2));
    }
    if (c.mask & CUT_THRUST) ok = ok && 2.0 * m.e <= __dmul_rn(c.thrust_max, __dadd_rn(k[0].e, k[1].e));
    return ok;
  } else {
    return heavy_pass(k[2], c) && heavy_pass(k[3], c);
  }
}

// ---------------------------------------------------------------- tree |M|^2
// The tree kernels clear the ticket of the reduction that follows them.
__device__ __forceinline__ void clear_ticket(int* ticket) {
  if (blockIdx.x == 0 && threadIdx.x == 0 && ticket) *ticket = 0;
}

// out[i] = wgt[i] * |M|^2(p_i) * nlo_factor.  `count` (optional): the number of events,
// read on the device; `idx` (optional): the list of events to process (its length in
// `count`).  Momenta have stride n either way.  (g g -> t tbar g g runs k_tree_tt4 and, in
// float32, k_tree_tt4f below instead.)
template <int PID, typename T, int LPE>
__global__ void __launch_bounds__(128, ME_MINB) k_tree(const double* __restrict__ p, const double* __restrict__ wgt,
                                                       long n, double* __restrict__ out, KParams kp,
                                                       const int* __restrict__ idx, const int* __restrict__ count,
                                                       int* __restrict__ ticket) {
  static_assert(PID != P_GG_TTGG, "g g -> t tbar g g runs k_tree_tt4 and k_tree_tt4f");
  clear_ticket(ticket);
  constexpr int NEXT = Proc<PID>::NEXT;
  const long gid = ((long)blockIdx.x * blockDim.x + threadIdx.x) / LPE;
  const int lane = threadIdx.x % LPE;
  const long nev = count ? (long)*count : n;
  if (gid >= nev) return;
  const long ev = idx ? (long)idx[gid] : gid;
  r4<double> k[NEXT];
  load_event<NEXT>(p, n, ev, k);
  // Algorithm 2: every point is evaluated, and zeroed below where it fails the cuts
  const bool pass = !kp.cut.mask || pass_cuts<PID>(k, kp.cut);
  const Kin<PID, T> K = prepare<PID, T>(k, unit_couplings(kp.cp));
  T acc = T(0);
  constexpr int NB = n_live_blocks<PID>(), NBL = (NB + LPE - 1) / LPE;
#pragma unroll 1
  for (int b = lane * NBL; b < (lane + 1) * NBL && b < NB; ++b) acc += block_sum<PID, T>(K, b, kp);
  const double tot = 2.0 * (double)group_sum<LPE>(acc, group_mask<LPE>());
  if (lane == 0) {
    const double w = wgt ? wgt[ev] : 1.0;
    out[ev] = pass ? w * tot * kp.tree_scale : 0.0;
  }
}

// g g -> t tbar g g in float64: as k_tree, with the L = 2^lg lanes of an event in different warps
// (half warps for L = 8), so that the beam gluons' helicities, which choose the form of a block,
// are the same across a warp.  The float64 pipe bounds it (85 % at 8191 events, whose 2048 warps
// fill the schedulers unevenly): 3.96 ms with general polarisations, every current and product
// built on its own and the triangle of the colour matrix, 2.13 ms like this.
template <int PID>
__global__ void __launch_bounds__(128, ME_MINB) k_tree_tt4(const double* __restrict__ p, const double* __restrict__ wgt,
                                                           long n, double* __restrict__ out, KParams kp,
                                                           const int* __restrict__ idx, const int* __restrict__ count,
                                                           int* __restrict__ ticket, int lg) {
  static_assert(PID == P_GG_TTGG, "eight blocks");
  clear_ticket(ticket);
  __shared__ double part[128];
  const int slot = threadIdx.x & ((128 >> lg) - 1), lane = threadIdx.x >> (7 - lg);
  const long gid = ((long)blockIdx.x << (7 - lg)) + slot;
  const long nev = count ? (long)*count : n;
  const bool live = gid < nev;
  const long ev = live ? (idx ? (long)idx[gid] : gid) : 0;
  double acc = 0.0;
  bool pass = false;
  if (live) {
    r4<double> k[6];
    load_event<6>(p, n, ev, k);
    pass = !kp.cut.mask || pass_cuts<PID>(k, kp.cut);
    const Kin<PID, double> K = prepare<PID, double>(k, unit_couplings(kp.cp));
#pragma unroll 1
    for (int b = lane << (3 - lg); b < (lane + 1) << (3 - lg); ++b)
      acc += block_sum<PID, double>(K, ((b & 3) << 1) | (b >> 2), kp);  // leg 1 in the top bit
  }
  part[threadIdx.x] = acc;
  __syncthreads();
  if (!live || lane > 0) return;
  for (int i = 1; i < 1 << lg; ++i) acc += part[(i << (7 - lg)) + slot];
  out[ev] = pass ? (wgt ? wgt[ev] : 1.0) * (2.0 * acc) * kp.tree_scale : 0.0;
}

// The closed 2 -> 2 trees: one lane per event, bound by the momenta's DRAM traffic and, in
// the float64 products, by the float64 pipe.  A call with 2^20 g g -> t tbar points: 113 us with the helicity
// amplitudes (float32), 42 us here.
template <int PID, typename T>
__global__ void __launch_bounds__(256) k_tree_closed(const double* __restrict__ p, const double* __restrict__ wgt,
                                                     long n, double* __restrict__ out, KParams kp,
                                                     const int* __restrict__ idx, const int* __restrict__ count,
                                                     int* __restrict__ ticket) {
  clear_ticket(ticket);
  const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long nev = count ? (long)*count : n;
  if (gid >= nev) return;
  const long ev = idx ? (long)idx[gid] : gid;
  r4<double> k[4];
  if (PID == P_GG_TT && !kp.cut.mask) {
    load_legs<4, 3>(p, n, ev, k);  // leg 3 enters the cuts only
  } else {
    load_event<4>(p, n, ev, k);
  }
  const bool pass = !kp.cut.mask || pass_cuts<PID>(k, kp.cut);
  const double tot = (double)closed_sum<PID, T>(k, unit_couplings(kp.cp)) * kp.tree_scale;
  out[ev] = pass ? (wgt ? wgt[ev] * tot : tot) : 0.0;
}

// ---------------------------------------------------------------- g g -> t tbar g g, float32
// Four lanes share one event and one helicity block at a time (me_procs.cuh: the gluon
// helicities fixed, the four (t, tbar) helicities open).  Lane w works on what belongs to
// gluon w, the other gluons counted as w ^ 1, w ^ 2, w ^ 3, so that every index into the
// event's shared-memory area is an exclusive or:
//  1. polarisation w; pair currents J(xy) in both orders; the three triples J(xyz) of the
//     gluons other than w; the quadruples J(wxyz), x < y, to the ends z = w ^ 1 and w ^ 2,
//     and to w ^ 3 from decoupling, J(wxyz) = -J(xwyz) - J(xywz) - J(xyzw);
//  2. the quark line of the six orderings that start with w, U(w) -> U(wx) -> U(wxy), for
//     both top helicities, the partial amplitudes of both antitop helicities going to
//     shared-memory rows;
//  3. the colour sum of heavy-pair helicity w.
// Everything a lane needs stays on chip, so the 3e5 flops of an event run from registers
// and shared memory; instruction issue bounds the kernel.  2^18 events: 4.42 ms with four lanes
// that picked currents from tables and a bf16 x 3 mma colour sum, 2.15 ms like this; three
// blocks per SM (168 registers) 2.47 ms.  In a warp that holds the end of the
// batch, events past it compute a fixed finite configuration and are discarded, so every
// warp-wide step stays converged; warps entirely past the end return at once.
// An event's shared-memory area: 40 four-vectors x 8 floats, the gluon momenta q[4], the
// reciprocal denominators ig[16], iq[16], padded so that 8 events hit distinct banks.
constexpr int TT4_Q = 320, TT4_IG = 336, TT4_IQ = 352, TT4_EV = 372;
constexpr int TT4_ROW = 52;  // floats per amplitude row (24 complex, padded)
constexpr int TT4_WARP = 8 * TT4_EV + 32 * TT4_ROW;
constexpr int TT4_THREADS = 128;
constexpr int TT4_SMEM = (TT4_THREADS / 32) * TT4_WARP * 4;
// slots: polarisations 0 .. 3; ordered pairs J(xy); triples by missing and middle gluon;
// quadruples J(w..z) by first and last gluon, the two in between in increasing order
__device__ __forceinline__ int tt4_pair(int x, int y) { return 4 + 3 * x + (x ^ y) - 1; }
__device__ __forceinline__ int tt4_triple(int miss, int mid) { return 16 + 3 * miss + (miss ^ mid) - 1; }
__device__ __forceinline__ int tt4_quad(int w, int z) { return 28 + 3 * w + (w ^ z) - 1; }

__device__ __forceinline__ void st8(float* b, int slot, cx<float> a, cx<float> c, cx<float> d, cx<float> e) {
  float4* p = reinterpret_cast<float4*>(b + 8 * slot);
  p[0] = make_float4(a.re, a.im, c.re, c.im);
  p[1] = make_float4(d.re, d.im, e.re, e.im);
}
__device__ __forceinline__ void st_c4(float* b, int slot, const c4<float>& v) { st8(b, slot, v.v[0], v.v[1], v.v[2], v.v[3]); }
__device__ __forceinline__ c4<float> ld_c4(const float* b, int slot) {
  const float4* p = reinterpret_cast<const float4*>(b + 8 * slot);
  const float4 a = p[0], c = p[1];
  return c4<float>{{{a.x, a.y}, {a.z, a.w}, {c.x, c.y}, {c.z, c.w}}};
}
// slots 0 .. 3: a polarisation (no time component, real z)
__device__ __forceinline__ pol<float> ld_pol(const float* b, int slot) {
  const float4* p = reinterpret_cast<const float4*>(b + 8 * slot);
  const float4 a = p[0], c = p[1];
  return pol<float>{{a.z, a.w}, {c.x, c.y}, c.z};
}
__device__ __forceinline__ r4<float> ld_q(const float* b, int g) {
  const float4 a = *reinterpret_cast<const float4*>(b + TT4_Q + 4 * g);
  return r4<float>{a.x, a.y, a.z, a.w};
}
// the same eight floats read as the chiral combinations (V0 - V3, V0 + V3, V1 - i V2,
// V1 + i V2) once a slot has been converted in place for the quark lines
__device__ __forceinline__ sl4<float> ld_sl4(const float* b, int slot) {
  const float4* p = reinterpret_cast<const float4*>(b + 8 * slot);
  const float4 a = p[0], c = p[1];
  return sl4<float>{{a.x, a.y}, {a.z, a.w}, {c.x, c.y}, {c.z, c.w}};
}
__device__ __forceinline__ spol<float> ld_spol(const float* b, int slot) {
  const float4* p = reinterpret_cast<const float4*>(b + 8 * slot);
  const float4 a = p[0], c = p[1];
  return spol<float>{a.z, {c.x, c.y}, {c.z, c.w}};
}
__device__ __forceinline__ void st_sl4(float* b, int slot, const sl4<float>& S) { st8(b, slot, S.a, S.b, S.c, S.d); }

template <int PID>
__global__ void __launch_bounds__(TT4_THREADS, 2) k_tree_tt4f(const double* __restrict__ p, const double* __restrict__ wgt,
                                                              long n, double* __restrict__ out, KParams kp,
                                                              const int* __restrict__ idx, const int* __restrict__ count,
                                                              int* __restrict__ ticket) {
  static_assert(PID == P_GG_TTGG, "eight blocks");
  clear_ticket(ticket);
  extern __shared__ __align__(16) float tt4_smem[];
  const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
  float* wsm = tt4_smem + warp * TT4_WARP;
  float* cur = wsm + (wl >> 2) * TT4_EV;  // this event's area
  float* rows = wsm + 8 * TT4_EV;         // amplitude rows [32][TT4_ROW]: 4 event + helicity
  const long gid = ((long)blockIdx.x * blockDim.x + threadIdx.x) / 4;
  const int w = threadIdx.x & 3;
  const long nev = count ? (long)*count : n;
  // a warp whose eight events all lie past the batch leaves together (every
  // synchronisation below is warp-wide), so a grid sized for a capacity costs little
  if (((long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) / 4 >= nev) return;
  const bool active = gid < nev;
  const long ev = active ? (idx ? (long)idx[gid] : gid) : 0;
  r4<double> k[6];
  if (active) {
    load_event<6>(p, n, ev, k);
  } else {
    const double d[6][4] = {{1000, 0, 0, 1000},     {1000, 0, 0, -1000},     {600, 100, 200, 300},
                            {700, -150, -100, 200}, {400, 30, -80, -300}, {300, 20, -20, -200}};
#pragma unroll
    for (int l = 0; l < 6; ++l) k[l] = r4<double>{d[l][0], d[l][1], d[l][2], d[l][3]};
  }
  const Kin<PID, float> K = prepare<PID, float>(k, unit_couplings(kp.cp));
  const float mt = kp.cp.mtf;
  const r4<float> kt = K.pl[2];
  {
    // lane l writes momentum l and a quarter of the denominators
    const r4<float> ql = w == 0 ? K.q[0] : w == 1 ? K.q[1] : w == 2 ? K.q[2] : K.q[3];
    *reinterpret_cast<float4*>(cur + TT4_Q + 4 * w) = make_float4(ql.e, ql.x, ql.y, ql.z);
#pragma unroll
    for (int S = 0; S < 16; ++S)
      if ((S & 3) == w) {
        cur[TT4_IG + S] = K.ig[S];
        cur[TT4_IQ + S] = K.iq[S];
      }
  }
  const wf_v<float> wg = w == 0 ? K.wg[0] : w == 1 ? K.wg[1] : w == 2 ? K.wg[2] : K.wg[3];
  const int leg = w < 2 ? w : w + 2;
  __syncwarp();
  const float* ig = cur + TT4_IG;
  const float* iq = cur + TT4_IQ;
  float acc = 0.0f;
#pragma unroll 1
  for (int b = 0; b < n_live_blocks<PID>(); ++b) {
    const int hb = live_block_hel<PID>(b);
    {
      const pol<float> e = pol_of(wg, hel_of(hb, leg), w >= 2);
      st_c4(cur, w, c4<float>{{{0.0f, 0.0f}, e.x, e.y, {e.z, 0.0f}}});
    }
    __syncwarp();
    // pairs (0, 1), (2, 3), (0, 2), (1, 3), then (0, 3), (1, 2)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      if (r == 1 && w >= 2) break;
      const int x = r == 0 ? (w < 2 ? 2 * w : w - 2) : w;
      const int y = r == 0 ? (w < 2 ? x + 1 : w) : 3 - w;
      cx<float> exy;
      const c4<float> J = bracket(ld_pol(cur, x), ld_q(cur, x), ld_pol(cur, y), ld_q(cur, y), -ig[(1 << x) | (1 << y)], exy);
      st_c4(cur, tt4_pair(x, y), J);
      st_c4(cur, tt4_pair(y, x), cneg(J));
    }
    __syncwarp();
    // triples of x, y, z = w ^ 1, w ^ 2, w ^ 3: each bracket of a gluon and a pair enters two of
    // the three currents, and the three add up to zero
    {
      const int x = w ^ 1, y = w ^ 2, z = w ^ 3;
      const pol<float> ex = ld_pol(cur, x), ey = ld_pol(cur, y), ez = ld_pol(cur, z);
      const r4<float> qx = ld_q(cur, x), qy = ld_q(cur, y), qz = ld_q(cur, z);
      const float i3 = ig[15 ^ (1 << w)];
      const cx<float> exy = i3 * cdot(ex, ey), eyz = i3 * cdot(ey, ez), exz = i3 * cdot(ex, ez);
      c4<float> Jy = czero<float>(), Jx = czero<float>();
      {
        const c4<float> P = ld_c4(cur, tt4_pair(y, z));
        bracket_acc(Jy, ex, qx, P, qy + qz, -i3, cdot(ex, P));  // x (yz)
      }
      {
        const c4<float> P = ld_c4(cur, tt4_pair(x, z));
        bracket_acc(Jx, ey, qy, P, qx + qz, -i3, cdot(ey, P));  // y (xz)
      }
      {
        const c4<float> P = ld_c4(cur, tt4_pair(x, y));
        c4<float> Bz = czero<float>();
        bracket_acc(Bz, ez, qz, P, qx + qy, -i3, cdot(ez, P));  // z (xy)
        csub(Jy, Bz);
        cadd(Jx, Bz);
      }
      quartic_acc(Jy, ex, ey, ez, exz, exy, eyz);  // J(xyz)
      quartic_acc(Jx, ey, ex, ez, eyz, exy, exz);  // J(yxz)
      st_c4(cur, tt4_triple(w, y), Jy);
      st_c4(cur, tt4_triple(w, x), Jx);
      cadd(Jx, Jy);
      st_c4(cur, tt4_triple(w, z), cneg(Jx));
    }
    __syncwarp();
    // quadruples J(w x y z), z = w ^ 1, w ^ 2, slashed as they are stored
    const pol<float> ew = ld_pol(cur, w);
    const r4<float> qw = ld_q(cur, w);
    const float i4 = ig[15];
#pragma unroll
    for (int pz = 1; pz < 3; ++pz) {
      const int z = w ^ pz, o = w ^ (3 - pz), o3 = w ^ 3, x = min(o, o3), y = max(o, o3);
      const pol<float> ex = ld_pol(cur, x), ey = ld_pol(cur, y), ez = ld_pol(cur, z);
      const c4<float> jwx = ld_c4(cur, tt4_pair(w, x)), jyz = ld_c4(cur, tt4_pair(y, z));
      const r4<float> qz = ld_q(cur, z), qwx = qw + ld_q(cur, x), qyz = ld_q(cur, y) + qz;
      c4<float> J = czero<float>();
      bracket_acc(J, jwx, qwx, jyz, qyz, -i4);
      quartic_acc(J, ew, ex, jyz, i4 * cdot(ew, jyz), i4 * cdot(ew, ex), i4 * cdot(ex, jyz));
      quartic_acc(J, jwx, ey, ez, i4 * cdot(ez, jwx), i4 * cdot(ey, jwx), i4 * cdot(ey, ez));
      {
        const c4<float> jxy = ld_c4(cur, tt4_pair(x, y));
        quartic_acc(J, ew, jxy, ez, i4 * cdot(ew, ez), i4 * cdot(ew, jxy), i4 * cdot(ez, jxy));
      }
      {
        const c4<float> P = ld_c4(cur, tt4_triple(w, y));
        bracket_acc(J, ew, qw, P, (qwx - qw) + qyz, -i4, cdot(ew, P));
      }
      {
        const c4<float> P = ld_c4(cur, tt4_triple(z, x));
        bracket_acc(J, ez, qz, P, qwx + (qyz - qz), i4, cdot(ez, P));
      }
      st_sl4(cur, tt4_quad(w, z), slashed(J));
    }
    __syncwarp();
    // the quark lines only slash the other vectors too: convert them in place; and the
    // quadruples to z = w ^ 3, x < y: J(xwyz) + J(xywz) = J(x..z) - J(z..x) of increasing middles
#pragma unroll
    for (int i = 0; i < 7; ++i) st_sl4(cur, 4 * i + w, slashed(ld_c4(cur, 4 * i + w)));
    {
      const int z = w ^ 3, x = min(w ^ 1, w ^ 2), y = max(w ^ 1, w ^ 2);
      const sl4<float> A = ld_sl4(cur, tt4_quad(x, z)), B = ld_sl4(cur, tt4_quad(z, x));
      const sl4<float> C = ld_sl4(cur, y < z ? tt4_quad(x, w) : tt4_quad(w, x));
      const float s = y < z ? -1.0f : 1.0f;
      auto f = [&](cx<float> a, cx<float> b, cx<float> c) { return rmac(b - a, s, c); };
      st8(cur, tt4_quad(w, z), f(A.a, B.a, C.a), f(A.b, B.b, C.b), f(A.c, B.c, C.c), f(A.d, B.d, C.d));
    }
    __syncwarp();
    // quark lines.  Products of U(w) and U(wx) with a pair or triple current serve an
    // ordering and its reflection in the rest: J(yx) = -J(xy), J(zyx) = J(xyz).
    const r4<float> ktw = kt + qw;
#pragma unroll
    for (int ht = 0; ht < 2; ++ht) {
      asm volatile("" ::: "memory");  // currents are read again: held for both spins, or for all x, they spill
      float2* row = reinterpret_cast<float2*>(rows + ((wl & ~3) + 2 * ht) * TT4_ROW) + 6 * w;  // hv = 0; hv = 1 in the next
      const c4<float> U1 = row_prop(ubar_slash(K.wt, ht, ld_spol(cur, w)), scaled_prop(ktw, mt, -iq[1 << w]));
      c4<float> P[3], Q[3];  // by the gluon left out of the pair, the middle of the triple
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        P[i] = row_slash(U1, ld_sl4(cur, tt4_pair(w ^ (i == 0 ? 2 : 1), w ^ (i == 2 ? 2 : 3))));
        Q[i] = row_slash(U1, ld_sl4(cur, tt4_triple(w, w ^ (i + 1))));
      }
#pragma unroll
      for (int px = 1; px < 4; ++px) {
        const int x = w ^ px;
        asm volatile("" ::: "memory");
        const r4<float> kwx = ktw + ld_q(cur, x);
        c4<float> r2 = ubar_slash(K.wt, ht, ld_sl4(cur, tt4_pair(w, x)));
        row_slash_acc(r2, U1, ld_spol(cur, x));
        const c4<float> U2 = row_prop(r2, scaled_prop(kwx, mt, -iq[(1 << w) | (1 << x)]));
        const int pl = px == 1 ? 2 : 1, ph = px == 3 ? 2 : 3;
        const c4<float> D = row_slash(U2, ld_sl4(cur, tt4_pair(w ^ pl, w ^ ph)));
#pragma unroll
        for (int ky = 0; ky < 2; ++ky) {
          const int py = ky ? ph : pl, pz = ky ? pl : ph, y = w ^ py, z = w ^ pz;
          c4<float> r3 = px < py ? P[pz - 1] : cneg(P[pz - 1]);
          ubar_slash_acc(r3, K.wt, ht, ld_sl4(cur, tt4_triple(z, x)));
          row_slash_acc(r3, U2, ld_spol(cur, y));
          const c4<float> U3 = row_prop(r3, scaled_prop(kwx + ld_q(cur, y), mt, -iq[15 ^ (1 << z)]));
          c4<float> R = Q[py - 1];
          if (ky) csub(R, D);
          else cadd(R, D);
          const bool up = x < y;  // J(wxyz), or -J(zyxw)
          ubar_slash_acc(R, scaled(K.wt, up ? 1.0f : -1.0f), ht, ld_sl4(cur, up ? tt4_quad(w, z) : tt4_quad(z, w)));
          row_slash_acc(R, U3, ld_spol(cur, z));
          const cx<float> a0 = dot_v(R, K.wtb, 0), a1 = dot_v(R, K.wtb, 1);
          const int a = 2 * (px - 1) + ky;
          row[a] = make_float2(a0.re, a0.im);
          row[TT4_ROW / 2 + a] = make_float2(a1.re, a1.im);
        }
      }
    }
    __syncwarp();
    // colour sum of row wl: this event, heavy-pair helicity w
    const float2* mine = reinterpret_cast<const float2*>(rows + wl * TT4_ROW);
    const float* coef = kp.tab->S4f;
    asm volatile("" : "+l"(coef));  // 60 coefficients from L1 for each block, not from registers across blocks
    const float sres = s4_colour_sum(coef, [&](int v, int a) {
      const float2 z = mine[6 * v + a];
      return cx<float>{z.x, z.y};
    });
    if (active) acc += sres;
    // the next block's writes to the rows come after its __syncwarp calls
  }
  const double tot = 2.0 * (double)group_sum<4>(acc, group_mask<4>());
  if (active && w == 0) {
    const double w8 = wgt ? wgt[ev] : 1.0;
    bool pass = true;
    if (kp.cut.mask) {
      r4<double> kc[6];
      load_event<6>(p, n, ev, kc);
      pass = pass_cuts<P_GG_TTGG>(kc, kp.cut);
    }
    out[ev] = pass ? w8 * tot * kp.tree_scale : 0.0;
  }
}

// ---------------------------------------------------------------- FKS kinematics (double)
// Float64 throughout (the maps fix the counter-event kinematics that the subtraction
// compares with the real).  GB300 issues float64 at 1/64 of the float32 rate, and a
// float64 division or square root costs ~10 pipe instructions, so the maps use reciprocal
// square roots and shared reciprocals, and boost with the system momentum and mass.

// p (given in the rest frame of a system with momentum Q, mass M) in the frame where the
// system has momentum Q:  E' = (E Q0 + Q.p)/M,  p' = p + Q (E' + E)/(Q0 + M).
__device__ __forceinline__ r4<double> boost_by(const r4<double>& p, const r4<double>& Q, double inv_m, double inv_qm) {
  const double qp = Q.x * p.x + Q.y * p.y + Q.z * p.z;
  const double e = (p.e * Q.e + qp) * inv_m;
  const double c = (e + p.e) * inv_qm;
  return r4<double>{e, p.x + c * Q.x, p.y + c * Q.y, p.z + c * Q.z};
}

__device__ __forceinline__ void unit3(const r4<double>& p, double& x, double& y, double& z) {
  const double a = rsqrt(p.x * p.x + p.y * p.y + p.z * p.z);
  x = p.x * a;
  y = p.y * a;
  z = p.z * a;
}

constexpr double PI = 3.14159265358979323846;
constexpr double CF_ = 4.0 / 3.0;
constexpr double CA_ = 3.0;

// ---------------------------------------------------------------- real - counterterms
// One point of the subtracted real, summed over FKS sectors (ME units):
//   W_j = R S_j - [Th_s G(0,y) + Th_c G(xi,1) - Th_s Th_c G(0,1)] / (xi^2 (1-y) K),
// with the error scale of the stability test.  The LPE lanes of a group evaluate one
// point together and all return the same result.
//
// W = R + W_B, R = sum_b R_b (helicity blocks) the real matrix element -- the sector functions
// add up to 1 -- and W_B the counterterms.  Their
// Born values are closed forms of some 40 float64 operations, so they are evaluated in
// float64 for every point, in every precision, and only the real's blocks have a
// bulk-precision value.  The item rescue re-evaluates in float64 the blocks whose float32
// error the point's tolerance cannot absorb, and recombines W.
template <int PID>
struct RealLayout {
  static constexpr int NB = n_live_blocks<PID>();  // the real's blocks
  // block code depends on the parity of b (the helicity of beam gluon 1, amp_tt3_block): lanes
  // of a warp should run blocks of one parity together
  static constexpr bool BY_PARITY = PID == P_GG_TTG;
};
constexpr int MAX_BLOCKS = 4;

struct RealSubOut {
  double W;     // subtracted real, summed over sectors
  double magR;  // error scale: sum_j |R S_j|
  double magB;  // and |CT_coll| + |CT_soft - CT_softcoll| per sector
  double y[2];  // y_j of both sectors (collinear resolution of the test)
  bool near;    // inside xi_thr / y_thr of an active counterterm
};

// Everything of a point but the real matrix element.
struct PointTerms {
  bool real;     // the real passes its cuts (the sector functions add up to 1)
  double w_born; // the counterterms (with their sign): W = R + w_born, or w_born
  double mag_b;  // their error scale, |CT_coll| + |CT_soft - CT_softcoll| per sector
  double y[2];
  bool near;     // inside xi_thr / y_thr of an active counterterm
  bool inside;   // inside the FKS domain (false where a direction is NaN)
  bool need[2];  // active Born configurations: soft, collinear (initial state); sector 1, 2
};

// a < b for b >= 0, on the bit patterns: a float64 comparison occupies the float64 pipe like a
// multiply-add.  For a NaN the answer follows its sign bit; the domain test (PointTerms::inside)
// then discards the point.
__device__ __forceinline__ bool below(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b);
}
// a > 0, infinity included; false for a NaN of either sign
__device__ __forceinline__ bool positive(double a) {
  return (unsigned long long)(__double_as_longlong(a) - 1) < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool is_nan(double a) {
  return (unsigned long long)__double_as_longlong(a) << 1 > 0xffe0000000000000ull;
}
// Whether unit3 gives p a direction: no component infinite or NaN, and the largest at least
// 2^-537, whose square does not underflow.  From the exponents.
__device__ __forceinline__ bool has_direction(const r4<double>& p) {
  const int m = max(max(__double2hiint(p.x) & 0x7fffffff, __double2hiint(p.y) & 0x7fffffff), __double2hiint(p.z) & 0x7fffffff);
  return m >= 486 << 20 && m < 2047 << 20;
}

// Counterterms, error scale and regions of one point, from its momenta k, in float64; T is the
// precision of the evaluation it belongs to.  The float64 pipe bounds every kernel that runs
// this, so what the centre-of-mass frame of massless, back-to-back beams implies is put in by
// hand (65,536 e+e- -> u ubar g points, where this is most of the work: 187 -> 128 us):
//  * initial state (gluon leg 4, sectors: beam 0, beam 1): the pair recoils with mass^2
//    s (1 - xi) and momentum -k_g, its rest-frame direction n is kept.  The soft Born is the
//    pair at sqrt(s) along n, the collinear one has a beam scaled by 1 - xi and the pair
//    boosted along the beam; both are known from n and the velocities beta(s),
//    beta(s (1 - xi)).  The two sectors' collinear Borns are one 2 -> 2 configuration boosted
//    along the beam, so the Borns, plain and polarised along the gluon's transverse direction,
//    are shared; the rapidity cuts are not;
//  * final state (sectors: partner leg 2 or 3): a sector's soft and soft-collinear limits are
//    the same number, and its Born depends on the cosine of the partner to the beam alone.
// Close to a collinear limit the last bits of a weight are those of 1 - y_j = d_j as formed
// here, which the eikonal denominators p_j.q carry again, rounded differently; where the two
// meet, their ratio is kept as it comes out.  A float64 handle also keeps the beams' own eikonal
// terms (p^2 = 0 up to rounding) and the final state's eikonal factor (1 up to rounding): its weights
// serve as the reference for others and are held, to 1e-12 where the inputs fix them, to a
// term-by-term evaluation in float64, which carries these factors.  A mixed handle leaves them out.
template <int PID, typename T>
__device__ __forceinline__ PointTerms point_terms(const r4<double>* k, const KParams& kp) {
  constexpr bool F64 = !std::is_same<T, float>::value;
  PointTerms o{};
  const double rs = k[0].e + k[1].e, irs = 1.0 / rs;
  const double g2 = kp.cp.gs * kp.cp.gs;
  o.real = !kp.cut.mask || pass_cuts<PID>(k, kp.cut);
  const double xi = 2.0 * k[4].e * irs, z = 1.0 - xi;
  double q[3];
  unit3(k[4], q[0], q[1], q[2]);
  const double d_cut = kp.delta;  // y_j > 1 - delta  <=>  1 - y_j < delta
  const bool soft_xi = below(xi, kp.xi_cut), near_xi = below(xi, kp.xi_thr);
  double d0, d1;
  bool beams = true;  // both have a direction (known from d0 and d1 unless said otherwise)
  if constexpr (PID == P_EE_UUG) {
    double n[2][3];
    unit3(k[2], n[0][0], n[0][1], n[0][2]);
    unit3(k[3], n[1][0], n[1][1], n[1][2]);
    double d[2], c[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      o.y[j] = q[0] * n[j][0] + q[1] * n[j][1] + q[2] * n[j][2];
      d[j] = 1.0 - o.y[j];
      c[j] = 2.0 * irs * (k[0].x * n[j][0] + k[0].y * n[j][1] + k[0].z * n[j][2]);
    }
    d0 = d[0];
    d1 = d[1];
    const double s = rs * rs;
    // 1 / (xi^2 d_j K_j), K_j = s z / (16 pi^3 (2 - xi d_j)^2), from one reciprocal
    const double r = 16.0 * PI * PI * PI / (s * z * xi * xi * d0 * d1 * (d0 + d1));
    const double sum = d0 + d1;
    const double cs = g2 * (8.0 * CF_ / (64.0 * PI * PI * PI)), cc = 0.5 * cs * (1.0 + z * z);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const double t = 2.0 - xi * d[j];
      const double B = (16.0 / 3.0) * kp.born_scale * (1.0 + c[j] * c[j]);
      bool pass = true;
      if (kp.cut.mask) {
        const double e = 0.5 * rs;
        const r4<double> a{e, e * n[j][0], e * n[j][1], e * n[j][2]}, m{e, -a.x, -a.y, -a.z};
        const r4<double> kb[4] = {k[0], k[1], j == 0 ? a : m, j == 0 ? m : a};
        pass = pass_cuts<P_EE_UU>(kb, kp.cut);
      }
      const bool th_s = pass && soft_xi, th_c = pass && below(d[j], d_cut);
      const double id = (r * d[1 - j] * sum * t * t) * B;
      double soft = th_s && !th_c ? cs : 0.0;
      if constexpr (F64) {
        // (1 - y)(1 + y)/2 times the eikonal factor of partner and recoiler: 1 up to rounding
        const double e = 0.5 * rs;
        const r4<double> a{e, e * n[j][0], e * n[j][1], e * n[j][2]}, m{e, -a.x, -a.y, -a.z}, qq{1.0, q[0], q[1], q[2]};
        const double c1 = d[j] * 0.5 * (1.0 + o.y[j]) * (mdot(a, m) / (mdot(a, qq) * mdot(m, qq)));
        soft = th_s ? cs * (th_c ? c1 - 1.0 : c1) : 0.0;
      }
      const double x = (th_c ? cc : 0.0) * id, u = soft * id;
      o.w_born -= x + u;
      o.mag_b += fabs(x) + fabs(u);
      o.near |= (th_s && near_xi) || (th_c && below(d[j], kp.y_thr));
      o.need[j] = th_s || th_c;
    }
  } else {
    constexpr bool GG = PID == P_GG_TTG;
    const double mt = kp.cp.mt, is = irs * irs, rho = 4.0 * mt * mt * is;
    double b[3];
    unit3(k[0], b[0], b[1], b[2]);
    o.y[0] = q[0] * b[0] + q[1] * b[1] + q[2] * b[2];
    if constexpr (F64) {
      double b1[3];
      unit3(k[1], b1[0], b1[1], b1[2]);
      o.y[1] = q[0] * b1[0] + q[1] * b1[1] + q[2] * b1[2];
    } else {
      o.y[1] = -o.y[0];
      beams = has_direction(k[1]);
    }
    d0 = 1.0 - o.y[0];
    d1 = 1.0 - o.y[1];
    // the quark's direction in the pair's rest frame (the pair has momentum -k_g)
    const double s = rs * rs, sz = s * z, iM = rsqrt(sz), M = sz * iM, Q0 = rs - k[4].e;
    const double e2 = (k[2].e * Q0 + k[4].x * k[2].x + k[4].y * k[2].y + k[4].z * k[2].z) * iM;
    const double cq = (e2 + k[2].e) / (Q0 + M);
    const r4<double> ks{e2, k[2].x + cq * k[4].x, k[2].y + cq * k[4].y, k[2].z + cq * k[4].z};
    double n[3];
    unit3(ks, n[0], n[1], n[2]);
    const double cb = n[0] * b[0] + n[1] * b[1] + n[2] * b[2];
    const double nq = n[0] * q[0] + n[1] * q[1] + n[2] * q[2];
    const double b2 = 1.0 - rho, ibeta = rsqrt(b2), beta = b2 * ibeta;
    const double iz = 1.0 / z, rhoc = rho * iz, bQ2 = fmax(0.0, 1.0 - rhoc), bQ = sqrt(bQ2);
    bool cut_s = true, cut_c[2] = {true, true};
    if (kp.cut.mask) {
      const double e = 0.5 * rs, pa = e * beta, eQ = 0.5 * M, pQ = eQ * bQ;
      const r4<double> s2{e, pa * n[0], pa * n[1], pa * n[2]}, s3{e, -s2.x, -s2.y, -s2.z};
      const r4<double> tr{eQ, pQ * n[0], pQ * n[1], pQ * n[2]}, tb{eQ, -tr.x, -tr.y, -tr.z};
      cut_s = heavy_pass(s2, kp.cut) && heavy_pass(s3, kp.cut);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const r4<double> Q = j == 0 ? scale(z, k[0]) + k[1] : k[0] + scale(z, k[1]);
        const double Q2 = mdot(Q, Q), iMc = rsqrt(Q2), iqm = 1.0 / (Q.e + Q2 * iMc);
        cut_c[j] = heavy_pass(boost_by(tr, Q, iMc, iqm), kp.cut) && heavy_pass(boost_by(tb, Q, iMc, iqm), kp.cut);
      }
    }
    // soft and collinear Borns: tau_i = (1 -+ v cb) / 2 with v the quark's velocity
    const double hs = 0.5 * beta * cb, t0 = 0.5 - hs, t1 = 0.5 + hs, hc = 0.5 * bQ * cb;
    const Inv22<double> js{0.0, t0, t1, rho}, jc{0.0, 0.5 - hc, 0.5 + hc, rhoc};
    // eikonal factors times d_0 d_1; the beams' c_j = d_j E / (p_j.q) are 1 up to rounding
    const double f2 = 1.0 - beta * nq, f3 = 1.0 + beta * nq, rf = 1.0 / (f2 * f3), i2 = f3 * rf, i3 = f2 * rf;
    const r4<double> qq{1.0, q[0], q[1], q[2]};
    const double a0 = mdot(k[0], qq), a1 = mdot(k[1], qq), ra = 0.5 * rs / (a0 * a1);
    const double c0 = d0 * a1 * ra, c1 = d1 * a0 * ra;
    const double d01 = d0 * d1, u0 = 4.0 * d1 * c0, u1 = 4.0 * d0 * c1;
    const double w[7] = {4.0 * c0 * c1, u0 * t0 * i2, u0 * t1 * i3, u1 * t1 * i2, u1 * t0 * i3,
                         (4.0 - 2.0 * rho) * d01 * rf, rho * d01};
    double w00 = 0.0;
    if constexpr (F64) w00 = (mdot(k[0], k[0]) * (a1 * a1) + mdot(k[1], k[1]) * (a0 * a0)) * d01 / (a0 * a0 * (a1 * a1));
    double vE, vS, xiP;  // vE carries d_0 d_1
    if constexpr (GG) {
      const Couplings unit(1.0, 1.0, mt);
      const BornGG<double> bs = born_gg(js, unit), bc = born_gg(jc, unit);
      auto cE = [&](int pr) { return born_gg_form(bs, kp.tab->Ccorr[0][pr]); };
      // the massive legs' own terms share their correlator (C_F)
      vE = bs.f * (w[0] * cE(1) + w[1] * cE(2) + w[2] * cE(3) + w[3] * cE(5) + w[4] * cE(6) + w[5] * cE(8) +
                   w[6] * (i2 * i2 + i3 * i3) * cE(7));
      if constexpr (F64) vE += bs.f * w00 * cE(0);
      vS = (2.0 * CA_) * born_gg_colour(bs);
      const double pt2 = q[0] * q[0] + q[1] * q[1], ne = n[0] * q[0] + n[1] * q[1];
      const double ne2 = positive(pt2) ? ne * ne / pt2 : n[0] * n[0];
      const double Bp = born_gg_polarised(jc, bc, 0.5 * bQ2 * ne2, unit);
      xiP = 2.0 * CA_ * ((z + xi * xi * z) * born_gg_colour(bc) + 2.0 * xi * xi * iz * Bp);
    } else {
      const double* C = kp.tab->Cqq;
      const double fs = 8.0 * born_qq(js);
      vE = fs * (w[0] * C[1] + w[1] * C[2] + w[2] * C[3] + w[3] * C[5] + w[4] * C[6] + w[5] * C[8] +
                 w[6] * (i2 * i2 * C[7] + i3 * i3 * C[9]));
      if constexpr (F64) vE += fs * w00 * C[0];
      vS = (4.0 * CF_) * fs;
      xiP = CF_ * (1.0 + z * z) * 16.0 * born_qq(jc);
    }
    // G / (2 g^2 / (64 pi^3)) of the soft, collinear and soft-collinear limits, the Borns'
    // couplings and average taken out; K = s bQ / (64 pi^3 beta)
    const double kb = bQ * ibeta;
    const double Gs = -vE, Gc = 2.0 * kb * iz * xiP, Gsc = 2.0 * vS;
    // 1 / (xi^2 d_j K) of both sectors from one reciprocal
    const double pre = 2.0 * g2 * kp.born_scale / (xi * xi * d01 * s * kb);
    const bool th_s = soft_xi && cut_s;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const bool th_c = below(j == 0 ? d0 : d1, d_cut), th_cc = th_c && cut_c[j];
      const double id = pre * (j == 0 ? d1 : d0);
      const double a = th_cc ? Gc * id : 0.0, c = th_s ? (th_c ? Gs - Gsc : Gs) * id : 0.0;
      o.w_born -= a + c;
      // error scale: the collinear term, and the soft pair (whose Borns are shared)
      o.mag_b += fabs(a) + fabs(c);
      o.near |= (th_s && near_xi) || ((th_cc || (th_s && th_c)) && below(j == 0 ? d0 : d1, kp.y_thr));
      o.need[1] |= th_cc;
    }
    o.need[0] = th_s;
  }
  o.inside = positive(xi) && below(xi, 1.0) && positive(d0) && positive(d1) && beams;
  return o;
}

// One helicity block b of the real matrix element, colour-summed and averaged:
// R = sum over the live blocks.
template <int PID, typename T>
__device__ __forceinline__ double real_block_value(const Kin<PID, T>& K, int b, const KParams& kp) {
  return (double)block_sum<PID, T>(K, b, kp) * kp.real_scale;
}

// W and its error scale from a point's terms and R.
__device__ __forceinline__ RealSubOut combine_point(const PointTerms& t, double R) {
  if (!t.inside) return RealSubOut{0.0, 0.0, 0.0, {t.y[0], t.y[1]}, false};
  const double r = t.real ? R : 0.0, magR = fabs(r);
  return RealSubOut{r + t.w_born, magR, t.mag_b, {t.y[0], t.y[1]}, t.near};
}

// `items` (optional): filled with the terms and block values on group lane 0 (every lane of
// the group must pass it or none).
struct RealItems {
  PointTerms t;
  double v[MAX_BLOCKS];  // bulk-precision values of the R blocks
};
template <int PID, typename T, int LPE>
__device__ __forceinline__ RealSubOut real_sub_event(const double* __restrict__ p, long n, long ev, const KParams& kp,
                                                     int lane, unsigned mask, RealItems* items = nullptr) {
  constexpr int NEXT = Proc<PID>::NEXT;
  constexpr int NB = RealLayout<PID>::NB;
  constexpr int NBL = (NB + LPE - 1) / LPE;  // real blocks per lane
  r4<double> k[NEXT];
  load_event<NEXT>(p, n, ev, k);
  // real matrix element; lane l holds blocks l NBL, l NBL + 1, ... (one copy of the block
  // code: the loop is not unrolled)
  double blk[NBL];
  double mine = 0.0;
  {
    const Kin<PID, T> K = prepare<PID, T>(k, unit_couplings(kp.cp));
#pragma unroll 1
    for (int i = 0; i < NBL; ++i) {
      const int b = lane * NBL + i;
      const double v = b < NB ? real_block_value<PID, T>(K, b, kp) : 0.0;
      blk[i] = v;
      mine += v;
    }
  }
  const double R = group_sum<LPE>(mine, mask);
  const PointTerms t = point_terms<PID, T>(k, kp);
  if (items) {
    // every block value to lane 0 (block b lives on lane b / NBL, slot b % NBL)
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      double x = 0.0;
#pragma unroll
      for (int i = 0; i < NBL; ++i)
        if (i == b % NBL) x = blk[i];
      if constexpr (LPE > 1) x = __shfl_sync(mask, x, b / NBL, LPE);
      items->v[b] = x;
    }
    items->t = t;
  }
  return combine_point(t, R);
}

// Item rescue: a flagged point re-evaluates items in float64, largest error scale first,
// until the float32 error left is at most this fraction of tol |W| -- half the budget of
// an unflagged point, so that flagged points add little to the tail that the calibration
// of me_eps bounds (2^20 flat points: the 99.9th percentile of the error stays at 8.2e-6
// (g g -> t tbar g), 8.0e-6 (u ubar -> t tbar g) and 7.3e-6 (e+e- -> u ubar g) of tol =
// 1e-5; at 1 it reaches 1.5e-5).  A compile-time setting, like ME_MINB, for calibration
// studies: -DME_ITEM_BUDGET=x.
#ifndef ME_ITEM_BUDGET
#define ME_ITEM_BUDGET 0.5
#endif
constexpr double kItemBudget = ME_ITEM_BUDGET;

// Stability test of a bulk-precision result: the error of W is ~ me_eps x (error
// scale); the float32 error of the real's amplitudes per unit scale grows towards the
// collinear limit, as 1 + sqrt(rho_0 / rho) with rho = min_j (1 - y_j), rho_0 = 0.01.
// The counterterms' Born values are evaluated at regular 2 -> 2 kinematics, whose error
// does not grow there: error ~ me_eps x (growth x real part + Born part).
__device__ __forceinline__ double error_growth(const RealSubOut& r) {
  const float rho = fmaxf(fminf((float)(1.0 - r.y[0]), (float)(1.0 - r.y[1])), 1e-30f);
  return 1.0 + (double)sqrtf(0.01f / rho);
}
// The test itself in float64 (two operations; magnitudes compare like their bits, off the
// float64 pipe): weights have no fixed scale, and float32 would compare 0 <= 0 or inf <= inf
// where they leave its range, and call such a point stable.  A NaN is unstable.
__device__ __forceinline__ bool unstable_point(const RealSubOut& r, const KParams& kp, double g) {
  const double s = r.magR * g + r.magB;
  return r.near || below(kp.tol_eps * fabs(r.W), s) || is_nan(s);
}

__device__ __forceinline__ bool unstable_point(const RealSubOut& r, const KParams& kp) {
  return unstable_point(r, kp, error_growth(r));
}

// Blocks of a flagged point to re-evaluate in float64 (bit b: block b).  Largest error scale
// first, until the scale of what is left is within kItemBudget of what the test allows.  The
// Born part is float64 already but keeps its place in the order (without growth): what it no
// longer adds to the error is a margin.  Points inside the thresholds take every block, and so
// do those with a NaN.
template <int PID>
__device__ __forceinline__ unsigned rescue_mask(const RealSubOut& r, bool real, const double* v, const KParams& kp,
                                                double g) {
  constexpr int NB = RealLayout<PID>::NB;
  constexpr unsigned all = (1u << NB) - 1u;
  if (!real) return 0;
  double rest = r.magR * g + r.magB;
  if (r.near || is_nan(rest)) return all;
  double e[NB + 1];
#pragma unroll
  for (int b = 0; b < NB; ++b) e[b] = g * fabs(v[b]);
  e[NB] = r.magB;
  const double budget = kItemBudget * (kp.tol_eps * fabs(r.W));
  unsigned m = 0;
#pragma unroll
  for (int k = 0; k <= NB; ++k) {
    if (!below(budget, rest)) break;
    int pick = 0;
    double best = -1.0;
#pragma unroll
    for (int b = 0; b <= NB; ++b)
      if (!(m >> b & 1u) && below(best, e[b])) {
        best = e[b];
        pick = b;
      }
    m |= 1u << pick;
    rest -= best;
  }
  return m & all;
}

// Buffers of the item rescue (structure of arrays, capacity `cap` points): a record for
// each flagged point with blocks to re-evaluate -- ev[slot], pend[slot] (its blocks still
// to come), wb[slot] = W_B, v[b * cap + slot] -- and the item list,
// slot * 4 + b, from the front (where RealLayout::BY_PARITY asks for it, odd blocks from the
// back, so that a warp runs one kind).  Counters (`counts`): [0] flagged points, [2] and [7]
// blocks listed from the front and the back, [3] flagged points with
// an active counterterm, [4] / [5] their active Born configurations (soft, collinear, or
// sector 1, 2), [6] records; [1] is the queued kernel's tile counter.
struct ItemBufs {
  int* ev;
  int* pend;
  double* wb;
  double* v;
  int* list_r;
  long cap;
};

// Record a flagged point and list its blocks: called by the flagged lanes of a warp together
// (one atomic per warp and counter).
template <int PID>
__device__ __forceinline__ void append_flagged(int* __restrict__ counts, const ItemBufs& ib, long ev, double w_born,
                                               const bool* need, const double* v, unsigned m) {
  constexpr int NB = RealLayout<PID>::NB;
  const unsigned am = __activemask();
  const int wl = threadIdx.x & 31, leader = __ffs(am) - 1;
  const unsigned lt = (1u << wl) - 1u;
  const unsigned rec = __ballot_sync(am, m != 0);
  const unsigned c0 = __ballot_sync(am, need[0]), c1 = __ballot_sync(am, need[1]);
  constexpr bool SPLIT = RealLayout<PID>::BY_PARITY;
  unsigned bal[NB];
  int tot[2] = {0, 0};
#pragma unroll
  for (int b = 0; b < NB; ++b) tot[SPLIT ? b & 1 : 0] += __popc(bal[b] = __ballot_sync(am, m >> b & 1u));
  int base = 0, rbase[2] = {0, 0};
  if (wl == leader) {
    atomicAdd(counts, __popc(am));
    if (c0 | c1) atomicAdd(counts + 3, __popc(c0 | c1));
    if (c0) atomicAdd(counts + 4, __popc(c0));
    if (c1) atomicAdd(counts + 5, __popc(c1));
    if (rec) {
      base = atomicAdd(counts + 6, __popc(rec));
      if (tot[0]) rbase[0] = atomicAdd(counts + 2, tot[0]);
      if (tot[1]) rbase[1] = atomicAdd(counts + 7, tot[1]);
    }
  }
  const int slot = __shfl_sync(am, base, leader) + __popc(rec & lt);
  rbase[0] = __shfl_sync(am, rbase[0], leader);
  if (SPLIT) rbase[1] = __shfl_sync(am, rbase[1], leader);
  if (m) {
    ib.ev[slot] = (int)ev;
    ib.pend[slot] = __popc(m);
    ib.wb[slot] = w_born;
#pragma unroll
    for (int b = 0; b < NB; ++b) ib.v[b * ib.cap + slot] = v[b];
  }
  // ordered by block, then lane
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int half = SPLIT ? b & 1 : 0;
    if (m >> b & 1u) {
      const long at = rbase[half] + __popc(bal[b] & lt);
      ib.list_r[half ? MAX_BLOCKS * ib.cap - 1 - at : at] = slot * 4 + b;
    }
    rbase[half] += __popc(bal[b]);
  }
}

// out[i] = wgt[i] * W(p_i).  In the bulk precision with kp.flag_unstable set, the
// points failing the stability test are appended to resc_list; the float64 launch over
// that list (idx, count) re-evaluates them.  With kp.item_rescue set as well, each
// flagged point gets a record and its float64 blocks are listed instead.
template <int PID, typename T, int LPE>
__global__ void __launch_bounds__(128, ME_MINB) k_real_sub(const double* __restrict__ p, const double* __restrict__ wgt,
                                                  long n, double* __restrict__ out, KParams kp,
                                                  const int* __restrict__ idx, const int* __restrict__ count,
                                                  int* __restrict__ resc_list, int* __restrict__ resc_count,
                                                  ItemBufs ib) {
  const long gid = ((long)blockIdx.x * blockDim.x + threadIdx.x) / LPE;
  const int lane = threadIdx.x % LPE;
  const long nev = count ? (long)*count : n;
  if (gid >= nev) return;
  const long ev = idx ? (long)idx[gid] : gid;
  RealItems it;
  const bool want = kp.flag_unstable && kp.item_rescue;
  const RealSubOut r = real_sub_event<PID, T, LPE>(p, n, ev, kp, lane, group_mask<LPE>(), want ? &it : nullptr);
  if (lane == 0) {
    out[ev] = (wgt ? wgt[ev] : 1.0) * r.W;
    if (kp.flag_unstable && unstable_point(r, kp)) {
      if (!kp.item_rescue) {
        const int slot = atomicAdd(resc_count, 1);
        resc_list[slot] = (int)ev;
      } else {
        append_flagged<PID>(resc_count, ib, ev, it.t.w_born, it.t.need, it.v,
                            rescue_mask<PID>(r, it.t.real, it.v, kp, error_growth(r)));
      }
    }
  }
}

// Float64 evaluation of the listed blocks (grid-stride over the list, its length read on the
// device).  The lane that delivers a record's last block recombines its W: the values are
// published with a fence before the count, and read from L2 after it.
// A list that leaves half the lanes idle takes the time of one block's serial float64 chain
// (a warp's float64 instruction holds its scheduler's pipe for 64 cycles, however few lanes it
// has): g g -> t tbar g then gives the two top spins of a block to lanes of different warps,
// which repeat the currents (calls of 4099 points, 68 -> 53 us each with several in flight).  The
// line is where both halves of every block still have lanes of their own; past it the repeated
// work would cost a second round.  Both ways add the spins' sums in the same order.
template <int PID>
__global__ void __launch_bounds__(128, ME_MINB) k_rescue_items(const double* __restrict__ p,
                                                               const double* __restrict__ wgt, long n,
                                                               double* __restrict__ out, KParams kp,
                                                               const int* __restrict__ counts, ItemBufs ib) {
  constexpr int NEXT = Proc<PID>::NEXT, NB = RealLayout<PID>::NB;
  __shared__ double part[64];
  const long stride = (long)gridDim.x * blockDim.x, front = counts[2], nit = front + counts[7];
  const bool split = PID == P_GG_TTG && 2 * nit <= stride;  // the same in every block
  const int half = split ? threadIdx.x >> 6 : 0, lane = split ? threadIdx.x & 63 : threadIdx.x;
  for (long t = split ? (long)blockIdx.x * 64 + lane : (long)blockIdx.x * blockDim.x + lane;; t += stride) {
    const bool live = t < nit;
    if (!split && !live) break;
    int slot = 0, b = 0, ev = 0;
    double s[2] = {0.0, 0.0};
    if (live) {
      const int item = ib.list_r[t < front ? t : MAX_BLOCKS * ib.cap - 1 - (t - front)];
      slot = item >> 2;
      b = item & 3;
      ev = ib.ev[slot];
      r4<double> k[NEXT];
      load_event<NEXT>(p, n, ev, k);
      const Kin<PID, double> K = prepare<PID, double>(k, unit_couplings(kp.cp));
      if constexpr (PID == P_GG_TTG) {
        amplitude_block<PID, double>(
            K, live_block_hel<PID>(b), unit_couplings(kp.cp),
            [&](int r, const cx<double>* J) { s[r & 1] += colour_sum<PID, double>(kp.tab, J); },
            split ? 1u << half : 3u);
      } else {
        s[0] = block_sum<PID, double>(K, b, kp);
      }
    }
    if (split) {
      if (half) part[lane] = s[1];
      __syncthreads();
      if (half || !live) return;
      s[1] = part[lane];
    }
    __stcg(ib.v + b * ib.cap + slot, (s[0] + s[1]) * kp.real_scale);
    __threadfence();
    if (atomicSub(ib.pend + slot, 1) == 1) {
      __threadfence();
      double R = 0.0;
#pragma unroll
      for (int i = 0; i < NB; ++i) R += __ldcg(ib.v + i * ib.cap + slot);
      out[ev] = (wgt ? wgt[ev] : 1.0) * (R + ib.wb[slot]);
    }
    if (split) return;
  }
}

// Mixed-precision subtracted real in one launch, with the float64 re-evaluation queued
// per block (the per-term queues of the event-parallel design, here for the unstable
// points).  A persistent grid takes tiles of QT points from a device counter.  Each
// point is evaluated in float32, one lane per point; a point that fails the stability
// test goes to a queue in shared memory.  Whenever the queue holds QT points the block
// re-evaluates them in float64, one lane per point with every lane busy, while the
// SM's other blocks run float32 tiles next to it.  The remainder is drained at the
// end.  A point's result depends only on the point, so the output does not depend on
// which block took which tile.  `count` (optional, device): number of points.
// `tiles` must be zero at launch; `resc_count` receives the number re-evaluated.
constexpr int QT = 128;

template <int PID>
__global__ void __launch_bounds__(QT, ME_MINB) k_real_sub_queued(const double* __restrict__ p,
                                                        const double* __restrict__ wgt, long n,
                                                        double* __restrict__ out, KParams kp,
                                                        const int* __restrict__ count, int* __restrict__ tiles,
                                                        int* __restrict__ resc_count) {
  __shared__ int q[2 * QT];
  __shared__ int qn, tile;
  const long nev = count ? (long)*count : n;
  const long ntile = (nev + QT - 1) / QT;
  const unsigned self = 1u << (threadIdx.x & 31u);
  if (threadIdx.x == 0) qn = 0;
  int done = 0;
  for (;;) {
    if (threadIdx.x == 0) tile = atomicAdd(tiles, 1);
    __syncthreads();
    const long t = tile;
    const bool last = t >= ntile;  // uniform over the block
    if (!last) {
      const long ev = t * QT + threadIdx.x;
      if (ev < nev) {
        const RealSubOut r = real_sub_event<PID, float, 1>(p, n, ev, kp, 0, self);
        out[ev] = (wgt ? wgt[ev] : 1.0) * r.W;
        if (unstable_point(r, kp)) q[atomicAdd(&qn, 1)] = (int)ev;
      }
    }
    __syncthreads();
    // a full queue, or the rest once the tiles are gone (then fewer than QT are left)
    const int qc = qn;  // uniform: qn is not written between this read and the barriers below
    if (qc >= QT || (last && qc > 0)) {
      const int take = qc < QT ? qc : QT;
      if ((int)threadIdx.x < take) {
        const int e = q[threadIdx.x];
        const RealSubOut r = real_sub_event<PID, double, 1>(p, n, e, kp, 0, self);
        out[e] = (wgt ? wgt[e] : 1.0) * r.W;
      }
      const int rest = qc - take;  // < QT: at most QT - 1 were left before this tile
      __syncthreads();
      if ((int)threadIdx.x < rest) q[threadIdx.x] = q[QT + threadIdx.x];
      done += take;
      __syncthreads();
      if (threadIdx.x == 0) qn = rest;  // ordered before any append by the next barrier
    }
    if (last) break;
  }
  if (threadIdx.x == 0 && done > 0) atomicAdd(resc_count, done);
}

// ---------------------------------------------------------------- per-term queues
// The variant of Algorithm 2 discussed after it (Sec. 4.3): rather than evaluating every
// term of every point and masking the ones whose cuts fail, a float64 pass (k_terms) maps
// each point, decides its cuts and counterterm regions, adds up its counterterms (closed
// forms, evaluated where they are needed) and queues the real matrix element if it passes
// its cuts; points without one are finished there.  k_term_reals evaluates the queued reals
// one lane each and combines W, in mixed precision with the stability test and the records
// and float64 items of the flagged points, as the masked evaluation (k_rescue_items follows).
// A queued real carries 24 B: its point with the active configurations, W_B, the Born error
// scale, and the error growth (negative for points inside the thresholds).
struct TermBufs {
  int* ev;      // [cap] point of the record; bits 29, 30: active Born configurations
  float* grow;  // [cap] error growth factor of the stability test, negative: near
  double* a;    // [2][cap] W_B, Born error scale
  int* cnt;     // records, zero at launch
  long cap;
};

// Reserve `c` consecutive entries of counter `ctr` for each lane of a full warp (every
// lane calls it; c = 0 reserves nothing): one atomic per warp.  Returns the lane's base.
__device__ __forceinline__ int warp_reserve(int* ctr, int c) {
  const int lane = threadIdx.x & 31;
  int incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  int base = 0;
  if (lane == 31 && total > 0) base = atomicAdd(ctr, total);
  base = __shfl_sync(0xffffffffu, base, 31);
  return base + incl - c;
}

// Float64 pass of the per-term queues: one thread per point.  `pc` (optional, device memory,
// same layout as p): the momenta are copied there, so that the item kernels read device
// memory when p is host memory read in place over the CPU-GPU link (p is then read once).
template <int PID, typename T>
__global__ void __launch_bounds__(128) k_terms(const double* __restrict__ p, const double* __restrict__ wgt, long n,
                                               double* __restrict__ out, KParams kp, const int* __restrict__ count,
                                               TermBufs tb, int* __restrict__ counts, ItemBufs ib,
                                               double* __restrict__ pc) {
  constexpr int NEXT = Proc<PID>::NEXT;
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long nev = count ? (long)*count : n;
  const bool act = i < nev;
  r4<double> k[NEXT];
  if (act) {
    load_event<NEXT>(p, n, i, k);
    if (pc) {
#pragma unroll
      for (int l = 0; l < NEXT; ++l) {
        pc[(0L * NEXT + l) * n + i] = k[l].e;
        pc[(1L * NEXT + l) * n + i] = k[l].x;
        pc[(2L * NEXT + l) * n + i] = k[l].y;
        pc[(3L * NEXT + l) * n + i] = k[l].z;
      }
    }
  } else {
#pragma unroll
    for (int l = 0; l < NEXT; ++l) k[l] = r4<double>{1.0, 0.0, 0.0, 0.0};
  }
  const PointTerms t = point_terms<PID, T>(k, kp);
  const bool rec = act && t.inside && t.real;
  const int slot = warp_reserve(tb.cnt, rec ? 1 : 0);
  const RealSubOut r = combine_point(t, 0.0);
  if (rec) {
    const float g = (float)error_growth(r);
    tb.ev[slot] = (int)i | (t.need[0] ? 1 << 29 : 0) | (t.need[1] ? 1 << 30 : 0);
    tb.grow[slot] = t.near ? -g : g;
    tb.a[slot] = t.w_born;
    tb.a[tb.cap + slot] = t.mag_b;
  } else if (act) {
    // no real matrix element: finished (a flagged one is float64 already)
    out[i] = r.W == 0.0 ? 0.0 : (wgt ? wgt[i] : 1.0) * r.W;
    if (kp.flag_unstable && t.inside && unstable_point(r, kp)) {
      const double none[MAX_BLOCKS] = {};
      append_flagged<PID>(counts, ib, i, 0.0, t.need, none, 0);
    }
  }
}

// The queued reals, one lane each, in precision T (grid-stride, their number read on the
// device), W and the stability test.
template <int PID, typename T>
__global__ void __launch_bounds__(128, ME_MINB) k_term_reals(const double* __restrict__ p,
                                                             const double* __restrict__ wgt, long n,
                                                             double* __restrict__ out, KParams kp, TermBufs tb,
                                                             int* __restrict__ counts, ItemBufs ib) {
  constexpr int NEXT = Proc<PID>::NEXT, NB = RealLayout<PID>::NB;
  const long nr = *tb.cnt;
  for (long slot = (long)blockIdx.x * blockDim.x + threadIdx.x; slot < nr; slot += (long)gridDim.x * blockDim.x) {
    const int code = tb.ev[slot], ev = code & 0x1fffffff;
    r4<double> k[NEXT];
    load_event<NEXT>(p, n, ev, k);
    double v[NB], R = 0.0;
    {
      const Kin<PID, T> K = prepare<PID, T>(k, unit_couplings(kp.cp));
#pragma unroll 1
      for (int b = 0; b < NB; ++b) R += (v[b] = real_block_value<PID, T>(K, b, kp));
    }
    const double wb = tb.a[slot], W = R + wb;
    out[ev] = (wgt ? wgt[ev] : 1.0) * W;
    if (kp.flag_unstable) {
      const double g = tb.grow[slot];
      const RealSubOut r{W, fabs(R), tb.a[tb.cap + slot], {0.0, 0.0}, g < 0.0};
      if (unstable_point(r, kp, fabs(g))) {
        const bool need[2] = {(code >> 29 & 1) != 0, (code >> 30 & 1) != 0};
        append_flagged<PID>(counts, ib, ev, wb, need, v, rescue_mask<PID>(r, true, v, kp, fabs(g)));
      }
    }
  }
}

// Tree-level entries with per-term queues: the points that pass the cuts are listed
// (list, *listed); the others get weight 0.
template <int PID>
__global__ void __launch_bounds__(128) k_cut_list(const double* __restrict__ p, long n, const int* __restrict__ count,
                                                  double* __restrict__ out, KParams kp, int* __restrict__ list,
                                                  int* __restrict__ listed) {
  constexpr int NEXT = Proc<PID>::NEXT;
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long nev = count ? (long)*count : n;
  bool pass = false;
  if (i < nev) {
    r4<double> k[NEXT];
    load_event<NEXT>(p, n, i, k);
    pass = pass_cuts<PID>(k, kp.cut);
    if (!pass) out[i] = 0.0;
  }
  const int at = warp_reserve(listed, pass ? 1 : 0);
  if (pass) list[at] = (int)i;
}

// ---------------------------------------------------------------- launch registry
struct LaunchArgs {
  const double* p;
  const double* wgt;
  long n;
  double* out;
  KParams kp;
  const int* idx;    // optional event list (rescue), length *count on the device
  const int* count;  // optional number of events, read on the device (events 0..*count-1 without idx)
  int* resc_list;    // real kernel in bulk precision: unstable points are appended here
  int* resc_count;   // counters: [1] the queued kernel's tiles, the others as in ItemBufs
  ItemBufs items;    // item rescue records and lists
  long groups;       // number of event groups to launch (n, or the list capacity)
  int* tiles;        // queued kernel: tile counter, zero at launch
  int* ticket;       // tree kernels: counter that they set to zero (the reduction's), or null
  double* p_copy;    // per-term queues: device copy of p made by k_terms (p in host memory), or null
};
enum KernelKind : int { K_TREE = 0, K_REAL = 1 };

template <int PID, typename T, int LPE>
cudaError_t launch_one(int kind, const LaunchArgs& a, cudaStream_t st) {
  (void)cudaGetLastError();  // the launch status below must not report an earlier call's error
  const int threads = 128;
  const long total = a.groups * LPE;
  const long blocks = (total + threads - 1) / threads;
  if (blocks <= 0) return cudaSuccess;
  if (kind == K_TREE) {
    if constexpr (PID == P_GG_TTGG && std::is_same<T, float>::value) {
      static_assert(LPE == 4, "four lanes per event");
      static bool attr_set[64] = {};
      int dev = 0;
      cudaGetDevice(&dev);
      if (dev < 64 && !attr_set[dev]) {
        cudaFuncSetAttribute(k_tree_tt4f<PID>, cudaFuncAttributeMaxDynamicSharedMemorySize, TT4_SMEM);
        attr_set[dev] = true;
      }
      const long tb = (total + TT4_THREADS - 1) / TT4_THREADS;
      k_tree_tt4f<PID><<<(unsigned)tb, TT4_THREADS, TT4_SMEM, st>>>(a.p, a.wgt, a.n, a.out, a.kp, a.idx, a.count, a.ticket);
    } else if constexpr (closed_tree<PID>()) {
      if constexpr (LPE != 1) return launch_one<PID, T, 1>(kind, a, st);
      else k_tree_closed<PID, T><<<(unsigned)((a.groups + 255) / 256), 256, 0, st>>>(a.p, a.wgt, a.n, a.out, a.kp, a.idx, a.count, a.ticket);
    } else if constexpr (PID == P_GG_TTGG) {
      constexpr int lg = LPE == 1 ? 0 : LPE == 2 ? 1 : LPE == 4 ? 2 : 3;
      k_tree_tt4<PID><<<(unsigned)blocks, threads, 0, st>>>(a.p, a.wgt, a.n, a.out, a.kp, a.idx, a.count, a.ticket, lg);
    } else {
      k_tree<PID, T, LPE><<<(unsigned)blocks, threads, 0, st>>>(a.p, a.wgt, a.n, a.out, a.kp, a.idx, a.count, a.ticket);
    }
  } else {
    if constexpr (PID == P_EE_UUG || PID == P_GG_TTG || PID == P_UU_TTG)
      k_real_sub<PID, T, LPE><<<(unsigned)blocks, threads, 0, st>>>(a.p, a.wgt, a.n, a.out, a.kp, a.idx, a.count,
                                                                       a.resc_list, a.resc_count, a.items);
    else
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// The item rescue after a bulk-precision launch: float64 items with their recombination.  A
// persistent grid (resident blocks x SMs, found once per device) walks the list, whose
// length is read on the device.
template <int PID>
cudaError_t launch_items_one(const LaunchArgs& a, cudaStream_t st) {
  (void)cudaGetLastError();
  static std::atomic<int> resident[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  int g = resident[dev].load(std::memory_order_relaxed);
  if (g == 0) {
    int per = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_rescue_items<PID>, 128, 0);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    g = (per > 0 ? per : 1) * (sms > 0 ? sms : 1);
    resident[dev].store(g, std::memory_order_relaxed);
  }
  const long cap_blocks = (a.items.cap * 4 + 127) / 128;
  const unsigned gx = (unsigned)std::max(1L, std::min<long>(g, cap_blocks));
  k_rescue_items<PID><<<gx, 128, 0, st>>>(a.p_copy ? a.p_copy : a.p, a.wgt, a.n, a.out, a.kp, a.resc_count, a.items);
  return cudaGetLastError();
}

// per-process launchers (one translation unit each); lpe in {1, 2, 4, 8, 16}
cudaError_t launch_ee(int pid, int kind, bool fp64, int lpe, const LaunchArgs& a, cudaStream_t st);
cudaError_t launch_gg(int pid, int kind, bool fp64, int lpe, const LaunchArgs& a, cudaStream_t st);
cudaError_t launch_ggg(int pid, int kind, bool fp64, int lpe, const LaunchArgs& a, cudaStream_t st);
cudaError_t launch_ggg64(int kind, int lpe, const LaunchArgs& a, cudaStream_t st);
cudaError_t launch_uu(int pid, int kind, bool fp64, int lpe, const LaunchArgs& a, cudaStream_t st);
// float64 items and recombination of the item rescue (one per process family)
cudaError_t launch_items_ee(const LaunchArgs& a, cudaStream_t st);
cudaError_t launch_items_gg(const LaunchArgs& a, cudaStream_t st);
cudaError_t launch_items_uu(const LaunchArgs& a, cudaStream_t st);
// mixed-precision subtracted real with the queued float64 re-evaluation (k_real_sub_queued)
cudaError_t launch_queued(int pid, const LaunchArgs& a, cudaStream_t st);
cudaError_t launch_queued_gg(const LaunchArgs& a, cudaStream_t st);

// One persistent launch of k_real_sub_queued: as many blocks as are resident at once
// (occupancy x SMs, found once per device), at most one per tile.
template <int PID>
cudaError_t launch_queued_one(const LaunchArgs& a, cudaStream_t st) {
  (void)cudaGetLastError();  // the launch status below must not report an earlier call's error
  static std::atomic<int> resident[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  int g = resident[dev].load(std::memory_order_relaxed);
  if (g == 0) {
    int per = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_real_sub_queued<PID>, QT, 0);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    g = (per > 0 ? per : 1) * (sms > 0 ? sms : 1);
    resident[dev].store(g, std::memory_order_relaxed);
  }
  const long ntile = (a.groups + QT - 1) / QT;
  if (ntile <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)(ntile < g ? ntile : g);
  k_real_sub_queued<PID><<<blocks, QT, 0, st>>>(a.p, a.wgt, a.n, a.out, a.kp, a.count, a.tiles, a.resc_count);
  return cudaGetLastError();
}

// Per-term queues: the float64 pass, then the queued reals (in mixed precision the item
// rescue follows, launch_items_*).
template <int PID>
cudaError_t launch_terms_one(bool mixed, const LaunchArgs& a, const TermBufs& tb, cudaStream_t st) {
  (void)cudaGetLastError();
  static std::atomic<int> resident[2][64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  int g = resident[mixed][dev].load(std::memory_order_relaxed);
  if (g == 0) {
    int per = 0, sms = 0;
    e = mixed ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_term_reals<PID, float>, 128, 0)
              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_term_reals<PID, double>, 128, 0);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    g = (per > 0 ? per : 1) * (sms > 0 ? sms : 1);
    resident[mixed][dev].store(g, std::memory_order_relaxed);
  }
  const long blocks = (a.groups + 127) / 128;
  if (blocks <= 0) return cudaSuccess;
  const double* pi = a.p_copy ? a.p_copy : a.p;
  const unsigned gr = (unsigned)std::min<long>(g, blocks), gt = (unsigned)blocks;
  if (mixed) {
    k_terms<PID, float><<<gt, 128, 0, st>>>(a.p, a.wgt, a.n, a.out, a.kp, a.count, tb, a.resc_count, a.items, a.p_copy);
    k_term_reals<PID, float><<<gr, 128, 0, st>>>(pi, a.wgt, a.n, a.out, a.kp, tb, a.resc_count, a.items);
  } else {
    k_terms<PID, double><<<gt, 128, 0, st>>>(a.p, a.wgt, a.n, a.out, a.kp, a.count, tb, a.resc_count, a.items, a.p_copy);
    k_term_reals<PID, double><<<gr, 128, 0, st>>>(pi, a.wgt, a.n, a.out, a.kp, tb, a.resc_count, a.items);
  }
  return cudaGetLastError();
}
cudaError_t launch_terms_ee(bool mixed, const LaunchArgs& a, const TermBufs& tb, cudaStream_t st);
cudaError_t launch_terms_gg(bool mixed, const LaunchArgs& a, const TermBufs& tb, cudaStream_t st);
cudaError_t launch_terms_uu(bool mixed, const LaunchArgs& a, const TermBufs& tb, cudaStream_t st);
// tree entries with per-term queues: list the points that pass the cuts (k_cut_list)
cudaError_t launch_cut_list(int pid, const LaunchArgs& a, int* list, int* listed, cudaStream_t st);

}  // namespace me

#define ME_LPE_SWITCH(PID, T)                                            \
  switch (lpe) {                                                         \
    case 1: return me::launch_one<PID, T, 1>(kind, a, st);               \
    case 2: return me::launch_one<PID, T, 2>(kind, a, st);               \
    case 4: return me::launch_one<PID, T, 4>(kind, a, st);               \
    case 8: return me::launch_one<PID, T, 8>(kind, a, st);               \
    case 16: return me::launch_one<PID, T, 16>(kind, a, st);             \
    default: return cudaErrorInvalidValue;                               \
  }
// g g -> t tbar g g runs at most 8 lanes per event (it has 8 helicity blocks)
#define ME_LPE_SWITCH8(PID, T)                                           \
  switch (lpe) {                                                         \
    case 1: return me::launch_one<PID, T, 1>(kind, a, st);               \
    case 2: return me::launch_one<PID, T, 2>(kind, a, st);               \
    case 4: return me::launch_one<PID, T, 4>(kind, a, st);               \
    case 8: return me::launch_one<PID, T, 8>(kind, a, st);               \
    default: return cudaErrorInvalidValue;                               \
  }
#define ME_PREC_SWITCH(PID)                      \
  if (fp64) {                                    \
    ME_LPE_SWITCH(PID, double)                   \
  } else {                                       \
    ME_LPE_SWITCH(PID, float)                    \
  }
