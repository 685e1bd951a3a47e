// Algorithmic operation count of the amplitude code (host program).
//
// The same templated amplitude routines that the kernels run are instantiated with a
// counting scalar type: every floating-point +, -, *, / and sqrt on the amplitude's
// arithmetic type counts as one operation (a fused multiply-add therefore counts two),
// sign flips and comparisons count zero.  Momentum sums and propagator denominators,
// which the kernels keep in float64, are not counted.  The colour sums are counted
// from their loop structure.  Per event, one helicity of each flipped pair (h, -h) is
// evaluated, as in the kernels, in helicity blocks.  Output: one JSON object with
// operations per helicity (per-event Born count over the helicities evaluated) and per
// event for every process and entry point.
#include <cmath>
#include <cstdio>

#include "me_procs.cuh"

static long g_ops = 0;
struct Flop {
  double v;
  Flop() = default;
  Flop(double x) : v(x) {}
};
inline Flop operator+(Flop a, Flop b) { ++g_ops; return Flop(a.v + b.v); }
inline Flop operator-(Flop a, Flop b) { ++g_ops; return Flop(a.v - b.v); }
inline Flop operator*(Flop a, Flop b) { ++g_ops; return Flop(a.v * b.v); }
inline Flop operator/(Flop a, Flop b) { ++g_ops; return Flop(a.v / b.v); }
inline Flop operator-(Flop a) { return Flop(-a.v); }
inline Flop& operator+=(Flop& a, Flop b) { ++g_ops; a.v += b.v; return a; }
inline bool operator>(Flop a, Flop b) { return a.v > b.v; }
inline bool operator>=(Flop a, Flop b) { return a.v >= b.v; }
inline bool operator==(Flop a, Flop b) { return a.v == b.v; }
inline Flop msqrt(Flop a) { ++g_ops; return Flop(std::sqrt(a.v)); }  // found by argument lookup

using namespace me;

// J^dagger C J per helicity as the kernels evaluate it (me_kernels.cuh: colour_sum): the
// triangular form over the doubled upper triangle, 2 NF^2 + 4 NF flops; for 24 flows
// s4_colour_sum, 96 additions and 2 S4_COEF + 48 multiply-adds
static double colour_flops(int nf) { return nf == 24 ? 96.0 + 4.0 * S4_COEF + 96.0 : 2.0 * nf * nf + 4.0 * nf; }

// one helicity block (me_procs.cuh): amplitudes of four helicities plus their colour sums
template <int PID>
static double block_ops(const r4<double>* p, int hb = 1) {
  const Couplings cp{1.2, 0.3, 173.0};
  const Kin<PID, Flop> K = prepare<PID, Flop>(p, cp);
  g_ops = 0;
  int calls = 0;
  if constexpr (PID == P_EE_UUG) ee_uug_block(K, 0);
  else amplitude_block<PID, Flop>(K, hb, cp, [&](int, const cx<Flop>*) { ++calls; });
  return (double)g_ops + calls * colour_flops(Proc<PID>::NFLOW);
}

// per-event preparation (reciprocal denominators etc. in the amplitude's type)
template <int PID>
static double prep_ops(const r4<double>* p) {
  const Couplings cp{1.2, 0.3, 173.0};
  g_ops = 0;
  const Kin<PID, Flop> K = prepare<PID, Flop>(p, cp);
  (void)K;
  return (double)g_ops;
}

// Born |M|^2 of one event: its closed form, or every block of the half helicity set plus the
// preparation
template <int PID>
static double born_ops(const r4<double>* p) {
  if constexpr (closed_tree<PID>()) {
    g_ops = 0;
    closed_sum<PID, Flop>(p, Couplings{1.2, 0.3, 173.0});
    return (double)g_ops;
  } else {
    double t = prep_ops<PID>(p);
    for (int b = 0; b < n_live_blocks<PID>(); ++b) t += block_ops<PID>(p, live_block_hel<PID>(b));
    return t;
  }
}

int main() {
  // a generic massive 2 -> 4 configuration is enough: the count does not depend on values
  r4<double> p[6] = {{1000, 0, 0, 1000},     {1000, 0, 0, -1000}, {600, 100, 200, 300},
                     {700, -150, -100, 200}, {400, 30, -80, -300}, {300, 20, -20, -200}};
  // Born values of the counterterms: soft (plain and with the eikonal-weighted correlator
  // matrix), collinear (plain and, for g g, polarised along the emission's direction)
  const Couplings cp{1.2, 0.3, 173.0};
  const Flop E[4] = {Flop(1.0), Flop(2.0), Flop(2.0), Flop(1.0)};
  const Inv22<Flop> k = inv22<Flop>(p, Flop(173.0));
  const BornGG<Flop> b2 = born_gg(k, cp);
  g_ops = 0;
  b2.f * born_gg_form(b2, E);
  const double matrix_gg = (double)g_ops;
  g_ops = 0;
  born_uu_matrix(Flop(1.0), E);
  const double matrix_uu = (double)g_ops;
  g_ops = 0;
  born_gg_polarised(k, b2, Flop(50.0), cp);
  const double polarised = (double)g_ops;
  const double soft_gg = born_ops<P_GG_TT>(p) + matrix_gg, coll_gg = born_ops<P_GG_TT>(p) + polarised;
  const double soft_uu = born_ops<P_UU_TT>(p) + matrix_uu, coll_uu = born_ops<P_UU_TT>(p);
  // subtracted real: real blocks and Born values; the collinear term of each g g sector adds
  // its plain and its polarised Born with the splitting kernels (the second sector's sum is
  // not part of a single configuration)
  const double real_ee = born_ops<P_EE_UUG>(p) + 2 * born_ops<P_EE_UU>(p);
  const double real_gg = born_ops<P_GG_TTG>(p) + soft_gg + coll_gg + 3;
  const double real_uu = born_ops<P_UU_TTG>(p) + soft_uu + coll_uu;
  const double b[7] = {born_ops<P_EE_UU>(p),  born_ops<P_EE_UUG>(p), born_ops<P_GG_TT>(p), born_ops<P_GG_TTG>(p),
                       born_ops<P_GG_TTGG>(p), born_ops<P_UU_TT>(p), born_ops<P_UU_TTG>(p)};
  const int nh[7] = {16, 32, 16, 32, 64, 16, 32};
  std::printf("{\"per_helicity\": {\"ee_uu\": %.0f, \"ee_uug\": %.0f, \"gg_tt\": %.0f, \"gg_ttg\": %.0f, "
              "\"gg_ttgg\": %.0f, \"uu_tt\": %.0f, \"uu_ttg\": %.0f},\n",
              2 * b[0] / nh[0], 2 * b[1] / nh[1], 2 * b[2] / nh[2], 2 * b[3] / nh[3], 2 * b[4] / nh[4],
              2 * b[5] / nh[5], 2 * b[6] / nh[6]);
  std::printf(" \"born_per_event\": {\"ee_uu\": %.0f, \"ee_uug\": %.0f, \"gg_tt\": %.0f, \"gg_ttg\": %.0f, "
              "\"gg_ttgg\": %.0f, \"uu_tt\": %.0f, \"uu_ttg\": %.0f},\n",
              b[0], b[1], b[2], b[3], b[4], b[5], b[6]);
  std::printf(" \"real_subtracted_per_event\": {\"ee_uug\": %.0f, \"gg_ttg\": %.0f, \"uu_ttg\": %.0f},\n", real_ee,
              real_gg, real_uu);
  // per-term queues: one Born configuration -- soft, collinear (one sector), or a final-state
  // sector's Born
  std::printf(" \"term_config_per_event\": {\"ee_uug\": [%.0f, %.0f], \"gg_ttg\": [%.0f, %.0f], "
              "\"uu_ttg\": [%.0f, %.0f]},\n", b[0], b[0], soft_gg, coll_gg, soft_uu, coll_uu);
  std::printf(" \"colour_sum_per_event\": {\"gg_ttgg\": %.0f}}\n", 32 * colour_flops(24));
  return 0;
}
