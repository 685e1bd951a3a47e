// Host check of the helicity-block amplitude routines (test program, built by the CPU
// test suite; no GPU needed).  For every point read from stdin it evaluates the
// colour-summed |M|^2 twice with the same templates the kernels use: over every
// helicity one at a time, and over the blocks of one member of each flipped pair
// (doubled; for processes without a block routine, the helicities of those blocks), in float64 and
// in float32.  It prints one line per point:
//   <block fp64> <single fp64> <block fp32> <single fp32>
// With the arguments "kernels <mt>" it prints what the kernels evaluate instead -- block_sum over
// the live blocks, or the closed form of a 2 -> 2 tree, at unit couplings and scaled in
// float64 -- with mt the top mass:
//   <fp64> <fp32>
// Input: "<pid> <n> <n_ext>" then the momenta [4][n_ext][n] (float64, SoA).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "me_internal.h"
#include "me_kernels.cuh"
#include "me_single.cuh"

using namespace me;

template <int PID, typename T>
static double csum(const ColourTables& tab, const cx<T>* J) {
  constexpr int NF = Proc<PID>::NFLOW;
  const double* C = tab.C[PID];
  double t = 0;
  for (int a = 0; a < NF; ++a)
    for (int b = 0; b < NF; ++b)
      t += C[a * NF + b] * ((double)J[a].re * (double)J[b].re + (double)J[a].im * (double)J[b].im);
  return t;
}
// the colour sum as the helicity blocks take it
template <int PID, typename T>
static double bsum(const ColourTables& tab, const cx<T>* J) {
  if constexpr (PID == P_GG_TTGG) {
    T coef[S4_COEF];
    for (int i = 0; i < S4_COEF; ++i) coef[i] = (T)tab.S4[i];
    return (double)s4_colour_sum(coef, [&](int v, int a) { return J[s4_flow(v, a)]; });
  }
  return csum<PID, T>(tab, J);
}

template <int PID, typename T>
static void eval(const ColourTables& tab, const r4<double>* k, const Couplings& cp, double* blk, double* single) {
  constexpr int NH = Proc<PID>::NHEL, NF = Proc<PID>::NFLOW;
  const Kin<PID, T> K = prepare<PID, T>(k, cp);
  double s = 0;
  for (int h = 0; h < NH; ++h) {
    cx<T> J[NF];
    amplitude<PID, T>(K, h, cp, J);
    s += csum<PID, T>(tab, J);
  }
  double b = 0;
  for (int i = 0; i < n_live_blocks<PID>(); ++i) {
    auto add = [&](int, const cx<T>* A) { b += bsum<PID, T>(tab, A); };
    if constexpr (closed_tree<PID>() || PID == P_EE_UUG) single_block<PID, T>(K, live_block_hel<PID>(i), cp, add);
    else amplitude_block<PID, T>(K, live_block_hel<PID>(i), cp, add);
  }
  *blk = 2.0 * b;
  *single = s;
}

template <int PID, typename T>
static double kernel_value(const ColourTables& tab, const r4<double>* k, const Couplings& cp) {
  if constexpr (closed_tree<PID>()) {
    return (double)closed_sum<PID, T>(k, unit_couplings(cp)) * tree_coupling(PID, cp);
  } else {
    KParams kp{};
    kp.cp = cp;
    kp.tab = &tab;
    const Kin<PID, T> K = prepare<PID, T>(k, unit_couplings(cp));
    T acc = T(0);
    for (int b = 0; b < n_live_blocks<PID>(); ++b) acc += block_sum<PID, T>(K, b, kp);
    return 2.0 * (double)acc * tree_coupling(PID, cp);
  }
}

static double g_mt = 0.0;  // > 0: the kernels' values with this top mass

template <int PID>
static void run(const ColourTables& tab, const std::vector<double>& p, int n, int next) {
  const Couplings cp{std::sqrt(4 * M_PI * 0.118), std::sqrt(4 * M_PI / 132.507), g_mt > 0.0 ? g_mt : 173.0};
  for (int i = 0; i < n; ++i) {
    r4<double> k[6];
    for (int l = 0; l < next; ++l)
      k[l] = {p[(0 * next + l) * n + i], p[(1 * next + l) * n + i], p[(2 * next + l) * n + i], p[(3 * next + l) * n + i]};
    if (g_mt > 0.0) {
      std::printf("%.17g %.17g\n", kernel_value<PID, double>(tab, k, cp), kernel_value<PID, float>(tab, k, cp));
      continue;
    }
    double b64, s64, b32, s32;
    eval<PID, double>(tab, k, cp, &b64, &s64);
    eval<PID, float>(tab, k, cp, &b32, &s32);
    std::printf("%.17g %.17g %.17g %.17g\n", b64, s64, b32, s32);
  }
}

int main(int argc, char** argv) {
  if (argc == 3 && std::strcmp(argv[1], "kernels") == 0) g_mt = std::atof(argv[2]);
  static ColourTables tab;
  if (me_internal_build_tables(&tab) != ME_OK) return 1;
  int pid, n, next;
  while (std::scanf("%d %d %d", &pid, &n, &next) == 3) {
    std::vector<double> p((size_t)4 * next * n);
    for (auto& x : p)
      if (std::scanf("%lf", &x) != 1) return 1;
    switch (pid) {
      case P_EE_UU: run<P_EE_UU>(tab, p, n, next); break;
      case P_EE_UUG: run<P_EE_UUG>(tab, p, n, next); break;
      case P_GG_TT: run<P_GG_TT>(tab, p, n, next); break;
      case P_GG_TTG: run<P_GG_TTG>(tab, p, n, next); break;
      case P_GG_TTGG: run<P_GG_TTGG>(tab, p, n, next); break;
      case P_UU_TT: run<P_UU_TT>(tab, p, n, next); break;
      case P_UU_TTG: run<P_UU_TTG>(tab, p, n, next); break;
      default: return 2;
    }
  }
  return 0;
}
