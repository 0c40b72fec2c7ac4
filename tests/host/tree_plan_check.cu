// Host-side check of the tree kernel's compile-time structure against the work
// plan: the CoM partial sum of every joint and the order within a partial are
// those of the plan's dq partition, the shared-memory slots are disjoint and
// fit, and the constants of the prismatic base (Jacobian columns and their
// share of J J^T) match a double-precision evaluation.  Runs on the CPU.
#include <cmath>
#include <cstdio>
#include "../../paper_2604_13323_gb300/csrc/mcp_tree.cuh"
using namespace mcp;
template <class P> int check() {
  int bad = 0;
  static GroupPlan<P> pl;
  if (!make_group_plan<P>(pl, nullptr)) return 1;
  for (int g = 0; g < GG; ++g) {
    bool trunk = false;
    int prev = -1;
    for (int k = 0; k < GMAX_DQ; ++k) {
      const int j = pl.dq_j[g][k];
      if (j < 0) continue;
      if (tree_part(j) != g) bad++, printf("joint %d: partial %d, plan %d\n", j, tree_part(j), g);
      const bool t = j < TR_LEG0 || j == TR_WAIST || j == TR_TORSO;  // limb joints first, then the trunk's, each ascending
      if (trunk && !t) bad++, printf("limb joint %d after the trunk's\n", j);
      if (t == trunk && j < prev) bad++, printf("joint %d out of order\n", j);
      trunk = t;
      prev = j;
    }
  }
  int used[TREE_PAIRS] = {0};
  auto mark = [&](int e, int n) { for (int i = 0; i < n; ++i) { if (e + i < 0 || e + i >= TREE_PAIRS) bad++; else used[e + i]++; } };
  for (int l = 0; l < TR_LEG; ++l) mark(TP_LEG + 8 * l, 8);
  for (int l = 0; l < TR_ARM; ++l) mark(TP_ARM + 8 * l, 8);
  for (int b = 0; b < 3; ++b) mark(TP_BASE + 7 * b, 7);
  mark(TP_UP, 4);
  for (int e = 0; e < TREE_PAIRS; ++e) if (used[e] != 1) bad++, printf("pair %d used %d times\n", e, used[e]);
  if (tree_smem_bytes<P>(TREE_WARPS) > 232448) bad++, printf("shared memory\n");
  // constants: a random base chain and error frames
  static ModelT<float> m{};
  static ModelT<double> m64{};
  unsigned long long x = 0x2545F4914F6CDD1Dull;
  auto rnd = [&]() { x ^= x << 13; x ^= x >> 7; x ^= x << 17; return (double)(x >> 11) / 9007199254740992.0 - 0.5; };
  for (int j = 0; j < P::D; ++j) {
    const double a = 3.0 * rnd(), c = std::cos(a), s = std::sin(a);
    const double X[12] = {1, 0, 0, rnd(), 0, c, -s, rnd(), 0, s, c, rnd()};
    for (int e = 0; e < 12; ++e) m64.X[j][e] = X[e], m.X[j][e] = (float)X[e];
    m64.mass[j] = 1.0 + rnd();
    m64.msub[j] = 3.0 + rnd();
    m.msub[j] = (float)m64.msub[j];
  }
  m64.inv_mass = 0.02;
  m.inv_mass = 0.02f;
  for (int s = 0; s < 2; ++s) for (int e = 0; e < 12; ++e) m64.cPinv[s][e] = rnd(), m.cPinv[s][e] = (float)m64.cPinv[s][e];
  const TreeConst<P> t = make_tree_const<P>(m, m64);
  double jt[2][3][3], jc[3][2];
  for (int i = 0; i < 3; ++i) {
    for (int r = 0; r < 2; ++r) jc[i][r] = m64.msub[i] * m64.inv_mass * t.a[i][r];
    for (int s = 0; s < 2; ++s) for (int r = 0; r < 3; ++r) {
      jt[s][i][r] = 0;
      for (int c = 0; c < 3; ++c) jt[s][i][r] += m64.cPinv[s][4 * r + c] * t.a[i][c];
    }
  }
  double err = 0;
  for (int s = 0; s < 2; ++s) for (int r = 0; r < 3; ++r) for (int c = 0; c < 3; ++c) {
    double ll = 0, lr = 0, cl = 0;
    for (int i = 0; i < 3; ++i) {
      err = std::max(err, std::fabs((s ? t.jt[i][r].y : t.jt[i][r].x) - jt[s][i][r]));
      if (r < 2) err = std::max(err, std::fabs(t.jc[i][r] - jc[i][r]));
      ll += jt[s][i][r] * jt[s][i][c];
      lr += jt[1][i][r] * jt[0][i][c];
      if (r < 2) cl += jc[i][r] * jt[s][i][c];
    }
    if (c <= r) err = std::max(err, std::fabs((s ? t.LL[tri(r, c)].y : t.LL[tri(r, c)].x) - ll));
    err = std::max(err, std::fabs(t.LR[3 * r + c] - lr));
    if (r < 2) err = std::max(err, std::fabs((s ? t.CL[3 * r + c].y : t.CL[3 * r + c].x) - cl));
  }
  if (!(err < 2e-6)) bad++, printf("constants off by %g\n", err);  // a few roundings of O(1) values in FP32
  printf("%s: %d problems\n", P::name, bad);
  return bad;
}
int main() { return check<ProbHumanoid36>() + check<ProbHumanoid36Hull>(); }
