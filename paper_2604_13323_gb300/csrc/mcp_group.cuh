// Reference of the order in which the humanoid's sums are taken, and of the
// state a four-lane Newton step would keep: a work plan that the host checks
// under tests/ build and compare with the library's kernel.  No kernel runs it.
//
// The plan fixes an order for every sum over joints: the limbs are assigned to
// four lanes by longest-first scheduling and the trunk joints to the lane with
// the fewest, the 6-row Gram blocks and refinement residuals run over the
// joints in ascending order, and the CoM sums in one partial per lane (the
// lane's limb joints, then its trunk joints) added pairwise.  The projection
// kernel (one lane per configuration, mcp_tree.cuh) takes its sums in this
// order.  What that kernel uses itself is in mcp_factor.cuh.
#pragma once

#include <algorithm>
#include <vector>

#include "mcp_factor.cuh"
#include "mcp_warp.cuh"

namespace mcp {

// Limits of the work plan, near what the humanoid classes need.
constexpr int GG = 4;            // lanes per configuration
constexpr int GCPW = 32 / GG;    // configurations per warp
constexpr int GMAX_FK = 20;      // FK steps per lane
constexpr int GMAX_CB = 16;      // own joints per lane (subtree moments)
constexpr int GMAX_CR = 16;      // trunk joints
constexpr int GMAX_CH = 4;       // children per joint
constexpr int GMAX_JI = 16;      // Jacobian segments per lane and segment size
constexpr int GMAX_DQ = 20;      // dq joints per lane
constexpr int GMAX_T = 2;        // Gram / refinement tasks per lane and phase
constexpr int GMAX_POOL = 192;   // joint lists of the tasks
constexpr int GMAX_PRE = PRE_JOINTS;  // prismatic root joints placed in closed form

template <class P>
__host__ __device__ constexpr bool grp_pose_like(int c) {
  return P::ckind(c) == K_POSE || P::ckind(c) == K_REL;
}
template <class P>
__host__ __device__ constexpr bool grp_com_like(int c) {
  return P::ckind(c) == K_COM || P::ckind(c) == K_HULL;
}
// Per-constraint data slots: the pose-like constraints (error frame G, point
// x, log-map vector) and the support-hull ones (nearest-edge data) are stored
// per kind, not per constraint, so that the shared state holds no unused rows.
template <class P>
__host__ __device__ constexpr int grp_pslot(int c) {
  int n = 0;
  for (int b = 0; b < c; ++b) n += grp_pose_like<P>(b) ? 1 : 0;
  return n;
}
template <class P>
__host__ __device__ constexpr int grp_hslot(int c) {
  int n = 0;
  for (int b = 0; b < c; ++b) n += P::ckind(b) == K_HULL ? 1 : 0;
  return n;
}
template <class P>
__host__ __device__ constexpr int grp_npose() { return grp_pslot<P>(P::NC); }
template <class P>
__host__ __device__ constexpr int grp_nhull() { return grp_hslot<P>(P::NC); }

// Jacobian segments: (joint j, constraint c) with a structural nonzero, j-major
template <class P>
__host__ __device__ constexpr int grp_nseg_floats() {
  int n = 0;
  for (int j = 0; j < P::D; ++j)
    for (int c = 0; c < P::NC; ++c)
      if (col_sign<P>(c, j) != 0) n += cdim(P::ckind(c));
  return n;
}
// Floats of the 2-row (CoM-like) segments, which come first in the Jacobian's
// space; the subtree moments C_j (3 floats per joint) are kept right after
// them, where the 6-row segments are written once the 2-row ones are built.
template <class P>
__host__ __device__ constexpr int grp_cbase() {
  int n = 0;
  for (int j = 0; j < P::D; ++j)
    for (int c = 0; c < P::NC; ++c)
      if (col_sign<P>(c, j) != 0 && grp_com_like<P>(c)) n += cdim(P::ckind(c));
  return (n + 3) & ~3;
}

// L by columns, packed: rows k .. K-1 of column k from lcol_base(k)
template <int K>
__host__ __device__ constexpr int lcol_base(int k) {
  int o = 0;
  for (int t = 0; t < k; ++t) o += K - t;
  return o;
}

// Tasks of the Gram build and of the refinement residual: row blocks (a, b)
// (b unused for the refinement) and a joint list pool[off, off + n).
struct GrpTask {
  int8_t a, b, n, pad;
  int16_t off, pad2;
};

template <class P>
struct GroupPlan {
  static constexpr int D = P::D, NC = P::NC;
  // 1. FK: per lane and step the joint, the parent source (0: the previous
  // step, 1 / 2: saved slot 0 / 1, 3: the world), the slot to save into and
  // whether this lane writes the joint's data
  int8_t fk_j[GG][GMAX_FK];
  int8_t fk_par[GG][GMAX_FK];
  int8_t fk_save[GG][GMAX_FK];
  int8_t fk_store[GG][GMAX_FK];
  // 2. subtree moments: own joints (reverse preorder) per lane, then the trunk
  int8_t cb_j[GG][GMAX_CB];
  int8_t cr_j[GMAX_CR];
  int8_t child[D][GMAX_CH];
  int8_t roots[4];
  // 4. Jacobian segments per lane: 6-row and 2-row
  int8_t j6_j[GG][GMAX_JI], j6_c[GG][GMAX_JI];
  int8_t j2_j[GG][GMAX_JI], j2_c[GG][GMAX_JI];
  // 7. dq joints per lane (every joint on exactly one lane)
  int8_t dq_j[GG][GMAX_DQ];
  int16_t joff[NC][D];  // segment offset of (j, c), -1: structural zero
  int8_t croff[NC];     // first row of constraint c
  int16_t lcol[GG * 5];  // start of column i of L (shared memory, by columns)
  uint32_t amask[GG * 5];  // row i of J J^T: bit b set if rows i and b share a joint
                           // (the other entries are never written: structural zeros)
  int8_t chull[NC];     // constraint c is the support-hull kind
  int8_t pslot[NC];     // slot of constraint c among the pose-like ones (-1: other kinds)
  int8_t hslot[NC];     // slot of constraint c among the support-hull ones (-1: other kinds)
  int8_t crel[NC];      // pose-like constraint c is the relative pose of two frames
  int8_t cfa[NC], cfb[NC];  // its frames (cfb: the relative pose's second frame, else cfa)
  // 5. Gram phases (6x6, 6x2, 2x6, 2x2 row-block pairs) and 7. refinement
  // phases (6-row, 2-row blocks): tasks per lane.  The diagonal blocks and
  // refinement rows of 2-row constraints (the CoM, over every joint) are
  // summed over the dq partition instead, four lanes and a group reduction.
  GrpTask gt[4][GG][GMAX_T];
  GrpTask rt[2][GG][GMAX_T];
  int8_t pool[GMAX_POOL];
  int n_fk, n_cb, n_cr, n_roots, n_j6, n_j2, n_dq;
  int n_pre;  // leading FK steps of every lane placed in closed form (a prismatic root chain)
  int g_nt[4], g_len[4][GMAX_T];  // per phase: task slots, longest list per slot
  int r_nt[2], r_len[2][GMAX_T];
};

// Host: the plan of problem class P.  Returns false (with the reason) when
// the tree or the constraint stack does not fit the plan's limits.
template <class P>
bool make_group_plan(GroupPlan<P> &pl, const char **why) {
  constexpr int D = P::D, NC = P::NC;
  pl = GroupPlan<P>{};
  auto fail = [&](const char *w) {
    if (why) *why = w;
    return false;
  };
  std::vector<std::vector<int>> ch(D);
  for (int j = 0; j < D; ++j)
    if (P::parent(j) >= 0) ch[P::parent(j)].push_back(j);
  // chains: maximal paths whose inner joints have exactly one child
  std::vector<std::vector<int>> chains;
  std::vector<int> chain_of(D, -1);
  for (int j = 0; j < D; ++j) {
    if (!(P::parent(j) < 0 || ch[P::parent(j)].size() != 1)) continue;
    std::vector<int> c{j};
    while (ch[c.back()].size() == 1) c.push_back(ch[c.back()][0]);
    for (int v : c) chain_of[v] = static_cast<int>(chains.size());
    chains.push_back(c);
  }
  const int nch = static_cast<int>(chains.size());
  // leaf chains to lanes, longest first, onto the least loaded lane
  std::vector<int> owner_c(nch, -2), load(GG, 0), leaves;
  for (int c = 0; c < nch; ++c)
    if (ch[chains[c].back()].empty()) leaves.push_back(c);
  std::stable_sort(leaves.begin(), leaves.end(),
                   [&](int x, int y) { return chains[x].size() > chains[y].size(); });
  for (int c : leaves) {
    const int g = static_cast<int>(std::min_element(load.begin(), load.end()) - load.begin());
    owner_c[c] = g;
    load[g] += static_cast<int>(chains[c].size());
  }
  // inner chains: the lane of all their descendants, else every lane (-1);
  // in preorder a chain's descendants start after it
  for (int c = nch - 1; c >= 0; --c) {
    if (owner_c[c] != -2) continue;
    int o = -2;
    for (int k : ch[chains[c].back()]) {
      const int oc = owner_c[chain_of[k]];
      o = (o == -2) ? oc : (o == oc ? o : -1);
    }
    owner_c[c] = o;
  }
  std::vector<int> owner(D);
  for (int j = 0; j < D; ++j) owner[j] = owner_c[chain_of[j]];
  // 1. FK schedules
  int n_fk = 0;
  for (int g = 0; g < GG; ++g) {
    std::vector<int> js;
    for (int j = 0; j < D; ++j)
      if (owner[j] == g || owner[j] == -1) js.push_back(j);
    if (static_cast<int>(js.size()) > GMAX_FK) return fail("FK schedule too long");
    std::vector<int> slot_of(D, -1);
    int nslot = 0;
    // a parent that is not the previous step must have been saved
    for (size_t k = 0; k < js.size(); ++k) {
      const int p = P::parent(js[k]);
      if (p >= 0 && !(k > 0 && js[k - 1] == p) && slot_of[p] < 0) {
        if (nslot >= 2) return fail("more than two saved FK transforms");
        slot_of[p] = nslot++;
      }
    }
    for (int k = 0; k < GMAX_FK; ++k) {
      pl.fk_j[g][k] = -1;
      pl.fk_par[g][k] = 0;
      pl.fk_save[g][k] = -1;
      pl.fk_store[g][k] = 0;
    }
    for (size_t k = 0; k < js.size(); ++k) {
      const int j = js[k], p = P::parent(j);
      pl.fk_j[g][k] = static_cast<int8_t>(j);
      pl.fk_par[g][k] = static_cast<int8_t>(p < 0 ? 3 : ((k > 0 && js[k - 1] == p) ? 0 : 1 + slot_of[p]));
      pl.fk_save[g][k] = static_cast<int8_t>(slot_of[j]);
      pl.fk_store[g][k] = static_cast<int8_t>(owner[j] == g || (owner[j] == -1 && g == 0));
    }
    n_fk = std::max(n_fk, static_cast<int>(js.size()));
  }
  pl.n_fk = n_fk;
  // prismatic root prefix: joints 0 .. n_pre-1, prismatic, each the child of
  // the one before, at the head of every lane's schedule, with no transform
  // saved and no task frame among them
  {
    int n = 0;
    while (n < GMAX_PRE && n < D && P::jtype(n) == PRIS && P::parent(n) == n - 1) ++n;
    for (int f = 0; f < P::NF; ++f) n = std::min(n, P::frame_link(f) < n ? P::frame_link(f) : n);
    for (int g = 0; g < GG; ++g)
      for (int k = 0; k < n; ++k)
        if (pl.fk_j[g][k] != k || pl.fk_save[g][k] >= 0) n = k;
    for (int g = 0; g < GG; ++g)
      if (n > 0 && pl.fk_j[g][n] >= 0 && pl.fk_par[g][n] != 0) n = 0;
    pl.n_pre = n;
  }
  // 2. subtree moments
  int n_cb = 0;
  for (int g = 0; g < GG; ++g) {
    int n = 0;
    for (int k = 0; k < GMAX_CB; ++k) pl.cb_j[g][k] = -1;
    for (int j = D - 1; j >= 0; --j)
      if (owner[j] == g) {
        if (n >= GMAX_CB) return fail("too many joints on one lane");
        pl.cb_j[g][n++] = static_cast<int8_t>(j);
      }
    n_cb = std::max(n_cb, n);
  }
  pl.n_cb = n_cb;
  int n_cr = 0, n_roots = 0;
  for (int k = 0; k < GMAX_CR; ++k) pl.cr_j[k] = -1;
  for (int j = D - 1; j >= 0; --j)
    if (owner[j] == -1) {
      if (n_cr >= GMAX_CR) return fail("trunk too long");
      pl.cr_j[n_cr++] = static_cast<int8_t>(j);
    }
  pl.n_cr = n_cr;
  for (int j = 0; j < D; ++j) {
    if (static_cast<int>(ch[j].size()) > GMAX_CH) return fail("too many children");
    for (int k = 0; k < GMAX_CH; ++k)
      pl.child[j][k] = static_cast<int8_t>(k < static_cast<int>(ch[j].size()) ? ch[j][k] : -1);
    if (P::parent(j) < 0) {
      if (n_roots >= 4) return fail("too many roots");
      pl.roots[n_roots++] = static_cast<int8_t>(j);
    }
  }
  pl.n_roots = n_roots;
  // segment offsets (every segment size is even: float2 loads): the 2-row
  // segments of the CoM-like constraints first, then the 6-row ones, so that
  // the subtree moments can live where the 6-row segments go until the 2-row
  // segments are built from them (grp_cbase)
  int off = 0;
  for (int pass = 0; pass < 2; ++pass)
    for (int j = 0; j < D; ++j)
      for (int c = 0; c < NC; ++c) {
        if (pass == 0) pl.joff[c][j] = -1;
        if (col_sign<P>(c, j) != 0 && grp_com_like<P>(c) == (pass == 0)) {
          pl.joff[c][j] = static_cast<int16_t>(off);
          off += cdim(P::ckind(c));
        }
      }
  for (int i = 0; i < GG * 5; ++i) {
    pl.lcol[i] = static_cast<int16_t>(i < kdim<P>() ? lcol_base<kdim<P>()>(i) : 0);
    pl.amask[i] = 0u;
    for (int b = 0; b < kdim<P>() && i < kdim<P>(); ++b)
      for (int j = 0; j < D; ++j)
        if (jnz<P>(i, j) && jnz<P>(b, j)) pl.amask[i] |= 1u << b;
  }
  for (int c = 0; c < NC; ++c) {
    pl.croff[c] = static_cast<int8_t>(roff<P>(c));
    pl.chull[c] = static_cast<int8_t>(P::ckind(c) == K_HULL);
    pl.pslot[c] = static_cast<int8_t>(grp_pose_like<P>(c) ? grp_pslot<P>(c) : -1);
    pl.hslot[c] = static_cast<int8_t>(P::ckind(c) == K_HULL ? grp_hslot<P>(c) : -1);
    pl.crel[c] = static_cast<int8_t>(P::ckind(c) == K_REL);
    pl.cfa[c] = static_cast<int8_t>(grp_pose_like<P>(c) ? P::cfa(c) : 0);
    pl.cfb[c] = static_cast<int8_t>(P::ckind(c) == K_REL ? P::cfb(c) : pl.cfa[c]);
  }
  // 4. segments: a limb's segments on its lane, the trunk's on the lane with
  // the fewest segments of that size
  {
    int n6[GG] = {0, 0, 0, 0}, n2[GG] = {0, 0, 0, 0};
    for (int g = 0; g < GG; ++g)
      for (int k = 0; k < GMAX_JI; ++k) pl.j6_j[g][k] = pl.j6_c[g][k] = pl.j2_j[g][k] = pl.j2_c[g][k] = -1;
    for (int pass = 0; pass < 2; ++pass)  // owned joints first, then the trunk
      for (int j = 0; j < D; ++j) {
        if ((owner[j] == -1) != (pass == 1)) continue;
        for (int c = 0; c < NC; ++c) {
          if (col_sign<P>(c, j) == 0) continue;
          const bool six = grp_pose_like<P>(c);
          int *cnt = six ? n6 : n2;
          int g = owner[j];
          if (g < 0) g = static_cast<int>(std::min_element(cnt, cnt + GG) - cnt);
          if (cnt[g] >= GMAX_JI) return fail("too many Jacobian segments on one lane");
          (six ? pl.j6_j : pl.j2_j)[g][cnt[g]] = static_cast<int8_t>(j);
          (six ? pl.j6_c : pl.j2_c)[g][cnt[g]] = static_cast<int8_t>(c);
          ++cnt[g];
        }
      }
    pl.n_j6 = *std::max_element(n6, n6 + GG);
    pl.n_j2 = *std::max_element(n2, n2 + GG);
  }
  // 7. dq joints
  {
    int nd[GG] = {0, 0, 0, 0};
    for (int g = 0; g < GG; ++g)
      for (int k = 0; k < GMAX_DQ; ++k) pl.dq_j[g][k] = -1;
    for (int pass = 0; pass < 2; ++pass)
      for (int j = 0; j < D; ++j) {
        if ((owner[j] == -1) != (pass == 1)) continue;
        int g = owner[j];
        if (g < 0) g = static_cast<int>(std::min_element(nd, nd + GG) - nd);
        if (nd[g] >= GMAX_DQ) return fail("too many dq joints on one lane");
        pl.dq_j[g][nd[g]++] = static_cast<int8_t>(j);
      }
    pl.n_dq = *std::max_element(nd, nd + GG);
  }
  // 5. Gram tasks: row-block pairs (a, b), rows of a at or below those of b,
  // sharing at least one joint; 7. refinement tasks: one per row block
  int pool_n = 0;
  auto add_list = [&](const std::vector<int> &js) -> int {
    if (pool_n + static_cast<int>(js.size()) > GMAX_POOL) return -1;
    const int o = pool_n;
    for (int j : js) pl.pool[pool_n++] = static_cast<int8_t>(j);
    return o;
  };
  auto schedule = [&](std::vector<std::pair<GrpTask, std::vector<int>>> &tasks, GrpTask (*dst)[GMAX_T],
                      int &nt, int *len) -> bool {
    std::stable_sort(tasks.begin(), tasks.end(),
                     [](const auto &x, const auto &y) { return x.second.size() > y.second.size(); });
    int cnt[GG] = {0, 0, 0, 0}, lo[GG] = {0, 0, 0, 0};
    for (int g = 0; g < GG; ++g)
      for (int t = 0; t < GMAX_T; ++t) dst[g][t] = GrpTask{-1, -1, 0, 0, 0, 0};
    for (auto &tk : tasks) {
      const int g = static_cast<int>(std::min_element(lo, lo + GG) - lo);
      if (cnt[g] >= GMAX_T || tk.second.size() > 127) return false;
      const int o = add_list(tk.second);
      if (o < 0) return false;
      GrpTask t = tk.first;
      t.n = static_cast<int8_t>(tk.second.size());
      t.off = static_cast<int16_t>(o);
      dst[g][cnt[g]++] = t;
      lo[g] += static_cast<int>(tk.second.size());
    }
    nt = *std::max_element(cnt, cnt + GG);
    for (int t = 0; t < GMAX_T; ++t) {
      len[t] = 0;
      for (int g = 0; g < GG; ++g) len[t] = std::max(len[t], static_cast<int>(dst[g][t].n));
    }
    return true;
  };
  for (int ph = 0; ph < 4; ++ph) {
    const bool a6 = ph < 2, b6 = (ph % 2) == 0;
    std::vector<std::pair<GrpTask, std::vector<int>>> tasks;
    for (int a = 0; a < NC; ++a)
      for (int b = 0; b < NC; ++b) {
        if (roff<P>(a) < roff<P>(b)) continue;
        if (grp_pose_like<P>(a) != a6 || grp_pose_like<P>(b) != b6) continue;
        if (a == b && grp_com_like<P>(a)) continue;  // summed over the dq partition instead
        std::vector<int> js;
        for (int j = 0; j < D; ++j)
          if (col_sign<P>(a, j) != 0 && col_sign<P>(b, j) != 0) js.push_back(j);
        if (!js.empty()) tasks.push_back({GrpTask{static_cast<int8_t>(a), static_cast<int8_t>(b), 0, 0, 0, 0}, js});
      }
    if (!schedule(tasks, pl.gt[ph], pl.g_nt[ph], pl.g_len[ph])) return fail("Gram tasks exceed the plan");
  }
  for (int ph = 0; ph < 2; ++ph) {
    std::vector<std::pair<GrpTask, std::vector<int>>> tasks;
    for (int a = 0; a < NC; ++a) {
      if (!grp_pose_like<P>(a) || ph == 1) continue;  // 2-row blocks: summed over the dq partition
      std::vector<int> js;
      for (int j = 0; j < D; ++j)
        if (col_sign<P>(a, j) != 0) js.push_back(j);
      tasks.push_back({GrpTask{static_cast<int8_t>(a), -1, 0, 0, 0, 0}, js});
    }
    if (!schedule(tasks, pl.rt[ph], pl.r_nt[ph], pl.r_len[ph])) return fail("refinement tasks exceed the plan");
  }
  return true;
}

// Per-configuration state in shared memory.
template <class P>
struct __align__(16) GrpState {
  static constexpr int D = P::D, K = kdim<P>(), KP = (K + 3) & ~3, NF = P::NF, NC = P::NC;
  static constexpr int DP = (D + 3) & ~3;
  static constexpr int NJ = (grp_nseg_floats<P>() + 3) & ~3;
  static constexpr int LC = lcol_base<K>(K);
  static constexpr int K2 = K * (K + 1) / 2;
  static constexpr int NPOSE = grp_npose<P>() > 0 ? grp_npose<P>() : 1;
  static constexpr int NHULL = grp_nhull<P>() > 0 ? grp_nhull<P>() : 1;
  struct Eval {           // FK and residual data, live until J is built
    float zo[D][6];       // joint axis z and origin o (world)
    float G[NPOSE][9];    // pose-like constraints: rotation into the error frame
    float x[NPOSE][4];    // reference point of the translational rows
    float phi[NPOSE][4];  // log-map vector and J_l^-1 coefficient (w)
    float hn[NHULL][2];   // support hull: normal of the nearest edge
    int hmode[NHULL];     // support hull: 0 inside, 1 edge, 2 vertex
  };
  struct Solve {         // after the Cholesky (the refinement's residual r overwrites F)
    float Lc[LC];        // L by columns (rows k..K-1 of column k at lcol_base(k))
    float y[KP];
    float dq[DP];
  };
  float q[DP];
  float F[KP];  // F, then the refinement's residual r = F - J dq - lambda y
  float J[NJ];  // Jacobian segments; before they are built, the task frames (NF x 12)
  union alignas(16) {
    Eval e;
    float A[K2];  // Gram (packed lower triangle, row-major), read into registers before
    Solve s;      // L's columns overwrite it (y and dq lie beyond A)
  } u;
  static_assert(NJ >= NF * 12, "task frames live in the Jacobian's space");
  static_assert(NF * 12 <= grp_cbase<P>() || !needs_com<P>(), "task frames must not overlap the subtree moments");
  static_assert(grp_cbase<P>() + 3 * D <= NJ || !needs_com<P>(), "subtree moments must fit the 6-row segments' space");
  // the subtree moments C_j (m_j c_j, then the sum over the subtree), in the
  // Jacobian's space until the 2-row segments are built
  __device__ __forceinline__ float *C(int j) { return J + grp_cbase<P>() + 3 * j; }
  static_assert(LC >= K2, "y and dq must not overlap the Gram matrix");
};

// Model data read with runtime joint indices (shared memory).
template <class P>
struct GrpTables {
  float X[P::D][12];
  float fX[P::NF][12];
  float com[P::D][3];
  float mass[P::D];
  float msub[P::D];
  int8_t rev[P::D];
  int8_t sgn[P::NC][P::D];  // column sign of joint j in constraint c
  // the prismatic root chain (PreChain)
  float pre_R[GMAX_PRE][9];
  float pre_a[GMAX_PRE][3];
  float pre_c[GMAX_PRE][3];
  float pre_mc[GMAX_PRE][3];
  int8_t pad[4 - (P::D * (P::NC + 1)) % 4];  // whole words
};
// Shared-memory stride between the states of consecutive configurations: an
// odd number of 16-byte units, so that the eight configurations of a warp
// start in eight different banks (with an even number the lanes of the eight
// groups reading the same field of their state collide in one bank, up to
// eight ways; measured: 43.7 ms instead of 32.3 ms on the full humanoid batch).
template <class P>
__host__ __device__ constexpr size_t grp_state_stride() {
  constexpr size_t u = (sizeof(GrpState<P>) + 15) / 16;
  return 16 * ((u % 2 == 0) ? u + 1 : u);
}

template <class P>
GrpTables<P> make_grp_tables(const ModelT<float> &m, const ModelT<double> &m64) {
  GrpTables<P> t{};
  const PreChain pc = make_pre_chain<P>(m64);
  for (int i = 0; i < GMAX_PRE; ++i) {
    for (int e = 0; e < 9; ++e) t.pre_R[i][e] = pc.R[i][e];
    for (int r = 0; r < 3; ++r) {
      t.pre_a[i][r] = pc.a[i][r];
      t.pre_c[i][r] = pc.c[i][r];
      t.pre_mc[i][r] = pc.mc[i][r];
    }
  }
  for (int j = 0; j < P::D; ++j) {
    for (int e = 0; e < 12; ++e) t.X[j][e] = m.X[j][e];
    for (int r = 0; r < 3; ++r) t.com[j][r] = m.com[j][r];
    t.mass[j] = m.mass[j];
    t.msub[j] = m.msub[j];
    t.rev[j] = P::jtype(j) == REV ? 1 : 0;
    for (int c = 0; c < P::NC; ++c) t.sgn[c][j] = static_cast<int8_t>(col_sign<P>(c, j));
  }
  for (int f = 0; f < P::NF; ++f)
    for (int e = 0; e < 12; ++e) t.fX[f][e] = m.fX[f][e];
  return t;
}

template <class P>
struct GroupArgs {
  ModelT<float> m;
  GrpTables<P> t;
  GroupPlan<P> pl;
  const ModelT<double> *__restrict__ m64;
  const double2 *__restrict__ tab;
  BatchSrc<float> src;
  float *q_out;
  long long ld_out;
  uint8_t *flags;
  uint8_t *iters;
  double *resid;
  unsigned long long *counter;
  long long total;
  int chunk;
  int cap;
  float tol2;
  float lambda;
  float max_step2;
  float pivot;
  double tol2_64;
  double lambda64;
  float alpha;
};

template <class P>
struct GrpShared {
  GrpTables<P> tb;
  GroupPlan<P> pl;
};

template <class P>
size_t group_smem_bytes(int W) {
  return ((sizeof(GrpShared<P>) + 15) & ~size_t(15)) + static_cast<size_t>(W) * GCPW * grp_state_stride<P>();
}

}  // namespace mcp
