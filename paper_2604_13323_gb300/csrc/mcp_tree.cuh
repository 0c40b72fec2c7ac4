// Thread-per-configuration projection of the 36-DoF humanoid classes.
//
// One lane holds one configuration; its Jacobian lives in shared memory and
// its 20 x 20 Gram matrix (138 structural nonzeros) and Cholesky factor in
// registers, so no stage of the Newton step has idle lanes, shuffles or
// shared-memory exchanges between lanes.
//
// What bounds it: instruction fetch and issue.  An iteration is about 12,800
// instructions for 32 configurations, most of them straight-line code of more
// than the instruction cache holds.  (Four lanes per configuration, with the
// Jacobian, Gram matrix and factor in shared memory, took 16,000
// warp-instructions per iteration for 8 configurations: 20.7 ms for 1,048,576
// configurations, 667 us for 4,099 and 410 us for 32, against 7.2 ms, 330 us
// and 150 us here.)  Layout:
//   * shared memory per configuration: 129 float2 (TREE_PAIRS), lane-major
//     (pair e of lane l at [e * 32 + l]: conflict-free 64-bit accesses at
//     immediate offsets); seven warps of 32 configurations fill an SM's 227 KB;
//   * the two legs, and the two arms, run the same code in a loop over the
//     side (half the instruction footprint);
//   * warps go through an iteration in step: a barrier between its phases
//     (TREE_SYNCS of them) keeps them within the same few KB of code, so that
//     one fetch serves several.  Without barriers the warps fetch seven places
//     at once: 13.0 ms instead of 8.5 ms for 1,048,576;
//   * in two teams, of the first TREE_TEAM warps and the rest (one warp of each
//     on a scheduler): a team takes its FP64 acceptances together, when one of
//     its warps has 32 configurations waiting (those with at least
//     TREE_ACCEPT_MIN take part), while the other team steps on in FP32.  Up to
//     96 configurations wait per warp, and a token lets one team at a time
//     accept: the teams settle in opposite phases instead of sharing the FP64
//     unit and then leaving it idle together (8.5 -> 7.2 ms for 1,048,576);
//   * the floating base's prismatic joints have constant Jacobian columns:
//     these, and their share of the Gram matrix, are kernel parameters.
//
// Every sum is taken in the order of the work plan (mcp_group.cuh; the CoM
// sums over the joints in four partial sums added pairwise), so that results
// do not depend on how lanes share the work.
#pragma once

#include "mcp_group.cuh"

namespace mcp {

// Structure of the humanoid tree (checked below): three prismatic and three
// revolute base joints, two legs of 6 from the pelvis, a waist of 2, a neck
// of 2 and two arms of 7 from the torso.
constexpr int TR_LEG = 6, TR_ARM = 7;
constexpr int TR_LEG0 = 6, TR_WAIST = 18, TR_TORSO = 19, TR_NECK = 20, TR_ARM0 = 22;

// float2 slots of one configuration's shared memory
constexpr int TP_LIMB = 0;                                  // per limb joint: 6-row segment (3), CoM (1)
constexpr int TP_ARM = TP_LIMB + 4 * 2 * TR_LEG;            // legs first, then arms
constexpr int TP_BASE = TP_ARM + 4 * 2 * TR_ARM;            // per revolute base joint: left foot (3), right foot (3), CoM (1)
constexpr int TP_UP = TP_BASE + 7 * 3;                      // waist, torso, neck joints: CoM
constexpr int TREE_PAIRS = TP_UP + 4;

template <class P>
__host__ __device__ constexpr bool tree_layout_matches() {
  if (P::D != 36 || P::NC != 4 || P::NF != 4) return false;
  for (int j = 0; j < 6; ++j)
    if (P::parent(j) != j - 1 || P::jtype(j) != (j < 3 ? PRIS : REV)) return false;
  for (int s = 0; s < 2; ++s) {
    for (int i = 0; i < TR_LEG; ++i) {
      const int j = TR_LEG0 + s * TR_LEG + i, r = TR_LEG0 + i;
      if (P::parent(j) != (i == 0 ? 5 : j - 1) || P::jtype(j) != REV) return false;
      if (P::xrot(j) != P::xrot(r) || P::xtmask(j) != P::xtmask(r) || P::xrot(j) == XR_GENERIC) return false;
    }
    for (int i = 0; i < TR_ARM; ++i) {
      const int j = TR_ARM0 + s * TR_ARM + i, r = TR_ARM0 + i;
      if (P::parent(j) != (i == 0 ? TR_TORSO : j - 1) || P::jtype(j) != REV) return false;
      if (P::xrot(j) != P::xrot(r) || P::xtmask(j) != P::xtmask(r) || P::xrot(j) == XR_GENERIC) return false;
    }
    if (P::frame_link(s) != TR_LEG0 + s * TR_LEG + TR_LEG - 1 || P::frot(s) != P::frot(0) || P::ftmask(s) != P::ftmask(0))
      return false;
    if (P::frame_link(2 + s) != TR_ARM0 + s * TR_ARM + TR_ARM - 1 || P::frot(2 + s) != P::frot(2) ||
        P::ftmask(2 + s) != P::ftmask(2))
      return false;
    if (P::ckind(s) != K_POSE || P::cfa(s) != s) return false;
  }
  for (int j = 3; j < TR_LEG0; ++j)
    if (P::xrot(j) == XR_GENERIC) return false;
  for (int j = TR_WAIST; j < TR_ARM0; ++j)
    if (P::jtype(j) != REV || P::xrot(j) == XR_GENERIC) return false;
  if (P::parent(TR_WAIST) != 5 || P::parent(TR_TORSO) != TR_WAIST || P::parent(TR_NECK) != TR_TORSO ||
      P::parent(TR_NECK + 1) != TR_NECK)
    return false;
  return P::ckind(2) == K_REL && P::cfa(2) == 2 && P::cfb(2) == 3 && (P::ckind(3) == K_COM || P::ckind(3) == K_HULL);
}

// Partial sum (0..3) that joint j's CoM terms belong to: the limbs one each
// (the left arm 0, the right arm 1, the left leg and the neck 2, the right leg
// 3), the trunk spread over them.  Within a partial the limb joints come
// first, in ascending order, then the trunk's.  This is the dq partition of
// the group kernel's work plan.
__host__ __device__ constexpr int tree_part(int j) {
  if (j >= TR_ARM0) return j < TR_ARM0 + TR_ARM ? 0 : 1;
  if (j >= TR_NECK) return 2;
  if (j >= TR_WAIST) return j == TR_WAIST ? 2 : 3;
  if (j >= TR_LEG0) return j < TR_LEG0 + TR_LEG ? 2 : 3;
  constexpr int base[6] = {3, 0, 1, 3, 0, 1};
  return base[j];
}

// Constants of the prismatic base chain (see GrpTables) and what follows from them.
template <class P>
struct TreeConst {
  float R[9];          // rotation after the chain
  float a[3][3];       // joint axes
  float c[3][3];       // origins at q = 0
  float mc[3][3];      // m_i R_i com_i
  float jt[2][3][3];   // translational rows of the feet's Jacobian columns
  float jc[3][2];      // CoM rows of their columns
  float LL[2][6];      // their share of J J^T: the feet's diagonal blocks (lower 3 x 3),
  float LR[9];         // right foot against left foot,
  float CL[2][6];      // CoM against each foot
};

template <class P>
struct TreeArgs {
  ModelT<float> m;
  TreeConst<P> t;
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

// Host: the constants, with the operations the kernel would use on them.
template <class P>
TreeConst<P> make_tree_const(const ModelT<float> &m, const ModelT<double> &m64) {
  const GrpTables<P> g = make_grp_tables<P>(m, m64);
  TreeConst<P> t{};
  for (int e = 0; e < 9; ++e) t.R[e] = g.pre_R[2][e];
  for (int i = 0; i < 3; ++i) {
    for (int r = 0; r < 3; ++r) {
      t.a[i][r] = g.pre_a[i][r];
      t.c[i][r] = g.pre_c[i][r];
      t.mc[i][r] = g.pre_mc[i][r];
    }
    const float f = m.msub[i] * m.inv_mass;
    t.jc[i][0] = f * t.a[i][0];
    t.jc[i][1] = f * t.a[i][1];
    for (int s = 0; s < 2; ++s)
      for (int r = 0; r < 3; ++r) {
        const float *Pi = m.cPinv[s] + 4 * r;
        const float p2 = Pi[2] * t.a[i][2];
        t.jt[s][i][r] = std::fmaf(Pi[0], t.a[i][0], std::fmaf(Pi[1], t.a[i][1], p2));
      }
  }
  for (int i = 0; i < 3; ++i) {
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c) t.LR[3 * r + c] = std::fmaf(t.jt[1][i][r], t.jt[0][i][c], t.LR[3 * r + c]);
    for (int s = 0; s < 2; ++s) {
      for (int r = 0; r < 3; ++r)
        for (int c = 0; c <= r; ++c) t.LL[s][tri(r, c)] = std::fmaf(t.jt[s][i][r], t.jt[s][i][c], t.LL[s][tri(r, c)]);
      for (int r = 0; r < 2; ++r)
        for (int c = 0; c < 3; ++c) t.CL[s][3 * r + c] = std::fmaf(t.jc[i][r], t.jt[s][i][c], t.CL[s][3 * r + c]);
    }
  }
  return t;
}

// T <- T X Rz(q) for a fixed offset X whose rotation is the signed permutation
// CODE and whose translation has the nonzero components TM.  The products of
// the dense composition with structural zeros are left out; those that remain
// are taken in its order (row index 2 first).
template <int CODE, int TM>
__device__ __forceinline__ void tree_joint(float (&T)[12], const float *X, float q) {
  constexpr int p0 = xr_perm(CODE, 0), p1 = xr_perm(CODE, 1), p2 = xr_perm(CODE, 2);
  float sn, cs;
  sincos_f32(q, sn, cs);
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    float p = T[4 * r + 3];
    if constexpr (TM & 4) p = fmaf(T[4 * r + 2], X[11], p);
    if constexpr (TM & 2) p = fmaf(T[4 * r + 1], X[7], p);
    if constexpr (TM & 1) p = fmaf(T[4 * r], X[3], p);
    const float a = xr_neg(CODE, 0) ? -T[4 * r + p0] : T[4 * r + p0];
    const float b = xr_neg(CODE, 1) ? -T[4 * r + p1] : T[4 * r + p1];
    const float c = xr_neg(CODE, 2) ? -T[4 * r + p2] : T[4 * r + p2];
    if constexpr (p0 < p1) {
      T[4 * r] = fmaf(cs, a, __fmul_rn(sn, b));
      T[4 * r + 1] = fmaf(-sn, a, __fmul_rn(cs, b));
    } else {
      T[4 * r] = fmaf(sn, b, __fmul_rn(cs, a));
      T[4 * r + 1] = fmaf(cs, b, -__fmul_rn(sn, a));
    }
    T[4 * r + 2] = c;
    T[4 * r + 3] = p;
  }
}

// Task frame on a link: rotation and origin of T Fx (signed permutation CODE, translation components TM).
template <int CODE, int TM>
__device__ __forceinline__ void tree_frame(const float (&T)[12], const float *Fx, float (&R)[9], V3<float> &p) {
  float o[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float v = T[4 * r + xr_perm(CODE, c)];
      R[3 * r + c] = xr_neg(CODE, c) ? -v : v;
    }
    float v = T[4 * r + 3];
    if constexpr (TM & 4) v = fmaf(T[4 * r + 2], Fx[11], v);
    if constexpr (TM & 2) v = fmaf(T[4 * r + 1], Fx[7], v);
    if constexpr (TM & 1) v = fmaf(T[4 * r], Fx[3], v);
    o[r] = v;
  }
  p = V3<float>{o[0], o[1], o[2]};
}

// m_j c_j of a placed link
__device__ __forceinline__ V3<float> tree_moment(const float (&T)[12], const float *com, float mass) {
  float v[3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
    v[r] = __fmul_rn(mass, fmaf(T[4 * r], com[0], fmaf(T[4 * r + 1], com[1], fmaf(T[4 * r + 2], com[2], T[4 * r + 3]))));
  return V3<float>{v[0], v[1], v[2]};
}
__device__ __forceinline__ V3<float> tree_add(V3<float> a, V3<float> b) {
  return V3<float>{__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z)};
}
// CoM rows of a revolute joint's Jacobian column: (1/M) z x (C - M_j o), x and y
__device__ __forceinline__ float2 tree_com_col(V3<float> z, V3<float> o, V3<float> C, float Mj, float inv_mass) {
  const V3<float> rr{fmaf(-Mj, o.x, C.x), fmaf(-Mj, o.y, C.y), fmaf(-Mj, o.z, C.z)};
  const V3<float> d = cross(z, rr);
  return make_float2(__fmul_rn(d.x, inv_mass), __fmul_rn(d.y, inv_mass));
}

// What the Jacobian of a pose-like constraint needs from its residual.
struct TreePose {
  V3<float> x, phi;
  float beta;
};
// Log map, stored residual rows and squared norm of a pose-like constraint.
__device__ __forceinline__ float tree_pose_tail(const float (&Rerr)[9], V3<float> t, TreePose &e, float (&F)[6]) {
  const auto lg = so3_log<OpsF32, float>(Rerr);
  e.phi = lg.phi;
  e.beta = jl_inv_beta<float>(lg.theta, lg.s, lg.c);
  F[0] = t.x;
  F[1] = t.y;
  F[2] = t.z;
  F[3] = lg.phi.x;
  F[4] = lg.phi.y;
  F[5] = lg.phi.z;
  return fmaf(t.x, t.x, fmaf(t.y, t.y, fmaf(t.z, t.z, fmaf(lg.phi.x, lg.phi.x, fmaf(lg.phi.y, lg.phi.y, lg.phi.z * lg.phi.z)))));
}
// 6-row segment of a revolute joint with axis z and origin o
__device__ __forceinline__ void tree_seg6(const float (&G)[9], const TreePose &e, V3<float> z, V3<float> o, float2 (&v)[3]) {
  const V3<float> vt = mulv(G, cross(z, sub(e.x, o)));
  const V3<float> w = jl_inv_apply(e.phi, e.beta, mulv(G, z));
  v[0] = make_float2(vt.x, vt.y);
  v[1] = make_float2(vt.z, w.x);
  v[2] = make_float2(w.y, w.z);
}
__device__ __forceinline__ void unpack6(const float2 (&v)[3], float (&f)[6]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    f[2 * i] = v[i].x;
    f[2 * i + 1] = v[i].y;
  }
}

// Warps of a block that go through the iterations in step with one another.
struct TreeTeam {
  int id, threads;  // named barrier and the number of threads that meet at it
  __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
  __device__ __forceinline__ bool any(bool v) const {
    int r;
    asm volatile(
        "{\n .reg .pred p, o;\n setp.ne.s32 p, %3, 0;\n bar.red.or.pred o, %1, %2, p;\n selp.s32 %0, 1, 0, o;\n}"
        : "=r"(r)
        : "r"(id), "r"(threads), "r"(static_cast<int>(v))
        : "memory");
    return r != 0;
  }
};

// Barriers of one iteration after its stopping test (before the hands' Gram
// block, the feet's, the Cholesky factorisation and each solve pass).
constexpr int TREE_SYNCS = 5;

// One FP32 iteration for the lane's configuration q.  Every lane of the warp
// runs it (idle lanes compute on whatever they hold and change nothing);
// returns true when the configuration leaves the FP32 loop (flags say why).
// Every warp of the block calls it (it holds block-wide barriers).
template <class P, class A>
__device__ __forceinline__ bool tree_iter(const A &a, const TreeTeam team, float2 *__restrict__ sm, float (&q)[P::D], bool act, int &it,
                                          uint32_t &fl) {
  static_assert(tree_layout_matches<P>(), "not the humanoid tree");
  constexpr int K = kdim<P>();
  constexpr bool HULL = P::ckind(3) == K_HULL;
  const ModelT<float> &m = a.m;
  const auto at = [&](int e) -> float2 & { return sm[e * 32]; };
  const float inv_mass = m.inv_mass;

  float F[K];
  float r2f[2] = {0.f, 0.f};           // squared residual norms of the feet
  V3<float> zb[3], ob[3], mb[3];       // revolute base joints: axis, origin, moment
  V3<float> zw[2], ow[2], mw[2];       // waist and torso
  V3<float> Cneck;                     // subtree moments of the torso's and pelvis's children
  V3<float> Cleg[2], Carm[2];
  float px[3][2];                      // prismatic joints: moments, x and y
  float T5[12], T19[12];
  // trunk and neck
  {
    float T[12];
    float o0 = 0.f, o1 = 0.f, o2 = 0.f, x0 = 0.f, x1 = 0.f, x2 = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      o0 = fmaf(q[i], a.t.a[i][0], o0);
      o1 = fmaf(q[i], a.t.a[i][1], o1);
      o2 = fmaf(q[i], a.t.a[i][2], o2);
      x0 = __fadd_rn(a.t.c[i][0], o0);
      x1 = __fadd_rn(a.t.c[i][1], o1);
      x2 = __fadd_rn(a.t.c[i][2], o2);
      px[i][0] = fmaf(m.mass[i], x0, a.t.mc[i][0]);
      px[i][1] = fmaf(m.mass[i], x1, a.t.mc[i][1]);
    }
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) T[4 * r + c] = a.t.R[3 * r + c];
    T[3] = x0;
    T[7] = x1;
    T[11] = x2;
    static_for<3>([&](auto II) {
      constexpr int i = decltype(II)::value, j = 3 + i;
      tree_joint<P::xrot(j), P::xtmask(j)>(T, m.X[j], q[j]);
      zb[i] = V3<float>{T[2], T[6], T[10]};
      ob[i] = V3<float>{T[3], T[7], T[11]};
      mb[i] = tree_moment(T, m.com[j], m.mass[j]);
    });
#pragma unroll
    for (int e = 0; e < 12; ++e) T5[e] = T[e];
    static_for<2>([&](auto II) {
      constexpr int i = decltype(II)::value, j = TR_WAIST + i;
      tree_joint<P::xrot(j), P::xtmask(j)>(T, m.X[j], q[j]);
      zw[i] = V3<float>{T[2], T[6], T[10]};
      ow[i] = V3<float>{T[3], T[7], T[11]};
      mw[i] = tree_moment(T, m.com[j], m.mass[j]);
    });
#pragma unroll
    for (int e = 0; e < 12; ++e) T19[e] = T[e];
    V3<float> zn[2], on[2], mn[2];
    static_for<2>([&](auto II) {
      constexpr int i = decltype(II)::value, j = TR_NECK + i;
      tree_joint<P::xrot(j), P::xtmask(j)>(T, m.X[j], q[j]);
      zn[i] = V3<float>{T[2], T[6], T[10]};
      on[i] = V3<float>{T[3], T[7], T[11]};
      mn[i] = tree_moment(T, m.com[j], m.mass[j]);
    });
    at(TP_UP + 3) = tree_com_col(zn[1], on[1], mn[1], m.msub[TR_NECK + 1], inv_mass);
    Cneck = tree_add(mn[0], mn[1]);
    at(TP_UP + 2) = tree_com_col(zn[0], on[0], Cneck, m.msub[TR_NECK], inv_mass);
  }
  // legs: FK, CoM columns, the foot's residual and its 6-row segments
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    float T[12];
#pragma unroll
    for (int e = 0; e < 12; ++e) T[e] = T5[e];
    V3<float> z[TR_LEG], o[TR_LEG], C[TR_LEG];
    const int j0 = TR_LEG0 + s * TR_LEG;
    static_for<TR_LEG>([&](auto II) {
      constexpr int i = decltype(II)::value, jr = TR_LEG0 + i;
      tree_joint<P::xrot(jr), P::xtmask(jr)>(T, m.X[j0 + i], q[j0 + i]);
      z[i] = V3<float>{T[2], T[6], T[10]};
      o[i] = V3<float>{T[3], T[7], T[11]};
      C[i] = tree_moment(T, m.com[j0 + i], m.mass[j0 + i]);
    });
    float2 *leg = sm + (TP_LIMB + 4 * TR_LEG * s) * 32;
    static_for<TR_LEG>([&](auto II) {
      constexpr int i = TR_LEG - 1 - decltype(II)::value;
      if constexpr (i + 1 < TR_LEG) C[i] = tree_add(C[i], C[i + 1]);
      leg[(4 * i + 3) * 32] = tree_com_col(z[i], o[i], C[i], m.msub[j0 + i], inv_mass);
    });
    float Ra[9], Pr[9], Qr[9], RaQ[9], Rerr[9], f6[6];
    V3<float> pa;
    tree_frame<P::frot(0), P::ftmask(0)>(T, m.fX[s], Ra, pa);
    load_R(m.cPinv[s], Pr);
    load_R(m.cQinv[s], Qr);
    const V3<float> Pp = load_p(m.cPinv[s]);
    TreePose e;
    mul33(Ra, Qr, RaQ);
    mul33(Pr, RaQ, Rerr);
    e.x = add_rot_t<7>(pa, Ra, load_p(m.cQinv[s]));
    const V3<float> tx = mulv(Pr, e.x);
    const float n2 =
        tree_pose_tail(Rerr, V3<float>{__fadd_rn(tx.x, Pp.x), __fadd_rn(tx.y, Pp.y), __fadd_rn(tx.z, Pp.z)}, e, f6);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      float2 v[3];
      tree_seg6(Pr, e, zb[i], ob[i], v);
      float2 *b = sm + (TP_BASE + 7 * i + 3 * s) * 32;
#pragma unroll
      for (int r = 0; r < 3; ++r) b[r * 32] = v[r];
    }
#pragma unroll
    for (int i = 0; i < TR_LEG; ++i) {
      float2 v[3];
      tree_seg6(Pr, e, z[i], o[i], v);
#pragma unroll
      for (int r = 0; r < 3; ++r) leg[(4 * i + r) * 32] = v[r];
    }
    if (s == 0) {
      r2f[0] = n2;
      Cleg[0] = C[0];
#pragma unroll
      for (int i = 0; i < 6; ++i) F[i] = f6[i];
    } else {
      r2f[1] = n2;
      Cleg[1] = C[0];
#pragma unroll
      for (int i = 0; i < 6; ++i) F[6 + i] = f6[i];
    }
  }
  team.sync();
  // arms: FK, CoM columns, axes and origins into the segments' slots
  float Ra[9], Rb[9];
  V3<float> pa, pb{0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 9; ++i) Rb[i] = 0.f;
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    float T[12];
#pragma unroll
    for (int e = 0; e < 12; ++e) T[e] = T19[e];
    V3<float> z[TR_ARM], o[TR_ARM], C[TR_ARM];
    const int j0 = TR_ARM0 + s * TR_ARM;
    float2 *arm = sm + (TP_ARM + 4 * TR_ARM * s) * 32;
    static_for<TR_ARM>([&](auto II) {
      constexpr int i = decltype(II)::value, jr = TR_ARM0 + i;
      tree_joint<P::xrot(jr), P::xtmask(jr)>(T, m.X[j0 + i], q[j0 + i]);
      z[i] = V3<float>{T[2], T[6], T[10]};
      o[i] = V3<float>{T[3], T[7], T[11]};
      C[i] = tree_moment(T, m.com[j0 + i], m.mass[j0 + i]);
      arm[(4 * i) * 32] = make_float2(z[i].x, z[i].y);
      arm[(4 * i + 1) * 32] = make_float2(z[i].z, o[i].x);
      arm[(4 * i + 2) * 32] = make_float2(o[i].y, o[i].z);
    });
    static_for<TR_ARM>([&](auto II) {
      constexpr int i = TR_ARM - 1 - decltype(II)::value;
      if constexpr (i + 1 < TR_ARM) C[i] = tree_add(C[i], C[i + 1]);
      arm[(4 * i + 3) * 32] = tree_com_col(z[i], o[i], C[i], m.msub[j0 + i], inv_mass);
    });
#pragma unroll
    for (int i = 0; i < 9; ++i) Ra[i] = Rb[i];
    pa = pb;
    tree_frame<P::frot(2), P::ftmask(2)>(T, m.fX[2 + s], Rb, pb);
    if (s == 0) Carm[0] = C[0];
    else Carm[1] = C[0];
  }
  team.sync();
  // the hands' relative pose: G = P^-1_R R_a^T, R_err = G R_b, t = G (p_b - p_a) + P^-1_p
  float G[9];
  TreePose eh;
  float r2h;
  {
    float Pr[9], RaT[9], Rerr[9], f6[6];
    load_R(m.cPinv[2], Pr);
    const V3<float> Pp = load_p(m.cPinv[2]);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) RaT[3 * r + c] = Ra[3 * c + r];
    mul33(Pr, RaT, G);
    mul33(G, Rb, Rerr);
    const V3<float> tx = mulv(G, sub(pb, pa));
    eh.x = pb;
    r2h = tree_pose_tail(Rerr, V3<float>{__fadd_rn(tx.x, Pp.x), __fadd_rn(tx.y, Pp.y), __fadd_rn(tx.z, Pp.z)}, eh, f6);
#pragma unroll
    for (int i = 0; i < 6; ++i) F[12 + i] = f6[i];
  }
  // trunk moments and CoM columns, the CoM residual
  float r2c;
  [[maybe_unused]] int hmode = 2;
  [[maybe_unused]] float hn0 = 0.f, hn1 = 0.f;
  {
    V3<float> C = tree_add(tree_add(tree_add(mw[1], Cneck), Carm[0]), Carm[1]);
    at(TP_UP + 1) = tree_com_col(zw[1], ow[1], C, m.msub[TR_TORSO], inv_mass);
    C = tree_add(mw[0], C);
    at(TP_UP) = tree_com_col(zw[0], ow[0], C, m.msub[TR_WAIST], inv_mass);
    C = tree_add(tree_add(tree_add(mb[2], Cleg[0]), Cleg[1]), C);
    at(TP_BASE + 7 * 2 + 6) = tree_com_col(zb[2], ob[2], C, m.msub[5], inv_mass);
    C = tree_add(mb[1], C);
    at(TP_BASE + 7 * 1 + 6) = tree_com_col(zb[1], ob[1], C, m.msub[4], inv_mass);
    C = tree_add(mb[0], C);
    at(TP_BASE + 6) = tree_com_col(zb[0], ob[0], C, m.msub[3], inv_mass);
    const float t0 = __fadd_rn(px[0][0], __fadd_rn(px[1][0], __fadd_rn(px[2][0], C.x)));
    const float t1 = __fadd_rn(px[0][1], __fadd_rn(px[1][1], __fadd_rn(px[2][1], C.y)));
    float f0, f1;
    if constexpr (HULL) {
      const float cx = __fmul_rn(t0, inv_mass), cy = __fmul_rn(t1, inv_mass);
      float qx, qy;
      hmode = polygon_nearest<float>(m.cB[3], static_cast<int>(m.ctgt[3][0]), cx, cy, qx, qy, hn0, hn1);
      f0 = __fadd_rn(cx, -qx);
      f1 = __fadd_rn(cy, -qy);
    } else {
      f0 = fmaf(t0, inv_mass, -m.ctgt[3][0]);
      f1 = fmaf(t1, inv_mass, -m.ctgt[3][1]);
    }
    F[18] = f0;
    F[19] = f1;
    r2c = fmaf(f0, f0, __fmul_rn(f1, f1));
  }
  const float r2 = __fadd_rn(__fadd_rn(r2f[0], r2f[1]), __fadd_rn(r2h, r2c));
  bool done = false;
  if (act) {
    if (!(r2 <= FLT_MAX)) {
      fl |= FL_NONFINITE;
      done = true;
    } else if (r2 < a.tol2 && !(fl & FL_INT_FORCE)) {
      fl |= FL_INT_FP32CONV;
      done = true;
    } else if (it >= a.cap) {
      fl |= FL_CAP;
      done = true;
    }
  }
  const bool go = act && !done;
  if (!__any_sync(FULL, go)) {  // nothing to solve in this warp: only the barriers that follow
    for (int i = 0; i < TREE_SYNCS; ++i) team.sync();
    return done;
  }
  team.sync();
  float2 jc[3];  // CoM columns of the prismatic joints
#pragma unroll
  for (int i = 0; i < 3; ++i) jc[i] = make_float2(a.t.jc[i][0], a.t.jc[i][1]);
  if constexpr (HULL) {  // inside the polygon: 0; on an edge: n n^T g; at a vertex: g
    const auto fold = [&](float2 v) -> float2 {
      const float sd = fmaf(hn0, v.x, __fmul_rn(hn1, v.y));
      const float2 ed = make_float2(__fmul_rn(hn0, sd), __fmul_rn(hn1, sd));
      return hmode == 0 ? make_float2(0.f, 0.f) : (hmode == 1 ? ed : v);
    };
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      jc[i] = fold(jc[i]);
      at(TP_BASE + 7 * i + 6) = fold(at(TP_BASE + 7 * i + 6));
    }
#pragma unroll 2
    for (int l = 0; l < 2 * (TR_LEG + TR_ARM); ++l) at(TP_LIMB + 4 * l + 3) = fold(at(TP_LIMB + 4 * l + 3));
#pragma unroll
    for (int i = 0; i < 4; ++i) at(TP_UP + i) = fold(at(TP_UP + i));
  }
  // Gram matrix (then its factor) in packed lower-triangular form; only the
  // structural nonzeros are touched
  float L[K * (K + 1) / 2];
  // hands' block and their CoM rows, with the arms' segments built in place
  {
    float H[21], CH[12];
#pragma unroll
    for (int i = 0; i < 21; ++i) H[i] = 0.f;
#pragma unroll
    for (int i = 0; i < 12; ++i) CH[i] = 0.f;
    float2 *arm = sm + TP_ARM * 32;
#pragma unroll 1
    for (int l = 0; l < 2 * TR_ARM; ++l, arm += 4 * 32) {
      float2 v[3] = {arm[0], arm[32], arm[64]};
      const float2 c = arm[96];
      const float sg = l < TR_ARM ? -1.f : 1.f;  // joints above frame a enter with -1, above b with +1
      tree_seg6(G, eh, V3<float>{v[0].x, v[0].y, v[1].x}, V3<float>{v[1].y, v[2].x, v[2].y}, v);
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        v[r] = make_float2(sg * v[r].x, sg * v[r].y);
        arm[r * 32] = v[r];
      }
      float f[6];
      unpack6(v, f);
#pragma unroll
      for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int k = 0; k <= i; ++k) H[tri(i, k)] = fmaf(f[i], f[k], H[tri(i, k)]);
        CH[i] = fmaf(c.x, f[i], CH[i]);
        CH[6 + i] = fmaf(c.y, f[i], CH[6 + i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
#pragma unroll
      for (int k = 0; k <= i; ++k) L[tri(12 + i, 12 + k)] = H[tri(i, k)];
      L[tri(18, 12 + i)] = CH[i];
      L[tri(19, 12 + i)] = CH[6 + i];
    }
  }
  team.sync();
  // feet: diagonal blocks, right against left, CoM rows
  {
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int k = 0; k <= i; ++k) L[tri(6 * s + i, 6 * s + k)] = i < 3 ? a.t.LL[s][tri(i < 3 ? i : 0, i < 3 ? k : 0)] : 0.f;
        if constexpr (!HULL) {
          L[tri(18, 6 * s + i)] = i < 3 ? a.t.CL[s][i < 3 ? i : 0] : 0.f;
          L[tri(19, 6 * s + i)] = i < 3 ? a.t.CL[s][3 + (i < 3 ? i : 0)] : 0.f;
        } else {
          float c0 = 0.f, c1 = 0.f;
          if (i < 3) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              c0 = fmaf(jc[k].x, a.t.jt[s][k][i < 3 ? i : 0], c0);
              c1 = fmaf(jc[k].y, a.t.jt[s][k][i < 3 ? i : 0], c1);
            }
          }
          L[tri(18, 6 * s + i)] = c0;
          L[tri(19, 6 * s + i)] = c1;
        }
      }
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int k = 0; k < 6; ++k) L[tri(6 + i, k)] = i < 3 && k < 3 ? a.t.LR[i < 3 && k < 3 ? 3 * i + k : 0] : 0.f;
    const auto own = [&](auto SS, const float (&f)[6], float2 c) {  // a foot's block and CoM rows
      constexpr int r0 = 6 * decltype(SS)::value;
#pragma unroll
      for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int k = 0; k <= i; ++k) L[tri(r0 + i, r0 + k)] = fmaf(f[i], f[k], L[tri(r0 + i, r0 + k)]);
        L[tri(18, r0 + i)] = fmaf(c.x, f[i], L[tri(18, r0 + i)]);
        L[tri(19, r0 + i)] = fmaf(c.y, f[i], L[tri(19, r0 + i)]);
      }
    };
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      float2 v[3];
      float fl6[6], fr6[6];
#pragma unroll
      for (int r = 0; r < 3; ++r) v[r] = at(TP_BASE + 7 * b + r);
      unpack6(v, fl6);
#pragma unroll
      for (int r = 0; r < 3; ++r) v[r] = at(TP_BASE + 7 * b + 3 + r);
      unpack6(v, fr6);
      const float2 c = at(TP_BASE + 7 * b + 6);
      own(std::integral_constant<int, 0>{}, fl6, c);
      own(std::integral_constant<int, 1>{}, fr6, c);
#pragma unroll
      for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int k = 0; k < 6; ++k) L[tri(6 + i, k)] = fmaf(fr6[i], fl6[k], L[tri(6 + i, k)]);
    }
    static_for<2>([&](auto SS) {
      constexpr int s = decltype(SS)::value;
#pragma unroll
      for (int i = 0; i < TR_LEG; ++i) {
        const int e = TP_LIMB + 4 * (TR_LEG * s + i);
        const float2 v[3] = {at(e), at(e + 1), at(e + 2)};
        float f[6];
        unpack6(v, f);
        own(SS, f, at(e + 3));
      }
    });
    // CoM block: four partial sums, limbs first
    float p[4][3];
#pragma unroll
    for (int g = 0; g < 4; ++g) p[g][0] = p[g][1] = p[g][2] = 0.f;
    const auto add = [&](int g, float2 c) {
      p[g][0] = fmaf(c.x, c.x, p[g][0]);
      p[g][1] = fmaf(c.y, c.x, p[g][1]);
      p[g][2] = fmaf(c.y, c.y, p[g][2]);
    };
#pragma unroll
    for (int i = 0; i < TR_ARM; ++i) {
      add(0, at(TP_ARM + 4 * i + 3));
      add(1, at(TP_ARM + 4 * (TR_ARM + i) + 3));
    }
#pragma unroll
    for (int i = 0; i < TR_LEG; ++i) {
      add(2, at(TP_LIMB + 4 * i + 3));
      add(3, at(TP_LIMB + 4 * (TR_LEG + i) + 3));
    }
    add(2, at(TP_UP + 2));
    add(2, at(TP_UP + 3));
    static_for<6>([&](auto JJ) {
      constexpr int j = decltype(JJ)::value;
      if constexpr (j < 3) add(tree_part(j), jc[j]);
      else add(tree_part(j), at(TP_BASE + 7 * (j - 3) + 6));
    });
    add(tree_part(TR_WAIST), at(TP_UP));
    add(tree_part(TR_TORSO), at(TP_UP + 1));
    L[tri(18, 18)] = __fadd_rn(__fadd_rn(p[0][0], p[1][0]), __fadd_rn(p[2][0], p[3][0]));
    L[tri(19, 18)] = __fadd_rn(__fadd_rn(p[0][1], p[1][1]), __fadd_rn(p[2][1], p[3][1]));
    L[tri(19, 19)] = __fadd_rn(__fadd_rn(p[0][2], p[1][2]), __fadd_rn(p[2][2], p[3][2]));
  }
  team.sync();
  // Cholesky, right-looking, on the structural nonzeros
  float invd[K];
  float minpiv = FLT_MAX;
#pragma unroll
  for (int i = 0; i < K; ++i) L[tri(i, i)] = __fadd_rn(L[tri(i, i)], a.lambda);
  static_for<K>([&](auto KK) {
    constexpr int k = decltype(KK)::value;
    const float piv = L[tri(k, k)];
    minpiv = fminf(minpiv, piv);
    const float ik = rsqrtf(piv);
    invd[k] = ik;
    static_for<K>([&](auto II) {
      constexpr int i = decltype(II)::value;
      if constexpr (i > k && ((LRow<P, i>::value >> k) & 1u)) L[tri(i, k)] = __fmul_rn(L[tri(i, k)], ik);
    });
    static_for<K>([&](auto II) {
      constexpr int i = decltype(II)::value;
      if constexpr (i > k && ((LRow<P, i>::value >> k) & 1u))
        static_for<i + 1>([&](auto BB) {
          constexpr int b = decltype(BB)::value;
          if constexpr (b > k && ((LRow<P, b>::value >> k) & 1u))
            L[tri(i, b)] = fmaf(-L[tri(i, k)], L[tri(b, k)], L[tri(i, b)]);
        });
    });
  });
  if (go && !(minpiv >= a.pivot)) {  // includes NaN: this configuration continues in FP64
    fl |= FL_INT_NEEDS_F64;
    done = true;
  }
  const bool go2 = act && !done;
  // y = A^{-1} F, then one refinement step with r = F - J (J^T y) - lambda y:
  // y += A^{-1} r; dq = J^T y in both passes (the second is the step)
  float t[K], y[K], sp[4], db[3];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    t[i] = F[i];
    y[i] = 0.f;
  }
#pragma unroll
  for (int g = 0; g < 4; ++g) sp[g] = 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i) db[i] = 0.f;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    team.sync();
    static_for<K>([&](auto KK) {  // forward: L y = b
      constexpr int k = decltype(KK)::value;
      t[k] = __fmul_rn(t[k], invd[k]);
      static_for<K>([&](auto II) {
        constexpr int i = decltype(II)::value;
        if constexpr (i > k && ((LRow<P, i>::value >> k) & 1u)) t[i] = fmaf(-L[tri(i, k)], t[k], t[i]);
      });
    });
    static_for<K>([&](auto KB) {  // back: L^T x = y
      constexpr int k = K - 1 - decltype(KB)::value;
      t[k] = __fmul_rn(t[k], invd[k]);
      static_for<K>([&](auto II) {
        constexpr int i = decltype(II)::value;
        if constexpr (i < k && ((LRow<P, k>::value >> i) & 1u)) t[i] = fmaf(-L[tri(k, i)], t[k], t[i]);
      });
    });
#pragma unroll
    for (int i = 0; i < K; ++i) y[i] = __fadd_rn(y[i], t[i]);
    // per joint: dq_j = J_j . y and, for the refinement, r += J_j dq_j
    float r[18], pc[4][2], dqb[6];
#pragma unroll
    for (int i = 0; i < 18; ++i) r[i] = 0.f;
#pragma unroll
    for (int g = 0; g < 4; ++g) pc[g][0] = pc[g][1] = sp[g] = 0.f;
    const bool last = pass == 1;
    const auto step = [&](int g, float d, float2 c) -> float {  // CoM partial sums, the scaled step
      pc[g][0] = fmaf(c.x, d, pc[g][0]);
      pc[g][1] = fmaf(c.y, d, pc[g][1]);
      const float e = __fmul_rn(d, a.alpha);
      sp[g] = fmaf(e, e, sp[g]);
      return e;
    };
    const auto com_dot = [&](float2 c, float acc) { return fmaf(c.x, y[18], fmaf(c.y, y[19], acc)); };
    const auto seg_dot = [&](const float2 (&v)[3], const float (&w)[6], float acc) {
#pragma unroll
      for (int i = 0; i < 3; ++i) acc = fmaf(v[i].x, w[2 * i], fmaf(v[i].y, w[2 * i + 1], acc));
      return acc;
    };
    const auto seg_add = [&](const float2 (&v)[3], float d, float (&w)[6]) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        w[2 * i] = fmaf(v[i].x, d, w[2 * i]);
        w[2 * i + 1] = fmaf(v[i].y, d, w[2 * i + 1]);
      }
    };
    float yf[2][6], rf[2][6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      yf[0][i] = y[i];
      yf[1][i] = y[6 + i];
      rf[0][i] = rf[1][i] = 0.f;
    }
    // base: prismatic columns are constants (their rotational rows zero)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      float acc = 0.f;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        acc = fmaf(a.t.jt[s][i][0], yf[s][0], fmaf(a.t.jt[s][i][1], yf[s][1], acc));
        acc = fmaf(a.t.jt[s][i][2], yf[s][2], acc);
      }
      acc = com_dot(jc[i], acc);
      dqb[i] = acc;
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int k = 0; k < 3; ++k) rf[s][k] = fmaf(a.t.jt[s][i][k], acc, rf[s][k]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int e = TP_BASE + 7 * b;
      const float2 vl[3] = {at(e), at(e + 1), at(e + 2)}, vr[3] = {at(e + 3), at(e + 4), at(e + 5)};
      const float d = com_dot(at(e + 6), seg_dot(vr, yf[1], seg_dot(vl, yf[0], 0.f)));
      dqb[3 + b] = d;
      seg_add(vl, d, rf[0]);
      seg_add(vr, d, rf[1]);
    }
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {  // legs
      float w[6], ra[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        w[i] = s == 0 ? yf[0][i] : yf[1][i];
        ra[i] = s == 0 ? rf[0][i] : rf[1][i];
      }
      pc[2][0] = pc[2][1] = sp[2] = 0.f;
      float2 *leg = sm + (TP_LIMB + 4 * TR_LEG * s) * 32;
#pragma unroll
      for (int i = 0; i < TR_LEG; ++i) {
        const float2 v[3] = {leg[4 * i * 32], leg[(4 * i + 1) * 32], leg[(4 * i + 2) * 32]};
        const float2 c = leg[(4 * i + 3) * 32];
        const float d = com_dot(c, seg_dot(v, w, 0.f));
        seg_add(v, d, ra);
        const float e = step(2, d, c);
        if (last) leg[4 * i * 32].x = e;
      }
      if (s == 0) {  // the left leg's sums move on; partial 2 starts over for the right leg
#pragma unroll
        for (int i = 0; i < 6; ++i) r[i] = ra[i];
        pc[3][0] = pc[2][0];
        pc[3][1] = pc[2][1];
        sp[3] = sp[2];
      } else {
#pragma unroll
        for (int i = 0; i < 6; ++i) r[6 + i] = ra[i];
      }
    }
    // partial 2 is the left leg's, 3 the right leg's
    {
      const float u0 = pc[2][0], u1 = pc[2][1], u2 = sp[2];
      pc[2][0] = pc[3][0];
      pc[2][1] = pc[3][1];
      sp[2] = sp[3];
      pc[3][0] = u0;
      pc[3][1] = u1;
      sp[3] = u2;
    }
    {
      float w[6], ra[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        w[i] = y[12 + i];
        ra[i] = 0.f;
      }
#pragma unroll 1
      for (int s = 0; s < 2; ++s) {  // arms
        pc[1][0] = pc[1][1] = sp[1] = 0.f;
        float2 *arm = sm + (TP_ARM + 4 * TR_ARM * s) * 32;
#pragma unroll
        for (int i = 0; i < TR_ARM; ++i) {
          const float2 v[3] = {arm[4 * i * 32], arm[(4 * i + 1) * 32], arm[(4 * i + 2) * 32]};
          const float2 c = arm[(4 * i + 3) * 32];
          const float d = com_dot(c, seg_dot(v, w, 0.f));
          seg_add(v, d, ra);
          const float e = step(1, d, c);
          if (last) arm[4 * i * 32].x = e;
        }
        if (s == 0) {
          pc[0][0] = pc[1][0];
          pc[0][1] = pc[1][1];
          sp[0] = sp[1];
        }
      }
#pragma unroll
      for (int i = 0; i < 6; ++i) r[12 + i] = ra[i];
    }
    // neck, then the trunk joints, each in its partial sum
    static_for<4>([&](auto II) {
      constexpr int i = (decltype(II)::value + 2) % 4;  // neck (2, 3), then waist (0) and torso (1)
      if constexpr (i == 0) {
        static_for<6>([&](auto JJ) {
          constexpr int j = decltype(JJ)::value;
          float2 c;
          if constexpr (j < 3) c = jc[j];
          else c = at(TP_BASE + 7 * (j - 3) + 6);
          const float e = step(tree_part(j), dqb[j], c);
          if constexpr (j < 3) db[j] = e;
          else if (last) at(TP_BASE + 7 * (j - 3)).x = e;
        });
      }
      const float2 c = at(TP_UP + i);
      const float e = step(tree_part(TR_WAIST + i), com_dot(c, 0.f), c);
      if (last) at(TP_UP + i).x = e;
    });
    if (last) break;
#pragma unroll
    for (int i = 0; i < 18; ++i) t[i] = fmaf(-a.lambda, y[i], __fadd_rn(F[i], -r[i]));
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float s = __fadd_rn(__fadd_rn(pc[0][i], pc[1][i]), __fadd_rn(pc[2][i], pc[3][i]));
      t[18 + i] = fmaf(-a.lambda, y[18 + i], __fadd_rn(F[18 + i], -s));
    }
  }
  // MaxDistance, update (the scaled steps lie in the first word of each joint's slot)
  const float s2 = __fadd_rn(__fadd_rn(sp[0], sp[1]), __fadd_rn(sp[2], sp[3]));
  if (go2 && a.max_step2 > 0.f && s2 > a.max_step2) {
    fl |= FL_DIV;
    done = true;
  }
  if (act && !done) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      q[i] = __fadd_rn(q[i], -db[i]);
      q[3 + i] = __fadd_rn(q[3 + i], -at(TP_BASE + 7 * i).x);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) q[TR_WAIST + i] = __fadd_rn(q[TR_WAIST + i], -at(TP_UP + i).x);
#pragma unroll
    for (int l = 0; l < 2 * TR_LEG; ++l) q[TR_LEG0 + l] = __fadd_rn(q[TR_LEG0 + l], -at(TP_LIMB + 4 * l).x);
#pragma unroll
    for (int l = 0; l < 2 * TR_ARM; ++l) q[TR_ARM0 + l] = __fadd_rn(q[TR_ARM0 + l], -at(TP_ARM + 4 * l).x);
    ++it;
    fl &= ~FL_INT_FORCE;
    if (!(s2 <= FLT_MAX)) {
      fl |= FL_NONFINITE;
      done = true;
    }
  }
  return done;
}

// Persistent projection, one configuration per lane.  Configurations that
// left the FP32 loop wait in registers (TREE_SLOTS per lane: the pending
// list's positions lane, lane + 32, ...) until 32 are there for a full warp of
// FP64 acceptances; those sent back for another FP32 step wait likewise (one
// per lane).  A 32-word scratch per warp routes them.  An acceptance always
// runs once a warp could not hold another iteration's 32 configurations, or
// has nothing else to do, with or without the token.
constexpr int TREE_WARPS = 7;
constexpr int TREE_TEAM = 4;
constexpr int TREE_ACCEPT_MIN = 20;
constexpr int TREE_SLOTS = 3;
template <class P>
__host__ __device__ constexpr size_t tree_smem_bytes(int warps) {
  return static_cast<size_t>(warps) * 32 * (TREE_PAIRS * sizeof(float2) + sizeof(int));
}
template <class P>
__global__ void __launch_bounds__(TREE_WARPS * 32, 1) k_project_tree(const __grid_constant__ TreeArgs<P> a) {
  constexpr int D = P::D;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  float2 *sm = reinterpret_cast<float2 *>(smem_raw) + wib * TREE_PAIRS * 32 + lane;
  int *route = reinterpret_cast<int *>(smem_raw + (blockDim.x >> 5) * TREE_PAIRS * 32 * sizeof(float2)) + wib * 32;
  __shared__ int fp64_taken;
  if (threadIdx.x == 0) fp64_taken = 0;
  __syncthreads();
  const int warps = blockDim.x >> 5, team0 = wib < TREE_TEAM ? 0 : TREE_TEAM;  // first warp of the team
  const TreeTeam team{1 + (team0 > 0), 32 * (team0 > 0 ? warps - TREE_TEAM : min(warps, TREE_TEAM))};
  long long qn = 0, qe = 0;  // warp-local queue [qn, qe)
  bool more = true;
  bool act = false;
  int item = 0;
  int it = 0;
  uint32_t fl = 0;
  int pend = 0, nret = 0;                                    // warp-uniform
  int p_item[TREE_SLOTS] = {}, p_meta[TREE_SLOTS] = {};  // pending positions lane, lane + 32, ...
  int r_item = 0, r_meta = 0;                              // retry position lane
  float q[D];
#pragma unroll 1
  for (int j = 0; j < D; ++j) q[j] = 0.f;
  while (true) {
    // refill idle lanes: retries first, then new work
    const unsigned idle = __ballot_sync(FULL, !act);
    if (idle != 0u && (nret > 0 || qn < qe || more)) {
      const int n_idle = __popc(idle);
      const int from_r = n_idle < nret ? n_idle : nret;
      const int need = n_idle - from_r;
      const long long avail = qe - qn;
      long long b0 = 0, b1 = 0;
      if (need > 0 && avail < need && more) {
        unsigned long long b = 0;
        if (lane == 0) b = atomicAdd(a.counter, static_cast<unsigned long long>(a.chunk));
        b = __shfl_sync(FULL, b, 0);
        if (static_cast<long long>(b) >= a.total) {
          more = false;
        } else {
          b0 = static_cast<long long>(b);
          b1 = b0 + a.chunk < a.total ? b0 + a.chunk : a.total;
        }
      }
      const int rank_all = __popc(idle & ((1u << lane) - 1u));
      const int pos = nret - 1 - rank_all;
      const int ri = __shfl_sync(FULL, r_item, pos & 31), rm = __shfl_sync(FULL, r_meta, pos & 31);
      if (!act) {
        const float *src = nullptr;
        long long ld = 0;
        if (rank_all < from_r) {  // one more FP32 step from the parked iterate
          item = ri;
          it = rm & 0xff;
          fl = ((static_cast<uint32_t>(rm) >> 8) & ~(FL_INT_FP32CONV | FL_INT_NEEDS_F64)) | FL_INT_FORCE;
          src = a.q_out;
          ld = a.ld_out;
        } else {
          const int rank = rank_all - from_r;
          long long cand = -1;
          if (rank < avail) cand = qn + rank;
          else if (rank - avail < b1 - b0) cand = b0 + (rank - avail);
          if (cand >= 0) {
            item = static_cast<int>(cand);
            it = 0;
            fl = 0;
            src = a.src.q;
            ld = a.src.ld;
          }
        }
        if (src) {
          act = true;
          const bool ok = MCP_CHK(item, ld);
#pragma unroll
          for (int j = 0; j < D; ++j) q[j] = ok ? src[j * ld + item] : 0.f;
        }
      }
      nret -= from_r;
      const long long used_old = need < avail ? need : avail;
      if (b1 > b0) {
        const long long rest = need - used_old;
        qn = b0 + (rest < b1 - b0 ? rest : b1 - b0);
        qe = b1;
      } else {
        qn += used_old;
      }
    }
    bool done = false;
    if (team.any(act)) done = tree_iter<P>(a, team, sm, q, act, it, fl);
    // park finished configurations
    const unsigned fin = __ballot_sync(FULL, done);
    if (fin != 0u) {
      const int nf = __popc(fin), rank = __popc(fin & ((1u << lane) - 1u));
      if (done) {
        if (MCP_CHK(item, a.ld_out)) {
#pragma unroll
          for (int j = 0; j < D; ++j) a.q_out[j * a.ld_out + item] = q[j];
        }
        route[rank] = item;
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < TREE_SLOTS; ++k) {  // the rank that lands on this lane's position k
        const int r = lane + 32 * k - pend;
        if (r >= 0 && r < nf) p_item[k] = route[r];
      }
      __syncwarp();
      if (done) route[rank] = static_cast<int>(static_cast<uint32_t>(it) | (fl << 8));
      __syncwarp();
#pragma unroll
      for (int k = 0; k < TREE_SLOTS; ++k) {
        const int r = lane + 32 * k - pend;
        if (r >= 0 && r < nf) p_meta[k] = route[r];
      }
      __syncwarp();
      if (done) act = false;
      pend += nf;
    }
    const bool drained = !__any_sync(FULL, act) && qn >= qe && !more && nret == 0;
    // FP64 acceptance, one configuration per lane, 32 at a time; a failed
    // acceptance with steps left goes back to the FP32 loop
    bool accept = false, token = false;
    if (team.any(pend >= 32 || (drained && pend > 0))) {
      if (wib == team0 && lane == 0) token = atomicCAS(&fp64_taken, 0, 1) == 0;
      accept = team.any(token || pend > 32 * (TREE_SLOTS - 1) || drained);
    }
    if (accept && pend > 0 && (pend >= TREE_ACCEPT_MIN || drained)) {
      const int take = pend < 32 ? pend : 32;
      const bool room = nret + take <= 32;
      const int pos = pend - take + lane;
      int it_item = 0, im = 0;
#pragma unroll
      for (int k = 0; k < TREE_SLOTS; ++k) {
        const int vi = __shfl_sync(FULL, p_item[k], pos & 31), vm = __shfl_sync(FULL, p_meta[k], pos & 31);
        if ((pos >> 5) == k) {
          it_item = vi;
          im = vm;
        }
      }
      const uint32_t meta = static_cast<uint32_t>(im);
      bool retry = false;
      if (lane < take) retry = accept_one<P, FORM_STACKED>(a, it_item, static_cast<int>(meta & 0xffu), meta >> 8, room);
      const unsigned rmask = __ballot_sync(FULL, retry);
      if (rmask != 0u) {
        const int nr = __popc(rmask), rank = __popc(rmask & ((1u << lane) - 1u)), s0 = lane - nret;
        if (retry) route[rank] = it_item;
        __syncwarp();
        if (s0 >= 0 && s0 < nr) r_item = route[s0];
        __syncwarp();
        if (retry) route[rank] = static_cast<int>(meta);
        __syncwarp();
        if (s0 >= 0 && s0 < nr) r_meta = route[s0];
        __syncwarp();
        nret += nr;
      }
      pend -= take;
    }
    const bool left = team.any(!(drained && pend == 0 && nret == 0));
    if (token) atomicExch(&fp64_taken, 0);
    if (!left) break;
  }
}

template <class P>
cudaError_t launch_project_tree(const HostModel &hm, const ProjCall &c, int *launches) {
  if (c.total <= 0) return cudaSuccess;
  if (c.precision == 1 || c.segments || c.outer || c.cyclic) return cudaErrorNotSupported;
  if (c.total > 0x7fffffffLL) return cudaErrorInvalidValue;  // parked indices are 32-bit
  TreeArgs<P> a;
  cudaError_t err = cudaMemsetAsync(c.counter, 0, sizeof(unsigned long long), c.stream);
  if (err != cudaSuccess) return err;
  a.m = hm.m32;
  a.t = make_tree_const<P>(hm.m32, hm.m64);
  a.m64 = hm.d_m64;
  a.tab = hm.d_tab;
  a.src = BatchSrc<float>{static_cast<const float *>(c.q_in), c.ld_in};
  a.q_out = static_cast<float *>(c.q_out);
  a.ld_out = c.ld_out;
  a.flags = c.flags;
  a.iters = c.iters;
  a.resid = c.resid;
  a.counter = c.counter;
  a.total = c.total;
  a.chunk = 32;
  a.cap = c.cap;
  a.tol2 = static_cast<float>(c.tol * c.tol);
  a.lambda = static_cast<float>(c.lambda);
  a.max_step2 = c.max_step > 0 ? static_cast<float>(c.max_step * c.max_step) : 0.f;
  a.pivot = static_cast<float>(c.pivot);
  a.tol2_64 = c.tol * c.tol;
  a.lambda64 = c.lambda;
  a.alpha = static_cast<float>(c.alpha);
  // warps per block: one until every SM has one, then up to what shared memory holds
  const long long warps = (c.total + 31) / 32;
  long long w = (warps + hm.sm_count - 1) / hm.sm_count;
  if (w > TREE_WARPS) w = TREE_WARPS;
  const size_t smem = tree_smem_bytes<P>(static_cast<int>(w));
  auto kern = k_project_tree<P>;
  err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (err != cudaSuccess) return err;
  long long blocks = (warps + w - 1) / w;
  if (blocks > hm.sm_count) blocks = hm.sm_count;
  kern<<<static_cast<unsigned>(blocks), static_cast<unsigned>(w) * 32, smem, c.stream>>>(a);
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace mcp
