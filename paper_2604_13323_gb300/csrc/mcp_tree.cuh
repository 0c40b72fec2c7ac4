// Thread-per-configuration projection of the 36-DoF humanoid classes.
//
// One lane holds one configuration; its Jacobian lives in shared memory and
// its 20 x 20 Gram matrix (138 structural nonzeros) and Cholesky factor in
// registers, so no stage of the Newton step has idle lanes, shuffles or
// shared-memory exchanges between lanes.
//
// What bounds it: instruction fetch and dependent latency.  An iteration is
// about 11,000 instructions for 32 configurations, most of them straight-line
// code of more than the instruction cache holds; a scheduler has two warps.
// (Four lanes per configuration, with the Jacobian, Gram matrix and factor in
// shared memory, took 16,000 warp-instructions per iteration for 8
// configurations.  Projection and check of 1,048,576 configurations 21.9 ms,
// of 4,099 742 us, projection of 32 459 us; here, in turn with it on the same
// device, 7.3 ms, 281 us and 153 us.)  Layout:
//   * shared memory per configuration: 129 float2 (TREE_PAIRS), lane-major
//     (pair e of lane l at [e * 32 + l]: conflict-free 64-bit accesses at
//     immediate offsets); seven warps of 32 configurations fill an SM's 227 KB;
//   * the left and the right leg, and the two arms, go through FK, Jacobian,
//     Gram and solve together, two values per instruction (mcp_pack.cuh; with
//     the limbs one after the other the projection took 6.9 ms instead of 6.2 ms);
//   * Jacobian segments are built in loops over a limb's joints that fit the
//     scheduler's own instruction buffer;
//   * warps go through an iteration in step: a barrier between its phases
//     (TREE_SYNCS of them after the stopping test) keeps them within the same
//     few KB of code, so that one fetch serves several.  Without barriers the
//     warps fetched seven places at once: 13.0 ms instead of 8.5 ms;
//   * in two teams, of the first TREE_TEAM warps and the rest (one warp of each
//     on a scheduler): a team takes its FP64 acceptances together, when each of
//     its warps has 32 configurations waiting, while the other team steps on in
//     FP32.  Up to 96 configurations wait per warp, and a token lets one team
//     at a time accept: the teams settle in opposite phases instead of sharing
//     the FP64 unit and then leaving it idle together (8.5 -> 7.2 ms);
//   * the next chunk of starts is claimed while the last is used up, and
//     prefetched (the refill 6,000 -> 3,000 cycles of an iteration of 65,000);
//   * the floating base's prismatic joints have constant Jacobian columns:
//     these, and their share of the Gram matrix, are kernel parameters.
//
// Every sum is taken in the order of the work plan (mcp_group.cuh; the CoM
// sums over the joints in four partial sums added pairwise), so that results
// do not depend on how lanes share the work.
#pragma once

#include "mcp_factor.cuh"
#include "mcp_group.cuh"  // only the order its host check compares with
#include "mcp_pack.cuh"

namespace mcp {

// Structure of the humanoid tree (checked below): three prismatic and three
// revolute base joints, two legs of 6 from the pelvis, a waist of 2, a neck
// of 2 and two arms of 7 from the torso.
constexpr int TR_LEG = 6, TR_ARM = 7;
constexpr int TR_LEG0 = 6, TR_WAIST = 18, TR_TORSO = 19, TR_NECK = 20, TR_ARM0 = 22;

// float2 slots of one configuration's shared memory; in a limb's slots x is
// the left limb's value, y the right limb's
constexpr int TP_LEG = 0;                        // per leg joint: axis and origin, then the 6-row segment (6), CoM (2)
constexpr int TP_ARM = TP_LEG + 8 * TR_LEG;      // per arm joint: the same
constexpr int TP_BASE = TP_ARM + 8 * TR_ARM;     // per revolute base joint: the feet's segments (6), CoM (1: x, y rows)
constexpr int TP_UP = TP_BASE + 7 * 3;           // waist, torso, neck joints: CoM (x, y rows)
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
// the work plan.
__host__ __device__ constexpr int tree_part(int j) {
  if (j >= TR_ARM0) return j < TR_ARM0 + TR_ARM ? 0 : 1;
  if (j >= TR_NECK) return 2;
  if (j >= TR_WAIST) return j == TR_WAIST ? 2 : 3;
  if (j >= TR_LEG0) return j < TR_LEG0 + TR_LEG ? 2 : 3;
  constexpr int base[6] = {3, 0, 1, 3, 0, 1};
  return base[j];
}

// Constants of the prismatic base chain (see PreChain) and what follows from
// them, and the limbs' model data in left / right pairs.
template <int N>
struct TreeLimb {
  float2 t[N][3];    // offset's translation
  float2 com[N][3];
  float2 mass[N];
  float2 nmsub[N];   // minus the subtree mass
  float2 ft[3];      // task frame's translation
};
template <class P>
struct TreeConst {
  TreeLimb<TR_LEG> leg;
  TreeLimb<TR_ARM> arm;
  float2 Pr[9], Pp[3], Qr[9], Qp[3];  // the feet's error frames: P^-1, Q^-1
  float2 jt[3][3];     // translational rows of the feet's Jacobian columns of the prismatic joints,
  float2 LL[6];        // their share of J J^T: the feet's diagonal blocks (lower 3 x 3),
  float2 CL[6];        // CoM against each foot,
  float LR[9];         // right foot against left foot
  float jc[3][2];      // CoM rows of their columns
  float R[9];          // rotation after the chain
  float a[3][3];       // joint axes
  float c[3][3];       // origins at q = 0
  float mc[3][3];      // m_i R_i com_i
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
template <int N>
void fill_limb(const ModelT<float> &m, int jl, int jr, int fl, int fr, TreeLimb<N> &t) {
  for (int i = 0; i < N; ++i) {
    for (int k = 0; k < 3; ++k) {
      t.t[i][k] = make_float2(m.X[jl + i][4 * k + 3], m.X[jr + i][4 * k + 3]);
      t.com[i][k] = make_float2(m.com[jl + i][k], m.com[jr + i][k]);
    }
    t.mass[i] = make_float2(m.mass[jl + i], m.mass[jr + i]);
    t.nmsub[i] = make_float2(-m.msub[jl + i], -m.msub[jr + i]);
  }
  for (int k = 0; k < 3; ++k) t.ft[k] = make_float2(m.fX[fl][4 * k + 3], m.fX[fr][4 * k + 3]);
}
template <class P>
TreeConst<P> make_tree_const(const ModelT<float> &m, const ModelT<double> &m64) {
  const PreChain g = make_pre_chain<P>(m64);
  TreeConst<P> t{};
  fill_limb(m, TR_LEG0, TR_LEG0 + TR_LEG, 0, 1, t.leg);
  fill_limb(m, TR_ARM0, TR_ARM0 + TR_ARM, 2, 3, t.arm);
  for (int r = 0; r < 3; ++r) {
    for (int c = 0; c < 3; ++c) {
      t.Pr[3 * r + c] = make_float2(m.cPinv[0][4 * r + c], m.cPinv[1][4 * r + c]);
      t.Qr[3 * r + c] = make_float2(m.cQinv[0][4 * r + c], m.cQinv[1][4 * r + c]);
    }
    t.Pp[r] = make_float2(m.cPinv[0][4 * r + 3], m.cPinv[1][4 * r + 3]);
    t.Qp[r] = make_float2(m.cQinv[0][4 * r + 3], m.cQinv[1][4 * r + 3]);
  }
  float jt[2][3][3], LL[2][6] = {}, CL[2][6] = {};
  for (int e = 0; e < 9; ++e) t.R[e] = g.R[2][e];
  for (int i = 0; i < 3; ++i) {
    for (int r = 0; r < 3; ++r) {
      t.a[i][r] = g.a[i][r];
      t.c[i][r] = g.c[i][r];
      t.mc[i][r] = g.mc[i][r];
    }
    const float f = m.msub[i] * m.inv_mass;
    t.jc[i][0] = f * t.a[i][0];
    t.jc[i][1] = f * t.a[i][1];
    for (int s = 0; s < 2; ++s)
      for (int r = 0; r < 3; ++r) {
        const float *Pi = m.cPinv[s] + 4 * r;
        const float p2 = Pi[2] * t.a[i][2];
        jt[s][i][r] = std::fmaf(Pi[0], t.a[i][0], std::fmaf(Pi[1], t.a[i][1], p2));
      }
    for (int r = 0; r < 3; ++r) {
      t.jt[i][r] = make_float2(jt[0][i][r], jt[1][i][r]);
      for (int c = 0; c < 3; ++c) t.LR[3 * r + c] = std::fmaf(jt[1][i][r], jt[0][i][c], t.LR[3 * r + c]);
    }
    for (int s = 0; s < 2; ++s) {
      for (int r = 0; r < 3; ++r)
        for (int c = 0; c <= r; ++c) LL[s][tri(r, c)] = std::fmaf(jt[s][i][r], jt[s][i][c], LL[s][tri(r, c)]);
      for (int r = 0; r < 2; ++r)
        for (int c = 0; c < 3; ++c) CL[s][3 * r + c] = std::fmaf(t.jc[i][r], jt[s][i][c], CL[s][3 * r + c]);
    }
  }
  for (int e = 0; e < 6; ++e) {
    t.LL[e] = make_float2(LL[0][e], LL[1][e]);
    t.CL[e] = make_float2(CL[0][e], CL[1][e]);
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

// The same for a left and a right joint of one structure: offset translation
// t, task-frame translation ft, masses and CoM offsets in pairs.
template <int CODE, int TM>
__device__ __forceinline__ void tree_joint2(float2 (&T)[12], const float2 *t, float2 q) {
  constexpr int p0 = xr_perm(CODE, 0), p1 = xr_perm(CODE, 1), p2 = xr_perm(CODE, 2);
  float2 sn, cs;
  sincos2_f32(q, sn, cs);
  const float2 nsn = neg2(sn);
  const float2 csa = xr_neg(CODE, 0) ? neg2(cs) : cs, sna = xr_neg(CODE, 0) ? sn : nsn;  // sna = -(sign sn)
  const float2 csb = xr_neg(CODE, 1) ? neg2(cs) : cs, snb = xr_neg(CODE, 1) ? nsn : sn;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    float2 p = T[4 * r + 3];
    if constexpr (TM & 4) p = fma2(T[4 * r + 2], t[2], p);
    if constexpr (TM & 2) p = fma2(T[4 * r + 1], t[1], p);
    if constexpr (TM & 1) p = fma2(T[4 * r], t[0], p);
    const float2 a = T[4 * r + p0], b = T[4 * r + p1], c = T[4 * r + p2];
    if constexpr (p0 < p1) {
      T[4 * r] = fma2(csa, a, mul2(snb, b));
      T[4 * r + 1] = fma2(sna, a, mul2(csb, b));
    } else {
      T[4 * r] = fma2(snb, b, mul2(csa, a));
      T[4 * r + 1] = fma2(csb, b, mul2(sna, a));
    }
    T[4 * r + 2] = xr_neg(CODE, 2) ? neg2(c) : c;
    T[4 * r + 3] = p;
  }
}
template <int CODE, int TM>
__device__ __forceinline__ void tree_frame2(const float2 (&T)[12], const float2 *ft, float2 (&R)[9], V3p &p) {
  float2 o[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float2 v = T[4 * r + xr_perm(CODE, c)];
      R[3 * r + c] = xr_neg(CODE, c) ? neg2(v) : v;
    }
    float2 v = T[4 * r + 3];
    if constexpr (TM & 4) v = fma2(T[4 * r + 2], ft[2], v);
    if constexpr (TM & 2) v = fma2(T[4 * r + 1], ft[1], v);
    if constexpr (TM & 1) v = fma2(T[4 * r], ft[0], v);
    o[r] = v;
  }
  p = V3p{o[0], o[1], o[2]};
}
__device__ __forceinline__ V3p load_axis(const float2 *s) { return V3p{s[0], s[32], s[64]}; }
__device__ __forceinline__ V3p load_origin(const float2 *s) { return V3p{s[96], s[128], s[160]}; }
// FK of a pair of limbs of N joints (the first joint's class index J0), from
// the frame T of their parent: axes and origins into the joints' slots (read
// back for the CoM columns: kept in registers they would spill), the CoM
// columns after them; returns the limbs' subtree moments, T the tip's frame.
template <class P, int J0, int N>
__device__ __forceinline__ V3p tree_limbs(const TreeLimb<N> &m, float2 (&T)[12], const float (&q)[P::D], float inv_mass,
                                          float2 *__restrict__ slot) {
  V3p C[N];
  static_for<N>([&](auto II) {
    constexpr int i = decltype(II)::value, j = J0 + i;
    tree_joint2<P::xrot(j), P::xtmask(j)>(T, m.t[i], make_float2(q[j], q[j + N]));
    float2 v[3];
#pragma unroll
    for (int r = 0; r < 3; ++r)
      v[r] = mul2(m.mass[i], fma2(T[4 * r], m.com[i][0],
                                              fma2(T[4 * r + 1], m.com[i][1],
                                                         fma2(T[4 * r + 2], m.com[i][2], T[4 * r + 3]))));
    C[i] = V3p{v[0], v[1], v[2]};
    float2 *s = slot + 8 * 32 * i;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      s[r * 32] = T[4 * r + 2];
      s[(3 + r) * 32] = T[4 * r + 3];
    }
  });
  static_for<N>([&](auto II) {
    constexpr int i = N - 1 - decltype(II)::value;
    if constexpr (i + 1 < N)
      C[i] = V3p{add2_apart(C[i].x, C[i + 1].x), add2_apart(C[i].y, C[i + 1].y), add2_apart(C[i].z, C[i + 1].z)};
    // (1/M) z x (C - M_j o), x and y
    const float2 nM = m.nmsub[i];
    const V3p z = load_axis(slot + 8 * 32 * i), o = load_origin(slot + 8 * 32 * i);
    const V3p rr{fma2(nM, o.x, C[i].x), fma2(nM, o.y, C[i].y), fma2(nM, o.z, C[i].z)};
    const float2 dx = fma2(z.y, rr.z, mul2(neg2(z.z), rr.y));
    const float2 dy = fma2(z.z, rr.x, mul2(neg2(z.x), rr.z));
    slot[(8 * i + 6) * 32] = mul2(dx, both(inv_mass));
    slot[(8 * i + 7) * 32] = mul2(dy, both(inv_mass));
  });
  return C[0];
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

  float qv[P::D];  // loaded together: one latency, not one per chain
#pragma unroll
  for (int j = 0; j < P::D; ++j) qv[j] = q[j];
  float F[K];
  V3<float> mb[3];                     // revolute base joints: moments
  V3<float> zw[2], ow[2], mw[2];       // waist and torso
  V3<float> Cneck;                     // subtree moments of the torso's and pelvis's children
  V3p Cleg, Carm;
  float px[3][2];                      // prismatic joints: moments, x and y
  float T5[12], T19[12];               // pelvis and torso frames
  // trunk and neck
  {
    float T[12];
    float o0 = 0.f, o1 = 0.f, o2 = 0.f, x0 = 0.f, x1 = 0.f, x2 = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      o0 = fmaf(qv[i], a.t.a[i][0], o0);
      o1 = fmaf(qv[i], a.t.a[i][1], o1);
      o2 = fmaf(qv[i], a.t.a[i][2], o2);
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
      tree_joint<P::xrot(j), P::xtmask(j)>(T, m.X[j], qv[j]);
#pragma unroll
      for (int r = 0; r < 3; ++r) {  // the same for both feet
        at(TP_BASE + 7 * i + r) = both(T[4 * r + 2]);
        at(TP_BASE + 7 * i + 3 + r) = both(T[4 * r + 3]);
      }
      mb[i] = tree_moment(T, m.com[j], m.mass[j]);
    });
#pragma unroll
    for (int e = 0; e < 12; ++e) T5[e] = T[e];
    static_for<2>([&](auto II) {
      constexpr int i = decltype(II)::value, j = TR_WAIST + i;
      tree_joint<P::xrot(j), P::xtmask(j)>(T, m.X[j], qv[j]);
      zw[i] = V3<float>{T[2], T[6], T[10]};
      ow[i] = V3<float>{T[3], T[7], T[11]};
      mw[i] = tree_moment(T, m.com[j], m.mass[j]);
    });
#pragma unroll
    for (int e = 0; e < 12; ++e) T19[e] = T[e];
    V3<float> zn[2], on[2], mn[2];
    static_for<2>([&](auto II) {
      constexpr int i = decltype(II)::value, j = TR_NECK + i;
      tree_joint<P::xrot(j), P::xtmask(j)>(T, m.X[j], qv[j]);
      zn[i] = V3<float>{T[2], T[6], T[10]};
      on[i] = V3<float>{T[3], T[7], T[11]};
      mn[i] = tree_moment(T, m.com[j], m.mass[j]);
    });
    at(TP_UP + 3) = tree_com_col(zn[1], on[1], mn[1], m.msub[TR_NECK + 1], inv_mass);
    Cneck = tree_add(mn[0], mn[1]);
    at(TP_UP + 2) = tree_com_col(zn[0], on[0], Cneck, m.msub[TR_NECK], inv_mass);
  }
  // legs and arms, left and right together
  float2 Rf[9], Rh[9];
  V3p pf, ph;
  {
    float2 T[12];
#pragma unroll
    for (int e = 0; e < 12; ++e) T[e] = both(T5[e]);
    Cleg = tree_limbs<P, TR_LEG0, TR_LEG>(a.t.leg, T, qv, inv_mass, sm + TP_LEG * 32);
    tree_frame2<P::frot(0), P::ftmask(0)>(T, a.t.leg.ft, Rf, pf);
  }
  team.sync();
  {
    float2 T[12];
#pragma unroll
    for (int e = 0; e < 12; ++e) T[e] = both(T19[e]);
    Carm = tree_limbs<P, TR_ARM0, TR_ARM>(a.t.arm, T, qv, inv_mass, sm + TP_ARM * 32);
    tree_frame2<P::frot(2), P::ftmask(2)>(T, a.t.arm.ft, Rh, ph);
  }
  team.sync();
  // error rotations and translations: the feet, R_err = P^-1_R R_a Q^-1_R,
  // t = P^-1_R x + P^-1_p at x = p_a + R_a Q^-1_p; the hands, G = P^-1_R R_a^T,
  // R_err = G R_b, t = G (p_b - p_a) + P^-1_p
  float2 Ef[9], tf[3];
  float G[9], Eh[9], th[3];
  PosePair ef;
  {
    float2 RaQ[9];
    mul33_2(Rf, a.t.Qr, RaQ);
    mul33_2(a.t.Pr, RaQ, Ef);
    ef.x = pf;
#pragma unroll
    for (int k = 0; k < 3; ++k)
      ef.x = V3p{fma2(Rf[k], a.t.Qp[k], ef.x.x), fma2(Rf[3 + k], a.t.Qp[k], ef.x.y),
                 fma2(Rf[6 + k], a.t.Qp[k], ef.x.z)};
#pragma unroll
    for (int r = 0; r < 3; ++r) tf[r] = add2(row2(a.t.Pr + 3 * r, ef.x), a.t.Pp[r]);
    float Pr[9], RaT[9], Rb[9];
    load_R(m.cPinv[2], Pr);
    const V3<float> Pp = load_p(m.cPinv[2]);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        RaT[3 * r + c] = Rh[3 * c + r].x;
        Rb[3 * r + c] = Rh[3 * r + c].y;
      }
    mul33(Pr, RaT, G);
    mul33(G, Rb, Eh);
    const V3<float> tx = mulv(G, V3<float>{ph.x.y - ph.x.x, ph.y.y - ph.y.x, ph.z.y - ph.z.x});
    th[0] = __fadd_rn(tx.x, Pp.x);
    th[1] = __fadd_rn(tx.y, Pp.y);
    th[2] = __fadd_rn(tx.z, Pp.z);
  }
  // log maps: left foot, right foot, hands, one copy of the code
  float n2[3];
  V3<float> phi[3];
  float beta[3];
#pragma unroll 1
  for (int s = 0; s < 3; ++s) {
    float E[9], t[3];
#pragma unroll
    for (int i = 0; i < 9; ++i) E[i] = s == 0 ? Ef[i].x : (s == 1 ? Ef[i].y : Eh[i]);
#pragma unroll
    for (int i = 0; i < 3; ++i) t[i] = s == 0 ? tf[i].x : (s == 1 ? tf[i].y : th[i]);
    const auto lg = so3_log<OpsF32, float>(E);
    const float be = jl_inv_beta<float>(lg.theta, lg.s, lg.c);
    const float f[6] = {t[0], t[1], t[2], lg.phi.x, lg.phi.y, lg.phi.z};
    const float n = fmaf(f[0], f[0], fmaf(f[1], f[1], fmaf(f[2], f[2], fmaf(f[3], f[3], fmaf(f[4], f[4], f[5] * f[5])))));
#pragma unroll
    for (int u = 0; u < 3; ++u)
      if (s == u) {
        n2[u] = n;
        phi[u] = lg.phi;
        beta[u] = be;
#pragma unroll
        for (int i = 0; i < 6; ++i) F[6 * u + i] = f[i];
      }
  }
  ef.phi = V3p{make_float2(phi[0].x, phi[1].x), make_float2(phi[0].y, phi[1].y), make_float2(phi[0].z, phi[1].z)};
  ef.nphi = neg2(ef.phi);
  ef.beta = make_float2(beta[0], beta[1]);
  // trunk moments and CoM columns, the CoM residual
  float r2c;
  [[maybe_unused]] int hmode = 2;
  [[maybe_unused]] float hn0 = 0.f, hn1 = 0.f;
  {
    const auto base_com = [&](int i, V3<float> C) {
      const float2 *b = sm + (TP_BASE + 7 * i) * 32;
      return tree_com_col(V3<float>{b[0].x, b[32].x, b[64].x}, V3<float>{b[96].x, b[128].x, b[160].x}, C, m.msub[3 + i],
                          inv_mass);
    };
    V3<float> C = tree_add(tree_add(tree_add(mw[1], Cneck), V3<float>{Carm.x.x, Carm.y.x, Carm.z.x}),
                           V3<float>{Carm.x.y, Carm.y.y, Carm.z.y});
    at(TP_UP + 1) = tree_com_col(zw[1], ow[1], C, m.msub[TR_TORSO], inv_mass);
    C = tree_add(mw[0], C);
    at(TP_UP) = tree_com_col(zw[0], ow[0], C, m.msub[TR_WAIST], inv_mass);
    C = tree_add(tree_add(tree_add(mb[2], V3<float>{Cleg.x.x, Cleg.y.x, Cleg.z.x}),
                          V3<float>{Cleg.x.y, Cleg.y.y, Cleg.z.y}), C);
    at(TP_BASE + 7 * 2 + 6) = base_com(2, C);
    C = tree_add(mb[1], C);
    at(TP_BASE + 7 * 1 + 6) = base_com(1, C);
    C = tree_add(mb[0], C);
    at(TP_BASE + 6) = base_com(0, C);
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
  const float r2 = __fadd_rn(__fadd_rn(n2[0], n2[1]), __fadd_rn(n2[2], r2c));
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
#pragma unroll 1
    for (int l = 0; l < TR_LEG + TR_ARM; ++l) {
      const float2 gx = at(TP_LEG + 8 * l + 6), gy = at(TP_LEG + 8 * l + 7);
      const float2 u = fold(make_float2(gx.x, gy.x)), w = fold(make_float2(gx.y, gy.y));
      at(TP_LEG + 8 * l + 6) = make_float2(u.x, w.x);
      at(TP_LEG + 8 * l + 7) = make_float2(u.y, w.y);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) at(TP_UP + i) = fold(at(TP_UP + i));
  }
  // Gram matrix (then its factor) in packed lower-triangular form; only the
  // structural nonzeros are touched
  float L[K * (K + 1) / 2];
  float2 ca[3], cl[3];  // CoM block: partial sums of the arms and of the legs
#pragma unroll
  for (int i = 0; i < 3; ++i) ca[i] = cl[i] = make_float2(0.f, 0.f);
  const auto com_add2 = [](float2 (&p)[3], float2 gx, float2 gy) {
    p[0] = fma2(gx, gx, p[0]);
    p[1] = fma2(gy, gx, p[1]);
    p[2] = fma2(gy, gy, p[2]);
  };
  // hands' block and their CoM rows, with the arms' segments built in place
  // (joints above frame a enter with -1, above b with +1): the left arm's
  // joints first, then the right's
  {
    float H[21], CH[12];
#pragma unroll
    for (int i = 0; i < 21; ++i) H[i] = 0.f;
#pragma unroll
    for (int i = 0; i < 12; ++i) CH[i] = 0.f;
    const auto add = [&](const float (&f)[6], float gx, float gy) {
#pragma unroll
      for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int k = 0; k <= i; ++k) H[tri(i, k)] = fmaf(f[i], f[k], H[tri(i, k)]);
        CH[i] = fmaf(gx, f[i], CH[i]);
        CH[6 + i] = fmaf(gy, f[i], CH[6 + i]);
      }
    };
    float2 G2[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) G2[i] = make_float2(-G[i], G[i]);
    PosePair eh;
    eh.x = V3p{both(ph.x.y), both(ph.y.y), both(ph.z.y)};
    eh.phi = V3p{both(phi[2].x), both(phi[2].y), both(phi[2].z)};
    eh.nphi = neg2(eh.phi);
    eh.beta = both(beta[2]);
    float2 *arm = sm + TP_ARM * 32;
#pragma unroll 1
    for (int l = 0; l < TR_ARM; ++l, arm += 8 * 32) {
      float2 v[6];
      float f[6];
      seg6_2(G2, eh, load_axis(arm), load_origin(arm), v);
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        arm[r * 32] = v[r];
        f[r] = v[r].x;
      }
      const float2 gx = arm[6 * 32], gy = arm[7 * 32];
      com_add2(ca, gx, gy);
      add(f, gx.x, gy.x);
    }
    arm = sm + TP_ARM * 32;
#pragma unroll 1
    for (int l = 0; l < TR_ARM; ++l, arm += 8 * 32) {
      float f[6];
#pragma unroll
      for (int r = 0; r < 6; ++r) f[r] = arm[r * 32].y;
      add(f, arm[6 * 32].y, arm[7 * 32].y);
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
  // feet: diagonal blocks and CoM rows (left and right together), right
  // against left, with the segments built on the way
  {
    float2 B[21], C[12];
#pragma unroll
    for (int i = 0; i < 21; ++i) B[i] = i < 6 ? a.t.LL[i < 6 ? i : 0] : make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      const int r = i / 6, k = i % 6;
      if (k >= 3) {
        C[i] = make_float2(0.f, 0.f);
      } else if constexpr (!HULL) {
        C[i] = a.t.CL[3 * r + (k < 3 ? k : 0)];
      } else {
        C[i] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 3; ++j) C[i] = fma2(both(r == 0 ? jc[j].x : jc[j].y), a.t.jt[j][k < 3 ? k : 0], C[i]);
      }
    }
    const auto add = [&](const float2 (&f)[6], float2 gx, float2 gy) {
#pragma unroll
      for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int k = 0; k <= i; ++k) B[tri(i, k)] = fma2(f[i], f[k], B[tri(i, k)]);
        C[i] = fma2(gx, f[i], C[i]);
        C[6 + i] = fma2(gy, f[i], C[6 + i]);
      }
    };
    float2 Pr[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) Pr[i] = a.t.Pr[i];
    // the base's joints, then the legs', in one loop body
#pragma unroll 1
    for (int l = 0; l < 3 + TR_LEG; ++l) {
      float2 *s = sm + (l < 3 ? TP_BASE + 7 * l : TP_LEG + 8 * (l - 3)) * 32;
      float2 v[6];
      seg6_2(Pr, ef, load_axis(s), load_origin(s), v);
#pragma unroll
      for (int r = 0; r < 6; ++r) s[r * 32] = v[r];
      float2 gx = s[6 * 32], gy = s[7 * 32];
      if (l < 3) {  // one column for both feet; the CoM block takes it later
        gy = both(gx.y);
        gx = both(gx.x);
      } else {
        com_add2(cl, gx, gy);
      }
      add(v, gx, gy);
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
#pragma unroll
      for (int k = 0; k <= i; ++k) {
        L[tri(i, k)] = B[tri(i, k)].x;
        L[tri(6 + i, 6 + k)] = B[tri(i, k)].y;
      }
      L[tri(18, i)] = C[i].x;
      L[tri(18, 6 + i)] = C[i].y;
      L[tri(19, i)] = C[6 + i].x;
      L[tri(19, 6 + i)] = C[6 + i].y;
    }
    // right foot against left: the base's joints only
    {
      float X[36];
#pragma unroll
      for (int i = 0; i < 36; ++i) X[i] = i / 6 < 3 && i % 6 < 3 ? a.t.LR[i / 6 < 3 && i % 6 < 3 ? 3 * (i / 6) + i % 6 : 0] : 0.f;
#pragma unroll 1
      for (int b = 0; b < 3; ++b) {
        float2 v[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) v[r] = sm[(TP_BASE + 7 * b + r) * 32];
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
          for (int k = 0; k < 6; ++k) X[6 * i + k] = fmaf(v[i].y, v[k].x, X[6 * i + k]);
      }
#pragma unroll
      for (int i = 0; i < 36; ++i) L[tri(6 + i / 6, i % 6)] = X[i];
    }
    // CoM block: four partial sums (the arms, the left leg and the neck, the
    // right leg), then the trunk joints, each in its partial
    float p[4][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      p[0][i] = ca[i].x;
      p[1][i] = ca[i].y;
      p[2][i] = cl[i].x;
      p[3][i] = cl[i].y;
    }
    const auto put = [&](int g, float2 c) {
      p[g][0] = fmaf(c.x, c.x, p[g][0]);
      p[g][1] = fmaf(c.y, c.x, p[g][1]);
      p[g][2] = fmaf(c.y, c.y, p[g][2]);
    };
    put(2, at(TP_UP + 2));
    put(2, at(TP_UP + 3));
    static_for<6>([&](auto JJ) {
      constexpr int j = decltype(JJ)::value;
      if constexpr (j < 3) put(tree_part(j), jc[j]);
      else put(tree_part(j), at(TP_BASE + 7 * (j - 3) + 6));
    });
    put(tree_part(TR_WAIST), at(TP_UP));
    put(tree_part(TR_TORSO), at(TP_UP + 1));
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
  float t[K], yh[6], yc[2], db[3];
  float2 yf[6];  // y of the feet (left, right); yh: of the hands; yc: of the CoM rows
  float2 sa = make_float2(0.f, 0.f), sl = sa;  // |dq|^2: partial sums of the arms, of the legs
#pragma unroll
  for (int i = 0; i < K; ++i) t[i] = F[i];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    yf[i] = make_float2(0.f, 0.f);
    yh[i] = 0.f;
  }
  yc[0] = yc[1] = 0.f;
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
    for (int i = 0; i < 6; ++i) {
      yf[i] = make_float2(__fadd_rn(yf[i].x, t[i]), __fadd_rn(yf[i].y, t[6 + i]));
      yh[i] = __fadd_rn(yh[i], t[12 + i]);
    }
    yc[0] = __fadd_rn(yc[0], t[18]);
    yc[1] = __fadd_rn(yc[1], t[19]);
    // per joint: dq_j = J_j . y and, for the refinement, r += J_j dq_j
    const bool last = pass == 1;
    float2 rf[6], pl[2];  // feet: r; CoM partial sums of the legs, of the arms
    float pa[2][2];
    float dqb[6], rh[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      rf[i] = make_float2(0.f, 0.f);
      rh[i] = 0.f;
    }
    sa = sl = pl[0] = pl[1] = make_float2(0.f, 0.f);
    pa[0][0] = pa[0][1] = pa[1][0] = pa[1][1] = 0.f;
    const auto com_dot = [&](float2 c, float acc) { return fmaf(c.x, yc[0], fmaf(c.y, yc[1], acc)); };
    // base: prismatic columns are constants (their rotational rows zero)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      float acc = 0.f;
      acc = fmaf(a.t.jt[i][0].x, yf[0].x, fmaf(a.t.jt[i][1].x, yf[1].x, acc));
      acc = fmaf(a.t.jt[i][2].x, yf[2].x, acc);
      acc = fmaf(a.t.jt[i][0].y, yf[0].y, fmaf(a.t.jt[i][1].y, yf[1].y, acc));
      acc = fmaf(a.t.jt[i][2].y, yf[2].y, acc);
      dqb[i] = com_dot(jc[i], acc);
#pragma unroll
      for (int k = 0; k < 3; ++k) rf[k] = fma2(a.t.jt[i][k], both(dqb[i]), rf[k]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      float2 v[6];
#pragma unroll
      for (int r = 0; r < 6; ++r) v[r] = at(TP_BASE + 7 * b + r);
      float acc = 0.f;
#pragma unroll
      for (int r = 0; r < 6; r += 2) acc = fmaf(v[r].x, yf[r].x, fmaf(v[r + 1].x, yf[r + 1].x, acc));
#pragma unroll
      for (int r = 0; r < 6; r += 2) acc = fmaf(v[r].y, yf[r].y, fmaf(v[r + 1].y, yf[r + 1].y, acc));
      dqb[3 + b] = com_dot(at(TP_BASE + 7 * b + 6), acc);
#pragma unroll
      for (int r = 0; r < 6; ++r) rf[r] = fma2(v[r], both(dqb[3 + b]), rf[r]);
    }
    // limbs: the scaled step of the last pass stays in the joint's first slot
    {
      float2 *leg = sm + TP_LEG * 32;
#pragma unroll 1
      for (int l = 0; l < TR_LEG; ++l, leg += 8 * 32) {
        float2 v[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) v[r] = leg[r * 32];
        const float2 gx = leg[6 * 32], gy = leg[7 * 32];
        float2 d = make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < 6; r += 2) d = fma2(v[r], yf[r], fma2(v[r + 1], yf[r + 1], d));
        d = fma2(gx, both(yc[0]), fma2(gy, both(yc[1]), d));
        pl[0] = fma2(gx, d, pl[0]);
        pl[1] = fma2(gy, d, pl[1]);
#pragma unroll
        for (int r = 0; r < 6; ++r) rf[r] = fma2(v[r], d, rf[r]);
        const float2 e = mul2(d, both(a.alpha));
        sl = fma2(e, e, sl);
        if (last) leg[0] = e;
      }
    }
    // the arms one after the other (r sums the left arm's terms first)
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      float sq = 0.f;
      float *arm = reinterpret_cast<float *>(sm + TP_ARM * 32) + s;
#pragma unroll 1
      for (int l = 0; l < TR_ARM; ++l, arm += 8 * 64) {
        float v[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) v[r] = arm[r * 64];
        const float gx = arm[6 * 64], gy = arm[7 * 64];
        float d = 0.f;
#pragma unroll
        for (int r = 0; r < 6; r += 2) d = fmaf(v[r], yh[r], fmaf(v[r + 1], yh[r + 1], d));
        d = fmaf(gx, yc[0], fmaf(gy, yc[1], d));
        pa[s][0] = fmaf(gx, d, pa[s][0]);
        pa[s][1] = fmaf(gy, d, pa[s][1]);
#pragma unroll
        for (int r = 0; r < 6; ++r) rh[r] = fmaf(v[r], d, rh[r]);
        const float e = __fmul_rn(d, a.alpha);
        sq = fmaf(e, e, sq);
        if (last) arm[0] = e;
      }
      if (s == 0) sa.x = sq;
      else sa.y = sq;
    }
    // neck, then the trunk joints, each in its partial sum
    float pc[4][2] = {{pa[0][0], pa[0][1]}, {pa[1][0], pa[1][1]}, {pl[0].x, pl[1].x}, {pl[0].y, pl[1].y}};
    float sp[4] = {sa.x, sa.y, sl.x, sl.y};
    const auto step = [&](int g, float d, float2 c) -> float {
      pc[g][0] = fmaf(c.x, d, pc[g][0]);
      pc[g][1] = fmaf(c.y, d, pc[g][1]);
      const float e = __fmul_rn(d, a.alpha);
      sp[g] = fmaf(e, e, sp[g]);
      return e;
    };
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
    sa = make_float2(sp[0], sp[1]);
    sl = make_float2(sp[2], sp[3]);
    if (last) break;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      t[i] = fmaf(-a.lambda, yf[i].x, __fadd_rn(F[i], -rf[i].x));
      t[6 + i] = fmaf(-a.lambda, yf[i].y, __fadd_rn(F[6 + i], -rf[i].y));
      t[12 + i] = fmaf(-a.lambda, yh[i], __fadd_rn(F[12 + i], -rh[i]));
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float s = __fadd_rn(__fadd_rn(pc[0][i], pc[1][i]), __fadd_rn(pc[2][i], pc[3][i]));
      t[18 + i] = fmaf(-a.lambda, yc[i], __fadd_rn(F[18 + i], -s));
    }
  }
  // MaxDistance, update (the scaled steps lie in the first word of each joint's slot)
  const float s2 = __fadd_rn(__fadd_rn(sa.x, sa.y), __fadd_rn(sl.x, sl.y));
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
    for (int l = 0; l < TR_LEG; ++l) {
      const float2 e = at(TP_LEG + 8 * l);
      q[TR_LEG0 + l] = __fadd_rn(q[TR_LEG0 + l], -e.x);
      q[TR_LEG0 + TR_LEG + l] = __fadd_rn(q[TR_LEG0 + TR_LEG + l], -e.y);
    }
#pragma unroll
    for (int l = 0; l < TR_ARM; ++l) {
      const float2 e = at(TP_ARM + 8 * l);
      q[TR_ARM0 + l] = __fadd_rn(q[TR_ARM0 + l], -e.x);
      q[TR_ARM0 + TR_ARM + l] = __fadd_rn(q[TR_ARM0 + TR_ARM + l], -e.y);
    }
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
// the team has nothing else to do, with or without the token.
// Whether a failed acceptance goes back is decided by the configuration alone
// (never by what the warp holds at that moment, which depends on the other
// warps): a warp accepts no more than still fit among its retries, and fills
// idle lanes only with at most 64 parked.  New work is claimed when every retry
// has found a lane; the warp then holds its lanes and at most 64 parked, and as
// nothing else adds to them, never more than 96.  With more than 64 parked, at
// most 31 retries are therefore waiting, and an acceptance can go on.
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
  long long an = 0, ae = 0;  // the chunk after it, claimed ahead and on its way into L2
  const long long margin = 2ll * a.chunk * gridDim.x * warps;
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
    const unsigned idle = __ballot_sync(FULL, !act && pend <= 32 * (TREE_SLOTS - 1));
    if (idle != 0u && (nret > 0 || qn < qe || an < ae || more)) {
      const int n_idle = __popc(idle);
      const int from_r = n_idle < nret ? n_idle : nret;
      const int need = n_idle - from_r;
      const long long avail = qe - qn;
      long long b0 = 0, b1 = 0;
      const auto claim = [&](long long &lo, long long &hi) {
        unsigned long long b = 0;
        if (lane == 0) b = atomicAdd(a.counter, static_cast<unsigned long long>(a.chunk));
        b = __shfl_sync(FULL, b, 0);
        if (static_cast<long long>(b) >= a.total) {
          more = false;
        } else {
          lo = static_cast<long long>(b);
          hi = lo + a.chunk < a.total ? lo + a.chunk : a.total;
        }
      };
      if (need > 0 && avail < need) {
        if (an < ae) {
          b0 = an;
          b1 = ae;
          an = ae = 0;
        } else if (more) {
          claim(b0, b1);
        }
        // while much work is left, the next chunk's rows start towards L2 now
        // (not near the end, where a chunk held back would leave others idle)
        if (more && b1 + margin < a.total) {
          claim(an, ae);
          if (an < ae)
            for (int j = lane; j < D; j += 32) {
              const float *row = a.src.q + j * a.src.ld;
              asm volatile("prefetch.global.L2 [%0];" ::"l"(row + an));
              asm volatile("prefetch.global.L2 [%0];" ::"l"(row + ae - 1));
            }
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
    const bool drained = !__any_sync(FULL, act) && qn >= qe && an >= ae && !more && nret == 0;
    // FP64 acceptance, one configuration per lane, 32 at a time; a failed
    // acceptance with steps left goes back to the FP32 loop
    bool accept = false, token = false;
    const bool full = team.any(pend > 32 * (TREE_SLOTS - 1)), wait = team.any(pend < 32 && !drained);
    if (full || !wait) {
      if (wib == team0 && lane == 0) token = atomicCAS(&fp64_taken, 0, 1) == 0;
      accept = full || team.any(token || drained);
    }
    const int take = min(min(pend, 32), 32 - nret);  // as many as could all be sent back
    if (accept && take > 0 && (take >= TREE_ACCEPT_MIN || drained || pend > 32 * (TREE_SLOTS - 1))) {
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
      if (lane < take) retry = accept_one<P, FORM_STACKED>(a, it_item, static_cast<int>(meta & 0xffu), meta >> 8);
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
  cudaError_t err = allow_smem(kern, tree_smem_bytes<P>(TREE_WARPS));
  if (err != cudaSuccess) return err;
  long long blocks = (warps + w - 1) / w;
  if (blocks > hm.sm_count) blocks = hm.sm_count;
  err = cudaMemsetAsync(c.counter, 0, sizeof(unsigned long long), c.stream);
  if (err != cudaSuccess) return err;
  kern<<<static_cast<unsigned>(blocks), static_cast<unsigned>(w) * 32, smem, c.stream>>>(a);
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace mcp
