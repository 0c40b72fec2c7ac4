// FP32 Newton step of the dual arm (two copies of one 7-joint chain under the
// relative pose of their end frames, Eq. 2), one lane per configuration, both
// chains in every instruction.
//
// What bounds it: instruction fetch.  Unrolled for one configuration in
// registers the step is 2,900 instructions (46 KB): with 11 unsynchronised
// warps on an SM two thirds of their time go to waiting for instructions
// (5.9 of 8 cycles per issue, 0.27 instructions per cycle and scheduler).  With
// fewer warps on an SM that step is still the faster one (dual_in_registers).
// Here the chains are the two halves of packed FP32x2 operations
// (mcp_pack.cuh), the Jacobian lives in shared memory (49 float2 per lane,
// lane-major) and is built and used in loops over the chain's joints: about
// 1,000 instructions of code, 2,000 executed, and registers for 16 warps on an
// SM instead of 12.
//
// Every sum is taken in the order of newton_iter_f32 on this class (left arm's
// joints, then the right's), on the same operands: the results are its bits.
#pragma once

#include <cfloat>

#include "mcp_accept.cuh"
#include "mcp_pack.cuh"

namespace mcp {

constexpr int DUAL_PAIRS = 49;  // 6 per joint of a chain, and its steps

// P is one chain twice: joints 0 .. H-1 and H .. 2H-1, end frames 0 and 1.
template <class P>
__host__ __device__ constexpr bool dual_layout_matches() {
  constexpr int H = P::D / 2;
  if (P::D % 2 != 0 || P::NF != 2 || P::NC != 1) return false;
  if (P::ckind(0) != K_REL || P::cfa(0) != 0 || P::cfb(0) != 1) return false;
  for (int j = 0; j < H; ++j) {
    if (P::parent(j) != j - 1 || P::parent(H + j) != (j == 0 ? -1 : H + j - 1)) return false;
    if (P::jtype(j) != REV || P::jtype(H + j) != REV) return false;
    if (P::xrot(j) != P::xrot(H + j) || P::xtmask(j) != P::xtmask(H + j) || P::xrot(j) == XR_GENERIC) return false;
  }
  return P::frame_link(0) == H - 1 && P::frame_link(1) == 2 * H - 1 && P::frot(0) == P::frot(1) &&
         P::ftmask(0) == P::ftmask(1) && P::frot(0) != XR_GENERIC;
}

// packed counterparts of pat_value / pat_fma / pat_rotate
template <int A>
__device__ __forceinline__ float2 pat2_value(float2 v) {
  return A == PZ ? both(0.f) : (A == PP ? both(1.f) : (A == PN ? both(-1.f) : v));
}
template <int A>
__device__ __forceinline__ float2 pat2_fma(float2 v, float2 t, float2 p) {
  if constexpr (A == PZ) return p;
  else if constexpr (A == PP) return add2(p, t);
  else if constexpr (A == PN) return sub2(p, t);
  else return fma2(v, t, p);
}
template <int A>
__device__ __forceinline__ float2 pat2_times(float2 x, float2 nx, float2 v) {  // x v, with nx = -x
  if constexpr (A == PP) return x;
  else if constexpr (A == PN) return nx;
  else return mul2(x, v);
}
template <int A, int B>
__device__ __forceinline__ void pat2_rotate(float2 c, float2 nc, float2 s, float2 ns, float2 &a, float2 &b) {
  const float2 a0 = a, b0 = b;
  if constexpr (A == PZ && B == PZ) {
    return;
  } else if constexpr (B == PZ) {
    a = pat2_times<A>(c, nc, a0);
    b = pat2_times<A>(ns, s, a0);
  } else if constexpr (A == PZ) {
    a = pat2_times<B>(s, ns, b0);
    b = pat2_times<B>(c, nc, b0);
  } else {
    static_assert(A == PG && B == PG, "a signed axis stands alone in its row");
    a = fma2(c, a0, mul2(s, b0));
    b = fma2(c, b0, mul2(ns, a0));
  }
}

// One FP32 Newton iteration (newton_iter_f32's exits, flags and results).  sm:
// this lane's slots, pair e at sm[e * 32].
template <class P, class A>
__device__ __forceinline__ bool dual_iter_f32(const A &a, float2 *__restrict__ sm, float (&q)[P::D], int &it, uint32_t &fl) {
  static_assert(dual_layout_matches<P>(), "not two copies of one chain");
  constexpr int D = P::D, H = D / 2, K = 6;
  const ModelT<float> &m = a.m;
  float G[9], F[K], pb[3], beta;
  V3<float> phi;
  {
    // FK of both chains: axes and origins into the slots
    float2 R[9], p[3];
    float R0[9];
    root_xrot<P::xrot(0)>(m.X[0], R0);
#pragma unroll
    for (int e = 0; e < 9; ++e) R[e] = both(R0[e]);
#pragma unroll
    for (int r = 0; r < 3; ++r) p[r] = make_float2(m.X[0][4 * r + 3], m.X[H][4 * r + 3]);
    static_for<H>([&](auto JJ) {
      constexpr int j = decltype(JJ)::value;
      constexpr Pat9 b = PatOf<P, j>::before;
      if constexpr (j > 0) {
        constexpr Pat9 u = PatOf<P, j - 1>::after;
        static_for<9>([&](auto EE) {
          constexpr int r = decltype(EE)::value % 3, k = decltype(EE)::value / 3;
          if constexpr ((P::xtmask(j) >> k) & 1)
            p[r] = pat2_fma<u.e[3 * r + k]>(R[3 * r + k], make_float2(m.X[j][4 * k + 3], m.X[H + j][4 * k + 3]), p[r]);
        });
        float2 Rn[9];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const float2 v = R[3 * r + xr_perm(P::xrot(j), k)];
            Rn[3 * r + k] = xr_neg(P::xrot(j), k) ? neg2(v) : v;
          }
#pragma unroll
        for (int e = 0; e < 9; ++e) R[e] = Rn[e];
      }
      static_for<3>([&](auto RR) {
        constexpr int r = decltype(RR)::value;
        sm[(6 * j + r) * 32] = pat2_value<b.e[3 * r + 2]>(R[3 * r + 2]);
        sm[(6 * j + 3 + r) * 32] = p[r];
      });
      float2 s, c;
      sincos2_f32(make_float2(q[j], q[H + j]), s, c);
      const float2 ns = neg2(s), nc = neg2(c);
      static_for<3>([&](auto RR) {
        constexpr int r = decltype(RR)::value;
        pat2_rotate<b.e[3 * r], b.e[3 * r + 1]>(c, nc, s, ns, R[3 * r], R[3 * r + 1]);
      });
    });
    constexpr Pat9 u = PatOf<P, H - 1>::after;
    static_for<9>([&](auto EE) {
      constexpr int r = decltype(EE)::value % 3, k = decltype(EE)::value / 3;
      if constexpr ((P::ftmask(0) >> k) & 1)
        p[r] = pat2_fma<u.e[3 * r + k]>(R[3 * r + k], make_float2(m.fX[0][4 * k + 3], m.fX[1][4 * k + 3]), p[r]);
    });
    float2 fR[9];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float2 v = R[3 * r + xr_perm(P::frot(0), k)];
        fR[3 * r + k] = xr_neg(P::frot(0), k) ? neg2(v) : v;
      }
    // Eq. 2: T_err = T_ref^-1 (T_a^-1 T_b); G = R_ref^T R_a^T
    float Pr[9], Rb[9], Rerr[9];
    load_R(m.cPinv[0], Pr);
    const V3<float> Pp = load_p(m.cPinv[0]);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        G[3 * r + k] = fmaf(Pr[3 * r], fR[3 * k].x, fmaf(Pr[3 * r + 1], fR[3 * k + 1].x, __fmul_rn(Pr[3 * r + 2], fR[3 * k + 2].x)));
        Rb[3 * r + k] = fR[3 * r + k].y;
      }
    mul33(G, Rb, Rerr);
    const V3<float> tx = mulv(G, V3<float>{__fadd_rn(p[0].y, -p[0].x), __fadd_rn(p[1].y, -p[1].x), __fadd_rn(p[2].y, -p[2].x)});
    const auto lg = so3_log<OpsF32, float>(Rerr);
    phi = lg.phi;
    beta = jl_inv_beta<float>(lg.theta, lg.s, lg.c);
    F[0] = __fadd_rn(tx.x, Pp.x);
    F[1] = __fadd_rn(tx.y, Pp.y);
    F[2] = __fadd_rn(tx.z, Pp.z);
    F[3] = phi.x;
    F[4] = phi.y;
    F[5] = phi.z;
#pragma unroll
    for (int r = 0; r < 3; ++r) pb[r] = p[r].y;
  }
  float r2 = 0.f;
#pragma unroll
  for (int i = 0; i < K; ++i) r2 = fmaf(F[i], F[i], r2);
  if (!(r2 <= FLT_MAX)) {
    fl |= FL_NONFINITE;
    return true;
  }
  if (r2 < a.tol2 && !(fl & FL_INT_FORCE)) {
    fl |= FL_INT_FP32CONV;
    return true;
  }
  if (it >= a.cap) {
    fl |= FL_CAP;
    return true;
  }
  // segments in place (chain a's joints enter with -1, chain b's with +1) and
  // A = J J^T + lambda I over the left joints, then over the right
  float L[K * (K + 1) / 2], inv[K];
#pragma unroll
  for (int i = 0; i < K; ++i)
#pragma unroll
    for (int k = 0; k <= i; ++k) L[tri(i, k)] = i == k ? a.lambda : 0.f;
  const auto add = [&](const float (&f)[K]) {
#pragma unroll
    for (int i = 0; i < K; ++i)
#pragma unroll
      for (int k = 0; k <= i; ++k) L[tri(i, k)] = fmaf(f[i], f[k], L[tri(i, k)]);
  };
  {
    float2 G2[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) G2[i] = make_float2(-G[i], G[i]);
    PosePair e;
    e.x = V3p{both(pb[0]), both(pb[1]), both(pb[2])};
    e.phi = V3p{both(phi.x), both(phi.y), both(phi.z)};
    e.nphi = neg2(e.phi);
    e.beta = both(beta);
    float2 *s = sm;
#pragma unroll 1
    for (int j = 0; j < H; ++j, s += 6 * 32) {
      float2 v[6];
      float f[K];
      seg6_2(G2, e, V3p{s[0], s[32], s[64]}, V3p{s[96], s[128], s[160]}, v);
#pragma unroll
      for (int r = 0; r < K; ++r) {
        s[r * 32] = v[r];
        f[r] = v[r].x;
      }
      add(f);
    }
    s = sm;
#pragma unroll 1
    for (int j = 0; j < H; ++j, s += 6 * 32) {
      float f[K];
#pragma unroll
      for (int r = 0; r < K; ++r) f[r] = s[r * 32].y;
      add(f);
    }
  }
  const float piv = cholesky_factor<K, OpsF32>(L, inv);
  if (!(piv >= a.pivot)) {  // also catches NaN: finish this configuration in FP64
    fl |= FL_INT_NEEDS_F64;
    return true;
  }
  // y = A^-1 F, then y += A^-1 (F - J (J^T y) - lambda y); dq = J^T y in the
  // slots 6 H .. 7 H - 1
  float y[K], b[K];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    y[i] = 0.f;
    b[i] = F[i];
  }
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    cholesky_subst<K>(L, inv, b);
    float2 y2[K];
    float r[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
      y[i] += b[i];
      y2[i] = both(y[i]);
      r[i] = 0.f;
    }
    float2 *s = sm;
#pragma unroll 1
    for (int j = 0; j < H; ++j, s += 6 * 32) {
      float2 v[K], d = both(0.f);
#pragma unroll
      for (int i = 0; i < K; ++i) {
        v[i] = s[i * 32];
        d = fma2(v[i], y2[i], d);
      }
      sm[(6 * H + j) * 32] = d;
#pragma unroll
      for (int i = 0; i < K; ++i) r[i] = fmaf(v[i].x, d.x, r[i]);
    }
    if (pass == 1) break;
    s = sm;
#pragma unroll 1
    for (int j = 0; j < H; ++j, s += 6 * 32) {
      const float d = sm[(6 * H + j) * 32].y;
#pragma unroll
      for (int i = 0; i < K; ++i) r[i] = fmaf(s[i * 32].y, d, r[i]);
    }
#pragma unroll
    for (int i = 0; i < K; ++i) b[i] = fmaf(-a.lambda, y[i], F[i] - r[i]);
  }
  float dq[D];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const float2 d = sm[(6 * H + j) * 32];
    dq[j] = d.x;
    dq[H + j] = d.y;
  }
  float s2 = 0.f;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    dq[j] *= a.alpha;
    s2 = fmaf(dq[j], dq[j], s2);
  }
  if (a.max_step2 > 0.f && s2 > a.max_step2) {
    fl |= FL_DIV;
    return true;
  }
#pragma unroll
  for (int j = 0; j < D; ++j) q[j] -= dq[j];
  ++it;
  fl &= ~FL_INT_FORCE;
  if (!(s2 <= FLT_MAX)) {
    fl |= FL_NONFINITE;
    return true;
  }
  return false;
}

}  // namespace mcp
