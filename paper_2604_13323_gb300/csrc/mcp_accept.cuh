// The FP64 residual of an FP32 iterate: what decides whether a configuration
// is accepted, and the residual that is returned with it.
//
// What bounds it: the FP64 unit.  On this part an FP64 add, multiply or fma of
// a warp takes 19 cycles of its SM (64 when a single warp issues them), while
// an FP32 instruction takes a quarter of a cycle and conversions between the
// two about 4; so the number of FP64 instructions is the cost.  Against the
// general FK and residual (which the FP32 and plain FP64 kernels use):
//   * entries of the link rotations that are 0 or +-1 by the structure of the
//     tree (a chain's first joints) are followed at compile time;
//   * sin and cos cost 6 FP64 operations (sincos_f64_split_f);
//   * only the off-diagonal entries of an error rotation are formed in FP64:
//     near the identity the squared angle follows from them, and the trace
//     only tells that case from the others, which FP32 can;
//   * a link's CoM terms with a zero offset or a zero mass, and a TSR's
//     identity offset, are skipped (masks made when the model is loaded).
// Counted in this source, FP64 operations per configuration: arm 90 -> 47, dual
// arm 450 -> 320, humanoid 1,468 -> 950.  Measured: arm, 65,536, 40.5 -> 38.2 us;
// dual arm, 262,144 waypoints near the manifold, 364 -> 341 us, its segments 649
// -> 621 us; extensions 1,170 -> 1,113 us; humanoid, 1,048,576 with the check,
// 8.34 -> 8.03 ms.
#pragma once

#include <cfloat>

#include "mcp_device.cuh"
#include "mcp_problems.cuh"

namespace mcp {

// ---------------------------------------------------------------------------
// Entries of a rotation known at compile time
// ---------------------------------------------------------------------------
enum : int { PZ = 0, PP = 1, PN = 2, PG = 3 };  // 0, +1, -1, a run-time value
struct Pat9 {
  int e[9];
};
__host__ __device__ constexpr Pat9 pat_identity() { return Pat9{{PP, PZ, PZ, PZ, PP, PZ, PZ, PZ, PP}}; }
__host__ __device__ constexpr Pat9 pat_offset(Pat9 in, int code) {  // times a fixed rotation
  Pat9 o{};
  for (int k = 0; k < 3; ++k)
    for (int r = 0; r < 3; ++r) {
      if (code == XR_GENERIC) {
        o.e[3 * r + k] = PG;
      } else {
        const int v = in.e[3 * r + xr_perm(code, k)];
        o.e[3 * r + k] = !xr_neg(code, k) ? v : (v == PP ? PN : (v == PN ? PP : v));
      }
    }
  return o;
}
template <class P>
__host__ __device__ constexpr Pat9 pat_link(int j) {  // joint frame j after its motion
  Pat9 o = pat_offset(P::parent(j) < 0 ? pat_identity() : pat_link<P>(P::parent(j)), P::xrot(j));
  if (P::jtype(j) == REV)
    for (int r = 0; r < 3; ++r)
      if (o.e[3 * r] != PZ || o.e[3 * r + 1] != PZ) o.e[3 * r] = o.e[3 * r + 1] = PG;
  return o;
}
template <class P, int J>
struct PatOf {
  static constexpr Pat9 before = pat_offset(P::parent(J) < 0 ? pat_identity() : pat_link<P>(P::parent(J)), P::xrot(J));
  static constexpr Pat9 after = pat_link<P>(J);
};

template <int A>
__device__ __forceinline__ double pat_value(double v) {
  return A == PZ ? 0.0 : (A == PP ? 1.0 : (A == PN ? -1.0 : v));
}
template <int A>
__device__ __forceinline__ double pat_times(double x, double v) {  // x v
  if constexpr (A == PZ) return 0.0;
  else if constexpr (A == PP) return x;
  else if constexpr (A == PN) return -x;
  else return x * v;
}
template <int A>
__device__ __forceinline__ double pat_fma(double v, double t, double p) {  // v t + p
  if constexpr (A == PZ) return p;
  else if constexpr (A == PP) return p + t;
  else if constexpr (A == PN) return p - t;
  else return fma(v, t, p);
}
// (a, b) <- (c a + s b, c b - s a)
template <int A, int B>
__device__ __forceinline__ void pat_rotate(double c, double s, double &a, double &b) {
  const double a0 = a, b0 = b;
  if constexpr (A == PZ && B == PZ) {
    return;
  } else if constexpr (B == PZ) {
    a = pat_times<A>(c, a0);
    b = -pat_times<A>(s, a0);
  } else if constexpr (A == PZ) {
    a = pat_times<B>(s, b0);
    b = pat_times<B>(c, b0);
  } else if constexpr (B != PG) {
    a = fma(c, a0, pat_times<B>(s, b0));
    b = fma(-s, a0, pat_times<B>(c, b0));
  } else if constexpr (A != PG) {
    a = fma(s, b0, pat_times<A>(c, a0));
    b = fma(c, b0, -pat_times<A>(s, a0));
  } else {
    a = fma(c, a0, s * b0);
    b = fma(c, b0, -(s * a0));
  }
}

// ---------------------------------------------------------------------------
// Squared rotation angle of R = A B
// ---------------------------------------------------------------------------
struct Rot9d {
  double r[9];
};
// the general case, out of line: far from the identity
static __device__ __noinline__ V3<double> accept_log(Rot9d R) {
  const auto lg = so3_log<OpsF64Plain, double>(R.r);
  return lg.phi;
}
__device__ __forceinline__ double entry(const double (&A)[9], const double (&B)[9], int r, int c) {
  return fma(A[3 * r], B[c], fma(A[3 * r + 1], B[3 + c], A[3 * r + 2] * B[6 + c]));
}
__device__ __forceinline__ float entry_f(const double (&A)[9], const double (&B)[9], int r) {
  return fmaf(static_cast<float>(A[3 * r]), static_cast<float>(B[r]),
              fmaf(static_cast<float>(A[3 * r + 1]), static_cast<float>(B[3 + r]),
                   static_cast<float>(A[3 * r + 2]) * static_cast<float>(B[6 + r])));
}
// The angle theta has sin theta = |w|, w = vee(R - R^T) / 2.  With D = 4 |w|^2
// below 4e-6 and a positive cosine,
//   theta^2 = asin(|w|)^2 = D / 4 + D^2 / 48 + D^3 / 360  (next term D^4 / 2240 < 4e-19 D);
// the general log map elsewhere (a cosine within 1e-3 of zero counts as
// elsewhere, so its FP32 rounding decides nothing).
__device__ __forceinline__ double accept_angle2(const double (&A)[9], const double (&B)[9]) {
  Rot9d E;
  E.r[1] = entry(A, B, 0, 1);
  E.r[2] = entry(A, B, 0, 2);
  E.r[3] = entry(A, B, 1, 0);
  E.r[5] = entry(A, B, 1, 2);
  E.r[6] = entry(A, B, 2, 0);
  E.r[7] = entry(A, B, 2, 1);
  const double d0 = E.r[7] - E.r[5], d1 = E.r[2] - E.r[6], d2 = E.r[3] - E.r[1];
  const double D = fma(d0, d0, fma(d1, d1, d2 * d2));
  const float c2 = entry_f(A, B, 0) + entry_f(A, B, 1) + entry_f(A, B, 2) - 1.f;  // 2 cos theta
  if (c2 > 1e-3f && D < 4e-6) return D * fma(D, fma(D, 1.0 / 360.0, 1.0 / 48.0), 0.25);
  E.r[0] = entry(A, B, 0, 0);
  E.r[4] = entry(A, B, 1, 1);
  E.r[8] = entry(A, B, 2, 2);
  const V3<double> phi = accept_log(E);
  return dot(phi, phi);
}

// ---------------------------------------------------------------------------
// Axis alignment only: one vector from the frame to the root
// ---------------------------------------------------------------------------
template <class P>
__host__ __device__ constexpr bool axis_only() {
  for (int c = 0; c < P::NC; ++c)
    if (P::ckind(c) != K_AXIS) return false;
  return true;
}
template <class P>
__host__ __device__ constexpr int chain_len(int link) {
  int n = 0;
  for (int l = link; l >= 0; l = P::parent(l)) ++n;
  return n;
}
template <class P>
__host__ __device__ constexpr int chain_at(int link, int k) {  // k-th joint from `link` towards the root
  int l = link;
  for (int i = 0; i < k; ++i) l = P::parent(l);
  return l;
}
// A revolute root joint whose axis is world z (X_0 without rotation) turns z
// about world z, which leaves z.x^2 + z.y^2 = |F|^2 unchanged: its rotation is
// skipped.
template <class P>
__host__ __device__ constexpr bool norm_invariant_root(int j) {
  return P::parent(j) < 0 && P::jtype(j) == REV && P::xrot(j) == XR_IDENTITY;
}
struct Pat3 {
  int e[3];
};
__host__ __device__ constexpr Pat3 pat_vec_offset(Pat3 v, int code) {  // a fixed rotation times the vector
  if (code == XR_GENERIC) return Pat3{{PG, PG, PG}};
  Pat3 o{};
  for (int k = 0; k < 3; ++k) {
    const int x = v.e[k];
    o.e[xr_perm(code, k)] = !xr_neg(code, k) ? x : (x == PP ? PN : (x == PN ? PP : x));
  }
  return o;
}
// z axis of frame f, k joints up its chain (before joint k's own rotation)
template <class P>
__host__ __device__ constexpr Pat3 pat_axis(int f, int k) {
  Pat3 v = pat_vec_offset(Pat3{{PZ, PZ, PP}}, P::frot(f));
  for (int i = 0; i < k; ++i) {
    const int j = chain_at<P>(P::frame_link(f), i);
    if (P::jtype(j) == REV && (v.e[0] != PZ || v.e[1] != PZ)) v.e[0] = v.e[1] = PG;
    v = pat_vec_offset(v, P::xrot(j));
  }
  return v;
}
template <class P, int F, int K>
struct PatAxis {
  static constexpr Pat3 value = pat_axis<P>(F, K);
};
// v <- R v for a fixed rotation given by its code (signed permutation: no arithmetic) or dense
template <int CODE>
__device__ __forceinline__ V3<double> xrot_apply(const double *X, V3<double> v) {
  if constexpr (CODE == XR_GENERIC) {
    return {fma(X[0], v.x, fma(X[1], v.y, X[2] * v.z)), fma(X[4], v.x, fma(X[5], v.y, X[6] * v.z)),
            fma(X[8], v.x, fma(X[9], v.y, X[10] * v.z))};
  } else {
    double o[3] = {0.0, 0.0, 0.0};
    const double in[3] = {v.x, v.y, v.z};
#pragma unroll
    for (int k = 0; k < 3; ++k) o[xr_perm(CODE, k)] = xr_neg(CODE, k) ? -in[k] : in[k];
    return {o[0], o[1], o[2]};
  }
}
template <class P, class Ops, typename Q>
__device__ __forceinline__ double axis_residual2_f64(const Ops &ops, const ModelT<double> &m, const Q (&q)[P::D]) {
  double r2 = 0.0;
  static_for<P::NC>([&](auto CC) {
    constexpr int c = decltype(CC)::value;
    constexpr int f = P::cfa(c);
    constexpr int l = P::frame_link(f);
    V3<double> v = xrot_apply<P::frot(f)>(m.fX[f], V3<double>{0.0, 0.0, 1.0});
    static_for<chain_len<P>(l)>([&](auto KK) {
      constexpr int k = decltype(KK)::value, j = chain_at<P>(l, k);
      constexpr Pat3 pv = PatAxis<P, f, k>::value;
      if constexpr (norm_invariant_root<P>(j)) {
        return;
      } else if constexpr (P::jtype(j) == REV && (pv.e[0] != PZ || pv.e[1] != PZ)) {
        double sn, cs;
        ops.sincos(q[j], sn, cs);
        pat_rotate<pv.e[1], pv.e[0]>(cs, sn, v.y, v.x);  // (y, x) <- (c y + s x, c x - s y)
      }
      v = xrot_apply<P::xrot(j)>(m.X[j], v);
    });
    r2 = fma(v.x, v.x, fma(v.y, v.y, r2));
  });
  return r2;
}

// ---------------------------------------------------------------------------
// General case
// ---------------------------------------------------------------------------
// A link whose CoM terms may be skipped by the masks: one with a link below it
// or a task frame on it, where a non-finite pose reaches the residual anyway.
template <class P>
__host__ __device__ constexpr bool com_skippable(int j) {
  for (int i = 0; i < P::D; ++i)
    if (P::parent(i) == j) return true;
  for (int f = 0; f < P::NF; ++f)
    if (P::frame_link(f) == j) return true;
  return false;
}

// Squared FP64 norm of F at q (FP32 values, as float or double).
template <class P, class Ops, typename Q>
__device__ __forceinline__ double residual2_f64(const Ops &ops, const ModelT<double> &m, const Q (&q)[P::D]) {
  if constexpr (axis_only<P>()) {
    return axis_residual2_f64<P>(ops, m, q);
  } else {
    constexpr bool COM = needs_com<P>();
    double R[P::D][9];
    V3<double> p[P::D];
    double fR[P::NF][9];
    V3<double> fp[P::NF];
    [[maybe_unused]] double mx = 0.0, my = 0.0;
    if constexpr (needs_fk<P>()) {
      static_for<P::D>([&](auto JJ) {
        constexpr int j = decltype(JJ)::value;
        constexpr int pa = P::parent(j), code = P::xrot(j);
        constexpr Pat9 b = PatOf<P, j>::before, a = PatOf<P, j>::after;
        if constexpr (pa < 0) {
          root_xrot<code>(m.X[j], R[j]);
          p[j] = load_p(m.X[j]);
        } else {
          constexpr Pat9 u = PatOf<P, pa>::after;
          apply_xrot<code>(R[pa], m.X[j], R[j]);
          double o[3] = {p[pa].x, p[pa].y, p[pa].z};
          static_for<9>([&](auto EE) {
            constexpr int r = decltype(EE)::value % 3, k = decltype(EE)::value / 3;
            if constexpr ((P::xtmask(j) >> k) & 1) o[r] = pat_fma<u.e[3 * r + k]>(R[pa][3 * r + k], m.X[j][4 * k + 3], o[r]);
          });
          p[j] = V3<double>{o[0], o[1], o[2]};
        }
        if constexpr (P::jtype(j) == REV) {
          double s, c;
          ops.sincos(q[j], s, c);
          static_for<3>([&](auto RR) {
            constexpr int r = decltype(RR)::value;
            pat_rotate<b.e[3 * r], b.e[3 * r + 1]>(c, s, R[j][3 * r], R[j][3 * r + 1]);
          });
        } else {
          const double d = static_cast<double>(q[j]);
          p[j] = V3<double>{pat_fma<b.e[2]>(R[j][2], d, p[j].x), pat_fma<b.e[5]>(R[j][5], d, p[j].y),
                            pat_fma<b.e[8]>(R[j][8], d, p[j].z)};
        }
        if constexpr (COM) {
          const unsigned nz = com_skippable<P>(j) ? m.com_nz[j] : 15u;
          if (nz & 8u) {
            double cx = p[j].x, cy = p[j].y;
            static_for<3>([&](auto KK) {
              constexpr int k = decltype(KK)::value;
              if ((nz >> k) & 1u) {
                cx = pat_fma<a.e[k]>(R[j][k], m.com[j][k], cx);
                cy = pat_fma<a.e[3 + k]>(R[j][3 + k], m.com[j][k], cy);
              }
            });
            mx = fma(m.mass[j], cx, mx);
            my = fma(m.mass[j], cy, my);
          }
        }
      });
      static_for<P::NF>([&](auto FF) {
        constexpr int f = decltype(FF)::value, l = P::frame_link(f);
        constexpr Pat9 u = PatOf<P, l>::after;
        double Rl[9];
        static_for<9>([&](auto EE) {
          constexpr int e = decltype(EE)::value;
          Rl[e] = pat_value<u.e[e]>(R[l][e]);
        });
        apply_xrot<P::frot(f)>(Rl, m.fX[f], fR[f]);
        double o[3] = {p[l].x, p[l].y, p[l].z};
        static_for<9>([&](auto EE) {
          constexpr int r = decltype(EE)::value % 3, k = decltype(EE)::value / 3;
          if constexpr ((P::ftmask(f) >> k) & 1) o[r] = pat_fma<u.e[3 * r + k]>(R[l][3 * r + k], m.fX[f][4 * k + 3], o[r]);
        });
        fp[f] = V3<double>{o[0], o[1], o[2]};
      });
    }
    double r2 = 0.0;
    const auto add = [&](double f) { r2 = fma(f, f, r2); };
    static_for<P::NC>([&](auto CC) {
      constexpr int c = decltype(CC)::value;
      constexpr int kind = P::ckind(c);
      constexpr int cm = c + CBase<P>::value;  // model slot
      if constexpr (kind == K_SPHERE) {
        double n2 = 0.0;
#pragma unroll
        for (int j = 0; j < P::D; ++j) {
          const double d = static_cast<double>(q[j]);
          n2 = fma(d, d, n2);
        }
        add(n2 * Ops::rsqrt_(n2) - m.ctgt[cm][0]);
      } else if constexpr (kind == K_AXIS) {
        constexpr int a = P::cfa(c);
        add(fR[a][2]);
        add(fR[a][5]);
      } else if constexpr (kind == K_POSE || kind == K_REL || kind == K_PBND) {
        constexpr int a = P::cfa(c);
        const double *Pi = m.cPinv[cm];
        double Pr[9], B[9];
        load_R(Pi, Pr);
        V3<double> x;  // the vector G maps to the error translation
        if constexpr (kind == K_REL) {  // G = P^-1_R R_a^T, R_err = G R_b, t = G (p_b - p_a) + P^-1_p
          constexpr int b = P::cfb(c);
          double G[9];
#pragma unroll
          for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int k = 0; k < 3; ++k)
              G[3 * r + k] = fma(Pr[3 * r], fR[a][3 * k], fma(Pr[3 * r + 1], fR[a][3 * k + 1], Pr[3 * r + 2] * fR[a][3 * k + 2]));
#pragma unroll
          for (int e = 0; e < 9; ++e) {
            Pr[e] = G[e];
            B[e] = fR[b][e];
          }
          x = sub(fp[b], fp[a]);
        } else {  // G = P^-1_R, R_err = G R_a Q^-1_R, t = G (p_a + R_a Q^-1_p) + P^-1_p
          if (m.cq_id[cm]) {
#pragma unroll
            for (int e = 0; e < 9; ++e) B[e] = fR[a][e];
            x = fp[a];
          } else {
            double Qr[9];
            load_R(m.cQinv[cm], Qr);
            mul33(fR[a], Qr, B);
            x = add_rot_t<7>(fp[a], fR[a], load_p(m.cQinv[cm]));
          }
        }
        const double t[3] = {fma(Pr[0], x.x, fma(Pr[1], x.y, fma(Pr[2], x.z, Pi[3]))),
                             fma(Pr[3], x.x, fma(Pr[4], x.y, fma(Pr[5], x.z, Pi[7]))),
                             fma(Pr[6], x.x, fma(Pr[7], x.y, fma(Pr[8], x.z, Pi[11])))};
        if constexpr (kind == K_PBND) {  // each component's distance outside [lo, hi]
          double E[9];
          mul33(Pr, B, E);
          const auto lg = so3_log<Ops, double>(E);
          const double v[6] = {t[0], t[1], t[2], lg.phi.x, lg.phi.y, lg.phi.z};
#pragma unroll
          for (int i = 0; i < 6; ++i) {
            const double lo = m.cB[cm][i], hi = m.cB[cm][6 + i];
            add(v[i] < lo ? v[i] - lo : (v[i] > hi ? v[i] - hi : 0.0));
          }
        } else {
#pragma unroll
          for (int i = 0; i < 3; ++i) add(t[i]);
          r2 += accept_angle2(Pr, B);
        }
      } else if constexpr (kind == K_PLANE || kind == K_LINE) {
        constexpr int a = P::cfa(c);
        const double *Pi = m.cPinv[cm];
        const V3<double> x = fp[a];
        if constexpr (kind == K_PLANE) {
          add(fma(Pi[8], x.x, fma(Pi[9], x.y, fma(Pi[10], x.z, Pi[11]))));
        } else {
          add(fma(Pi[0], x.x, fma(Pi[1], x.y, fma(Pi[2], x.z, Pi[3]))));
          add(fma(Pi[4], x.x, fma(Pi[5], x.y, fma(Pi[6], x.z, Pi[7]))));
        }
      } else if constexpr (kind == K_DIST) {
        constexpr int a = P::cfa(c), b = P::cfb(c);
        const V3<double> dv = sub(fp[b], fp[a]);
        const double n2 = fma(dv.x, dv.x, fma(dv.y, dv.y, dv.z * dv.z));
        add(n2 * Ops::rsqrt_(n2) - m.ctgt[cm][0]);
      } else if constexpr (kind == K_COM) {
        add(fma(mx, m.inv_mass, -m.ctgt[cm][0]));
        add(fma(my, m.inv_mass, -m.ctgt[cm][1]));
      } else if constexpr (kind == K_HULL) {
        const double cx = mx * m.inv_mass, cy = my * m.inv_mass;
        double px, py, nx, ny;
        polygon_nearest<double>(m.cB[cm], static_cast<int>(m.ctgt[cm][0]), cx, cy, px, py, nx, ny);
        add(cx - px);
        add(cy - py);
      }
    });
    return r2;
  }
}

}  // namespace mcp
