// Two FP32 values per instruction: the same operation on the left and the
// right limb of a symmetric robot (x = left, y = right).  Every lane of a
// packed instruction is the IEEE operation with round-to-nearest, so a packed
// chain returns the bits of the two scalar chains; what it saves is issue and
// fetch (the FP32 throughput of the unit is the same).
#pragma once

#include "mcp_device.cuh"

namespace mcp {

// The packed instructions (sm_100 and later; the host-side checks of plans and
// constants compile this header for the toolkit's default architecture).
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ < 1000
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y)); }
#else
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
#endif
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 v) { return mul2(v, make_float2(-1.f, -1.f)); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, make_float2(-1.f, -1.f), a); }

// The sum of two products' pairs: as scalar additions, because the compiler
// contracts a packed addition of a packed product into a packed fma (which it
// does not do to __fmul_rn and __fadd_rn).
__device__ __forceinline__ float2 add2_apart(float2 a, float2 b) { return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y)); }

struct V3p {
  float2 x, y, z;
};
__device__ __forceinline__ V3p neg2(V3p v) { return V3p{neg2(v.x), neg2(v.y), neg2(v.z)}; }
// a x b, with na = -a
__device__ __forceinline__ V3p cross2(V3p a, V3p na, V3p b) {
  return V3p{fma2(a.y, b.z, mul2(na.z, b.y)), fma2(a.z, b.x, mul2(na.x, b.z)),
             fma2(a.x, b.y, mul2(na.y, b.x))};
}
__device__ __forceinline__ float2 row2(const float2 *R, V3p v) {
  return fma2(R[0], v.x, fma2(R[1], v.y, mul2(R[2], v.z)));
}
__device__ __forceinline__ V3p mulv2(const float2 (&R)[9], V3p v) { return V3p{row2(R, v), row2(R + 3, v), row2(R + 6, v)}; }
__device__ __forceinline__ void mul33_2(const float2 *A, const float2 *B, float2 (&C)[9]) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c)
      C[r * 3 + c] = fma2(A[r * 3], B[c], fma2(A[r * 3 + 1], B[3 + c], mul2(A[r * 3 + 2], B[6 + c])));
}

// sincos_f32 of both values, operation by operation
__device__ __forceinline__ void sincos2_f32(float2 x, float2 &s, float2 &c) {
  const float2 t = mul2(x, both(0.636619772367581343f));
  const float2 k = make_float2(rintf(t.x), rintf(t.y));
  float2 r = fma2(k, both(-1.5703125f), x);
  r = fma2(k, both(-4.837512969970703e-4f), r);
  r = fma2(k, both(-7.549790126404332e-8f), r);
  const float2 r2 = mul2(r, r);
  float2 ps = fma2(r2, both(2.75573192e-6f), both(-1.98412698e-4f));
  ps = fma2(r2, ps, both(8.33333333e-3f));
  ps = fma2(r2, ps, both(-1.66666667e-1f));
  const float2 sr = fma2(mul2(r, r2), ps, r);
  float2 pc = fma2(r2, both(-2.75573192e-7f), both(2.48015873e-5f));
  pc = fma2(r2, pc, both(-1.38888889e-3f));
  pc = fma2(r2, pc, both(4.16666667e-2f));
  pc = fma2(r2, pc, both(-0.5f));
  const float2 cr = fma2(r2, pc, both(1.0f));
  const auto quadrant = [](float kf, float sr1, float cr1, float &s1, float &c1) {
    const int qd = static_cast<int>(kf) & 3;
    const float ss = (qd & 1) ? cr1 : sr1, cc = (qd & 1) ? sr1 : cr1;
    s1 = (qd & 2) ? -ss : ss;
    c1 = ((qd + 1) & 2) ? -cc : cc;
  };
  quadrant(k.x, sr.x, cr.x, s.x, c.x);
  quadrant(k.y, sr.y, cr.y, s.y, c.y);
}

// What the Jacobian of two pose-like constraints (or of one, both lanes the
// same) needs from the residuals.
struct PosePair {
  V3p x, phi, nphi;  // reference point, log-map vector and its negative
  float2 beta;
};
// 6-row segments of two revolute joints with axes z and origins o
__device__ __forceinline__ void seg6_2(const float2 (&G)[9], const PosePair &e, V3p z, V3p o, float2 (&v)[6]) {
  const V3p d{sub2(e.x.x, o.x), sub2(e.x.y, o.y), sub2(e.x.z, o.z)};
  const V3p vt = mulv2(G, cross2(z, neg2(z), d));
  const V3p w = mulv2(G, z);
  const V3p a = cross2(e.phi, e.nphi, w), b = cross2(e.phi, e.nphi, a);
  const float2 h = both(-0.5f);
  v[0] = vt.x;
  v[1] = vt.y;
  v[2] = vt.z;
  v[3] = fma2(e.beta, b.x, fma2(h, a.x, w.x));
  v[4] = fma2(e.beta, b.y, fma2(h, a.y, w.y));
  v[5] = fma2(e.beta, b.z, fma2(h, a.z, w.z));
}

}  // namespace mcp
