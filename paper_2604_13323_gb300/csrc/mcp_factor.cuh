// What the humanoid's projection kernel (mcp_tree.cuh) takes from the structure
// of its class: the zero pattern of the Cholesky factor and the constants of the
// floating base's prismatic chain.
#pragma once

#include "mcp_device.cuh"
#include "mcp_problems.cuh"

namespace mcp {

constexpr int PRE_JOINTS = 3;  // prismatic root joints placed in closed form

// Structural nonzeros of the Cholesky factor of A = J J^T + lambda I, row by
// row (bit b of row i: L[i][b] may be nonzero).  The symbolic factorisation:
// L[i][b] is nonzero where A[i][b] is (rows i and b of J share a joint) or
// where L[i][j] and L[b][j] are both nonzero for some column j < b.
template <class P>
__host__ __device__ constexpr uint32_t l_row_pattern(int row) {
  constexpr int K = kdim<P>();
  uint64_t jm[MAXK] = {};  // joints of row i of J
  for (int i = 0; i < K; ++i)
    for (int j = 0; j < P::D; ++j)
      if (jnz<P>(i, j)) jm[i] |= uint64_t(1) << j;
  uint32_t nz[MAXK] = {};
  for (int i = 0; i < K; ++i)
    for (int b = 0; b <= i; ++b) {
      bool v = (b == i) || (jm[i] & jm[b]) != 0;
      for (int j = 0; j < b && !v; ++j) v = ((nz[i] >> j) & 1u) != 0 && ((nz[b] >> j) & 1u) != 0;
      if (v) nz[i] |= 1u << b;
    }
  return nz[row];
}
template <class P, int I>
struct LRow {
  static constexpr uint32_t value = l_row_pattern<P>(I);
};
// The prismatic root chain in closed form (its first PRE_JOINTS joints): with
// q = 0 joint i's frame sits at c[i] with rotation R[i]; its axis is a[i] = R[i]
// e_z, so its origin is c[i] + sum_{k <= i} q_k a[k]; mc[i] = m_i R_i com_i.
struct PreChain {
  float R[PRE_JOINTS][9];
  float a[PRE_JOINTS][3];
  float c[PRE_JOINTS][3];
  float mc[PRE_JOINTS][3];
};
template <class P>
PreChain make_pre_chain(const ModelT<double> &m64) {  // in FP64, then rounded
  PreChain t{};
  double R[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1}, c[3] = {0, 0, 0};
  for (int i = 0; i < PRE_JOINTS && i < P::D && P::jtype(i) == PRIS && P::parent(i) == i - 1; ++i) {
    const double *X = m64.X[i];
    double Rn[9], cn[3];
    for (int r = 0; r < 3; ++r) {
      cn[r] = c[r] + R[r * 3] * X[3] + R[r * 3 + 1] * X[7] + R[r * 3 + 2] * X[11];
      for (int cc = 0; cc < 3; ++cc)
        Rn[r * 3 + cc] = R[r * 3] * X[cc] + R[r * 3 + 1] * X[4 + cc] + R[r * 3 + 2] * X[8 + cc];
    }
    for (int e = 0; e < 9; ++e) R[e] = Rn[e];
    for (int r = 0; r < 3; ++r) c[r] = cn[r];
    for (int e = 0; e < 9; ++e) t.R[i][e] = static_cast<float>(R[e]);
    for (int r = 0; r < 3; ++r) {
      t.a[i][r] = static_cast<float>(R[r * 3 + 2]);
      t.c[i][r] = static_cast<float>(c[r]);
      t.mc[i][r] = static_cast<float>(m64.mass[i] * (R[r * 3] * m64.com[i][0] + R[r * 3 + 1] * m64.com[i][1] +
                                                     R[r * 3 + 2] * m64.com[i][2]));
    }
  }
  return t;
}

}  // namespace mcp
