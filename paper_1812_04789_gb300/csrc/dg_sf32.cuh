// Shared by the FP32 Jacobian-vector product kernels (dg_vol32.cu,
// dg_face32.cu) and the block probe (dg_probe_sf.cuh) of 3-D P_p meshes: the one-dimensional tables as a kernel parameter
// (after unrolling, operands straight from the constant bank: a multiply-add
// of a contraction costs no load for its table entry) and the layout of the
// cached primal traces.
#pragma once
#include "dg_internal.h"

namespace dgk {

// N1 = p + 1 values of a one-dimensional degree, N1 + 1 Gauss-Legendre points
template <class T, int N1>
struct SfTab {
  T L[N1][N1 + 1], dL[N1][N1 + 1];   // values and reference derivatives
  T w[N1 + 1];                       // weights
  T Le[N1], dLe[N1];                 // end values at +1; at -1: (-1)^a Le, -(-1)^a dLe
  T met[3], detJ, faceJ[3];          // 2 / h_k, |J|, |J_F|
};
template <int N1>
using Sf32Tab = SfTab<float, N1>;

template <class T, int N1>
inline SfTab<T, N1> sf_tab(const Mesh& M) {
  constexpr int NQ = N1 + 1;
  SfTab<T, N1> t;
  const std::vector<double>& l = M.h_l1d;   // L[a][q], dL[a][q], w[q], Le(-1)[a], Le(+1)[a], dLe(-1)[a], dLe(+1)[a]
  for (int a = 0; a < N1; ++a) {
    for (int q = 0; q < NQ; ++q) {
      t.L[a][q] = (T)l[(size_t)a * NQ + q];
      t.dL[a][q] = (T)l[(size_t)(N1 + a) * NQ + q];
    }
    t.Le[a] = (T)l[(size_t)2 * N1 * NQ + NQ + N1 + a];
    t.dLe[a] = (T)l[(size_t)2 * N1 * NQ + NQ + 3 * N1 + a];
  }
  for (int q = 0; q < NQ; ++q) t.w[q] = (T)l[(size_t)2 * N1 * NQ + q];
  for (int k = 0; k < 3; ++k) {
    t.met[k] = (T)(2.0 / M.h[k]);
    t.faceJ[k] = (T)M.faceJ[k];
  }
  t.detJ = (T)M.detJ;
  return t;
}

// dimension of P_p in 3-D, and its (a0, a1) pairs, a0-major
__host__ __device__ constexpr int sf32_modes(int n1) { return n1 * (n1 + 1) * (n1 + 2) / 6; }
__host__ __device__ constexpr int sf32_pairs(int n1) { return n1 * (n1 + 1) / 2; }
__host__ __device__ constexpr int sf32_pair0(int n1, int a0) { return a0 * n1 - a0 * (a0 - 1) / 2; }

// Where the sums over the degree a_k of one direction k run, the modes are kept
// pair by pair ((a0, a1) the degrees of the two other directions, t0 < t1), a_k
// contiguous: first position of a pair, and of a mode given its tensor index.
__host__ __device__ constexpr int sf32_run(int n1, int a0, int a1) {
  return sf32_modes(n1) - sf32_modes(n1 - a0) + sf32_pairs(n1 - a0) - sf32_pairs(n1 - a0 - a1);
}
template <int N1>
__device__ __forceinline__ int sf32_pos(int t, int k) {
  const int x0 = t % N1, x1 = t / N1 % N1, x2 = t / (N1 * N1);
  const int ak = k == 0 ? x0 : k == 1 ? x1 : x2, a0 = k == 0 ? x1 : x0, a1 = k == 2 ? x1 : x2;
  return sf32_run(N1, a0, a1) + ak;
}

// Cached primal traces (u, grad u: 20 values in five 16-byte words), laid out
// so that the kernels' loads are coalesced over a line's or a face's points:
//   volume [e][q0][word][q2 + nq q1]: u[0..4], then d_k u[v] at 5 + 3 v + k
//   faces  [f][side][word][b1 + nq b0]: the same in the face's frame
//          (directions n, t0, t1; variables rho, momenta along n, t0, t1, rho e0)
__host__ __device__ inline size_t sf32_vol_word(long e, int q0, int w, int line, int nq) {
  return (((size_t)e * nq + q0) * 5 + w) * nq * nq + line;
}
__host__ __device__ inline size_t sf32_face_word(long f, int side, int w, int q, int nqf) {
  return (((size_t)f * 2 + side) * 5 + w) * nqf + q;
}

}  // namespace dgk
