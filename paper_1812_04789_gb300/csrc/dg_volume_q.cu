// Volume term of the residual / exact JVP for the tensor-product space Q_p by
// sum factorisation (Sec. 3.1 eq. dg_ns, volume part; the paper's
// quadrilateral basis of Sec. 3).
//
// With phi_(a0,a1,a2)(xi) = L_a0(xi_0) L_a1(xi_1) L_a2(xi_2) and the tensor
// Gauss-Legendre points, the interpolation of u and of its d reference
// derivatives at all n_q = nq^d points is d successive one-dimensional
// contractions (the last one fused into the pointwise flux evaluation), and
// the projection  R_i -= sum_q w_q grad phi_i(q) . F(q)  is the transposed
// sequence: O((p+1) nq^d) work per contraction instead of O((p+1)^d nq^d).
// The total-degree space P_p is the subset a0 + a1 + a2 <= p of the same
// products: every sum and every array runs over that subset only (pairs (a0,
// a1) with a0 + a1 <= p, a0-major), with the slowest thread index the one that
// sets a sum's length, so that the lanes of a warp run sums of one length.
// Running the whole tensor with the other coefficients zero cost 1.7 times the
// FP64 operations in the JVP, whose FP64 pipe is the bound (two lanes per clock
// and SM): JVP, FP64, volume: 32^3 p = 6 46.0 -> 22 ms, 16^3 p = 4 1.74 -> 1.22 ms.
// Interpolation (3-D): Z_s[v][a0][a1][q2] = sum_a2 W[v][a0 a1 a2] L^s_a2(q2)
// (s = value or derivative factor), Y_t[v][a0][q1][q2] = sum_a1 Z L^t_a1(q1)
// for the three patterns (L, L), (L', L)... needed by u, d/dxi_1, d/dxi_2,
// then per point u, du/dxi_0 from Y with L_a0, L'_a0.  Projection: P_j =
// sum_q0, Q_A, Q_B = sum_q1, R = sum_q2 with the matching factors; the
// metric 2/h_k multiplies each derivative factor.  One CTA per element;
// JVP: dual numbers carried as separate value / tangent arrays.
#include <algorithm>
#include <type_traits>

#include "dg_internal.h"

namespace dgk {

namespace {

struct QPlan {
  int n1, nq, nt, nqd, npair;
  size_t oL, oT, oW, oZ, oY, oF, oP, total;   // element offsets in shared memory (T)
};

__host__ __device__ constexpr size_t zmax(size_t a, size_t b) { return a > b ? a : b; }

// 3-D: two regions, each holding in turn what is live at that stage:
//   A: Z (interpolation), then F (pointwise fluxes), then R (modes)
//   B: the coefficients W, then Y (interpolation), then P, Q (projection)
// 2-D: W, the stages (Y, then P) and F apart.
template <int D>
__host__ __device__ inline QPlan q_plan(int p, int nq, int M, bool total_degree, bool jvp) {
  QPlan P;
  P.n1 = p + 1;
  P.nq = nq;
  P.nt = 1;
  P.nqd = 1;
  for (int k = 0; k < D; ++k) {
    P.nt *= P.n1;
    P.nqd *= nq;
  }
  P.npair = total_degree ? P.n1 * (P.n1 + 1) / 2 : P.n1 * P.n1;
  const size_t nc = jvp ? 2 : 1;   // value (+ tangent) copies
  const size_t n1 = P.n1;
  size_t o = 0;
  P.oL = o;
  o += 2 * n1 * nq + nq;
  P.oT = o;                        // mode -> tensor index (unsigned short), pair -> a0, a1 (unsigned short)
  o += (2 * ((size_t)P.nt + n1 * n1) + 3) / 4;   // room in 4-byte elements at least
  if (D == 3) {
    const size_t nZ = 2 * M * P.npair * nq, nY = 3 * M * n1 * nq * nq;
    const size_t nP = M * n1 * nq * nq, nQ = M * P.npair * nq;
    const size_t A = zmax(nc * nZ, (size_t)D * M * P.nqd);
    const size_t B = zmax(zmax(nc * M * P.nt, nc * nY), 3 * nP + 2 * nQ);
    P.oZ = P.oF = o;
    o += A;
    P.oW = P.oY = P.oP = o;
    o += B;
  } else {
    P.oW = o;
    o += nc * M * P.nt;
    P.oY = P.oP = P.oZ = o;
    o += zmax(nc * 2 * M * n1 * nq, (size_t)2 * M * n1 * nq);
    P.oF = o;
    o += (size_t)D * M * P.nqd;
  }
  P.total = o;
  return P;
}

template <int D, class T, bool JVP>
__global__ void __launch_bounds__(256) volume_q_kernel(MeshView<T> mv, Phys<T> ph, const T* __restrict__ l1g,
                                                       const int* __restrict__ qidx, const T* __restrict__ W,
                                                       const T* __restrict__ V, const T* __restrict__ slots,
                                                       const T* __restrict__ Src, T sigma, T* __restrict__ out,
                                                       int* status, int p, int nq, int total_degree, T m0, T m1,
                                                       T m2) {
  using S = typename std::conditional<JVP, Dual<T>, T>::type;
  constexpr int M = D + 2, NC = JVP ? 2 : 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  const QPlan P = q_plan<D>(p, nq, M, total_degree, JVP);
  const int n1 = P.n1, nt = P.nt, nqd = P.nqd, nb = mv.nb, nm = mv.nm, E = mv.E, npair = P.npair;
  unsigned short* mtab = reinterpret_cast<unsigned short*>(sm + P.oT);   // [nm]
  unsigned short* ptab = mtab + nt;                                      // [npair]: a0 | a1 << 8
  auto pair0 = [&](int a0) { return total_degree ? a0 * n1 - a0 * (a0 - 1) / 2 : a0 * n1; };
  for (int t = threadIdx.x; t < nt; t += blockDim.x)
    if (qidx[t] >= 0) mtab[qidx[t]] = (unsigned short)t;
  for (int t = threadIdx.x; t < n1 * n1; t += blockDim.x) {
    const int a0 = t / n1, a1 = t - a0 * n1;
    if (!total_degree || a0 + a1 <= p) ptab[pair0(a0) + a1] = (unsigned short)(a0 | a1 << 8);
  }
  const T* L = sm + P.oL;            // L[a][q]
  const T* dL = L + n1 * nq;         // dL[a][q]
  const T* w1 = dL + n1 * nq;        // w[q]
  T* Wt = sm + P.oW;                 // [c][v][t], c = value, tangent
  T* F = sm + P.oF;                  // [k][v][q]: w_q |J| F (value or tangent)
  const T met[3] = {m0, m1, m2};
  for (int t = threadIdx.x; t < 2 * n1 * nq + nq; t += blockDim.x) sm[P.oL + t] = l1g[t];
  for (int e = blockIdx.x; e < E; e += gridDim.x) {
    __syncthreads();   // the tables (first element) or the modes' sums (later ones) are done
    for (int t = threadIdx.x; t < nb; t += blockDim.x) {
      const int v = t / nm, ti = mtab[t - v * nm];
      Wt[v * nt + ti] = W[(size_t)e * nb + t];
      if (JVP) Wt[M * nt + v * nt + ti] = V[(size_t)e * nb + t];
    }
    __syncthreads();
    // ---------------- interpolation
    if (D == 3) {
      const int nz = NC * 2 * M * nq, ny = NC * 3 * M * nq * nq;
      T* Z = sm + P.oZ;       // [c][s][v][pair][q2]
      T* Y = sm + P.oY;       // [c][t][v][a0][q1][q2] (over W: Z is complete)
      for (int t = threadIdx.x; t < nz * npair; t += blockDim.x) {
        const int pr = t / nz, r = t - pr * nz, csv = r / nq, q2 = r - csv * nq;
        const int v = csv % M, s = (csv / M) % 2, c = csv / (2 * M);
        const int a0 = ptab[pr] & 255, a1 = ptab[pr] >> 8, na = total_degree ? n1 - a0 - a1 : n1;
        const T* Ls = (s ? dL : L) + q2;
        const T* w = Wt + (size_t)c * M * nt + v * nt + a0 + n1 * a1;
        T acc = T(0);
        for (int a2 = 0; a2 < na; ++a2) acc += w[n1 * n1 * a2] * Ls[a2 * nq];
        Z[((size_t)csv * npair + pr) * nq + q2] = acc;
      }
      __syncthreads();
      for (int t = threadIdx.x; t < ny * n1; t += blockDim.x) {
        const int a0 = t / ny, r = t - a0 * ny, q12 = r % (nq * nq), ctv = r / (nq * nq);
        const int q2 = q12 % nq, q1 = q12 / nq, v = ctv % M, ts = (ctv / M) % 3, c = ctv / (3 * M);
        // ts 0: (L on a1, L on a2); 1: (L' on a1, L on a2); 2: (L on a1, L' on a2)
        const T* Lt = (ts == 1 ? dL : L) + q1;
        const T* z = Z + ((size_t)((c * 2 + (ts == 2 ? 1 : 0)) * M + v) * npair + pair0(a0)) * nq + q2;
        const int na = total_degree ? n1 - a0 : n1;
        T acc = T(0);
        for (int a1 = 0; a1 < na; ++a1) acc += z[a1 * nq] * Lt[a1 * nq];
        Y[((size_t)ctv * n1 + a0) * nq * nq + q12] = acc;
      }
    } else {
      const int nY = 2 * M * n1 * nq;
      T* Y = sm + P.oY;   // [c][s][v][a0][q1]
      for (int t = threadIdx.x; t < NC * nY; t += blockDim.x) {
        const int c = t / nY, r = t - c * nY;
        const int q1 = r % nq, a0 = (r / nq) % n1, v = (r / (nq * n1)) % M, s = r / (nq * n1 * M);
        const T* Ls = s ? dL : L;
        const T* w = Wt + (size_t)c * M * nt + v * nt + a0;
        const int na = total_degree ? n1 - a0 : n1;
        T acc = T(0);
        for (int a1 = 0; a1 < na; ++a1) acc += w[n1 * a1] * Ls[a1 * nq + q1];
        Y[t] = acc;
      }
    }
    __syncthreads();
    // ---------------- pointwise flux (the last contraction fused in)
    for (int q = threadIdx.x; q < nqd; q += blockDim.x) {
      const int q0 = q % nq, qr = q / nq;   // qr = q1 (2-D) or q1 + nq q2 (3-D)
      const int yq = D == 3 ? (qr % nq) * nq + qr / nq : qr;   // (q1, q2) in the Y layout, q2 fastest
      S u[M], g[M][D];
#pragma unroll
      for (int v = 0; v < M; ++v) {
        T uu[NC], gg[NC][D];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          uu[c] = T(0);
#pragma unroll
          for (int k = 0; k < D; ++k) gg[c][k] = T(0);
        }
        if (D == 3) {
          const int nY = 3 * M * n1 * nq * nq;
          const T* Y = sm + P.oY;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const T* y0 = Y + (size_t)c * nY + ((size_t)(0 * M + v) * n1) * nq * nq + yq;
            const T* y1 = Y + (size_t)c * nY + ((size_t)(1 * M + v) * n1) * nq * nq + yq;
            const T* y2 = Y + (size_t)c * nY + ((size_t)(2 * M + v) * n1) * nq * nq + yq;
            for (int a0 = 0; a0 < n1; ++a0) {
              const T la = L[a0 * nq + q0], da = dL[a0 * nq + q0];
              const T v0 = y0[a0 * nq * nq];
              uu[c] += v0 * la;
              gg[c][0] += v0 * da;
              gg[c][1] += y1[a0 * nq * nq] * la;
              gg[c][2 % D] += y2[a0 * nq * nq] * la;
            }
          }
        } else {
          const int nY = 2 * M * n1 * nq;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const T* y0 = sm + P.oY + (size_t)c * nY + ((size_t)(0 * M + v) * n1) * nq + yq;
            const T* y1 = sm + P.oY + (size_t)c * nY + ((size_t)(1 * M + v) * n1) * nq + yq;
            for (int a0 = 0; a0 < n1; ++a0) {
              const T la = L[a0 * nq + q0], da = dL[a0 * nq + q0];
              const T v0 = y0[a0 * nq];
              uu[c] += v0 * la;
              gg[c][0] += v0 * da;
              gg[c][1] += y1[a0 * nq] * la;
            }
          }
        }
        if constexpr (JVP) {
          u[v] = S(uu[0], uu[1]);
#pragma unroll
          for (int k = 0; k < D; ++k) g[v][k] = S(gg[0][k] * met[k], gg[1][k] * met[k]);
        } else {
          u[v] = uu[0];
#pragma unroll
          for (int k = 0; k < D; ++k) g[v][k] = gg[0][k] * met[k];
        }
      }
      if (!physical<D>(u, ph.gm1)) atomicOr(status, ST_NONPHYSICAL);
      S Fl[M][D];
      flux_total<D, S, T>(u, g, Fl, ph);
      T wq = mv.detJ * w1[q0];
      int r = qr;
#pragma unroll
      for (int k = 1; k < D; ++k) {
        wq *= w1[r % nq];
        r /= nq;
      }
#pragma unroll
      for (int v = 0; v < M; ++v)
#pragma unroll
        for (int k = 0; k < D; ++k) F[((size_t)k * M + v) * nqd + q] = wq * (JVP ? tan_part(Fl[v][k]) : val(Fl[v][k]));
    }
    __syncthreads();
    // ---------------- projection onto grad phi
    const T* Qm = nullptr;   // the last stage's input
    if (D == 3) {
      const int nP = M * n1 * nq * nq, nQ = M * npair * nq;
      T* Pb = sm + P.oP;      // [j][v][a0][q2][q1] times the metric (over Y: F is complete)
      T* Qb = Pb + 3 * nP;    // [A, B][v][pair][q2]
      for (int t = threadIdx.x; t < 3 * nP; t += blockDim.x) {
        const int j = t / nP, r = t - j * nP;
        const int q12 = r % (nq * nq), a0 = (r / (nq * nq)) % n1, v = r / (nq * nq * n1);
        const T* f = F + ((size_t)j * M + v) * nqd + (size_t)q12 * nq;
        const T* La = (j == 0 ? dL : L) + a0 * nq;
        T acc = T(0);
        for (int q0 = 0; q0 < nq; ++q0) acc += La[q0] * f[q0];
        Pb[t] = acc * (j == 0 ? met[0] : j == 1 ? met[1] : met[2 % D]);
      }
      __syncthreads();
      for (int t = threadIdx.x; t < 2 * nQ; t += blockDim.x) {
        const int j = t / nQ, r = t - j * nQ;
        const int q2 = r % nq, vp = r / nq, pr = vp % npair, v = vp / npair;
        const int a0 = ptab[pr] & 255, a1 = ptab[pr] >> 8;
        T acc = T(0);
        if (j == 0) {
          const T* p0 = Pb + (((size_t)0 * M + v) * n1 + a0) * nq * nq + (size_t)q2 * nq;
          const T* p1 = Pb + (((size_t)1 * M + v) * n1 + a0) * nq * nq + (size_t)q2 * nq;
          for (int q1 = 0; q1 < nq; ++q1) acc += L[a1 * nq + q1] * p0[q1] + dL[a1 * nq + q1] * p1[q1];
        } else {
          const T* p2 = Pb + (((size_t)2 * M + v) * n1 + a0) * nq * nq + (size_t)q2 * nq;
          for (int q1 = 0; q1 < nq; ++q1) acc += L[a1 * nq + q1] * p2[q1];
        }
        Qb[t] = acc;
      }
      Qm = Qb;
    } else {
      const int nP = M * n1 * nq;
      T* Pb = sm + P.oP;   // [j][v][a0][q1] times the metric
      for (int t = threadIdx.x; t < 2 * nP; t += blockDim.x) {
        const int j = t / nP, r = t - j * nP;
        const int q1 = r % nq, a0 = (r / nq) % n1, v = r / (nq * n1);
        const T* f = F + ((size_t)j * M + v) * nqd + (size_t)q1 * nq;
        const T* La = (j == 0 ? dL : L) + a0 * nq;
        T acc = T(0);
        for (int q0 = 0; q0 < nq; ++q0) acc += La[q0] * f[q0];
        Pb[t] = acc * (j == 0 ? met[0] : met[1]);
      }
      Qm = Pb;
    }
    __syncthreads();
    // ---------------- modes: the last contraction of the volume part + face
    // slots (fixed order) + sigma |J| v or - source
    for (int t = threadIdx.x; t < nb; t += blockDim.x) {
      const int v = t / nm, ti = mtab[t - v * nm], a0 = ti % n1, a1 = (ti / n1) % n1, a2 = ti / (n1 * n1);
      T acc = T(0);
      if (D == 3) {
        const T* qa = Qm + ((size_t)v * npair + pair0(a0) + a1) * nq;
        const T* qb = qa + (size_t)M * npair * nq;
        for (int q2 = 0; q2 < nq; ++q2) acc -= L[a2 * nq + q2] * qa[q2] + dL[a2 * nq + q2] * qb[q2];
      } else {
        const T* p0 = Qm + ((size_t)v * n1 + a0) * nq;
        const T* p1 = p0 + (size_t)M * n1 * nq;
        for (int q1 = 0; q1 < nq; ++q1) acc -= L[a1 * nq + q1] * p0[q1] + dL[a1 * nq + q1] * p1[q1];
      }
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const int em = mv.nbr[(e * D + k) * 2 + 0];
        acc += slots[(((size_t)e * D + k) * 2 + 0) * nb + t];
        acc += slots[(((size_t)em * D + k) * 2 + 1) * nb + t];
      }
      if (JVP) acc += sigma * mv.detJ * V[(size_t)e * nb + t];
      else if (Src) acc -= Src[(size_t)e * nb + t];
      out[(size_t)e * nb + t] = acc;
    }
  }
}

template <int D, class T, bool JVP>
cudaError_t run_q(const Mesh& Ms, const T* W, const T* V, const T* S, T sigma, T* out, cudaStream_t st) {
  const int pdeg = Ms.desc.space == DG_SPACE_Q ? 0 : 1;
  const QPlan P = q_plan<D>(Ms.p, Ms.nq1d, Ms.m, pdeg, JVP);
  const size_t smem = P.total * sizeof(T);
  int dev = 0, smax = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (smem > (size_t)smax) return cudaErrorNotSupported;
  cudaError_t e = allow_max_smem(volume_q_kernel<D, T, JVP>);
  if (e != cudaSuccess) return e;
  const T* l1 = std::is_same<T, double>::value ? (const T*)Ms.t64.l1d : (const T*)Ms.t32.l1d;
  const T* slots = std::is_same<T, double>::value ? (const T*)Ms.t64.slots : (const T*)Ms.t32.slots;
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, volume_q_kernel<D, T, JVP>, 256, smem);
  int nsm = 1;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int grid = std::min(Ms.E, std::max(1, occ) * nsm);
  const T m0 = (T)(2.0 / Ms.h[0]), m1 = (T)(2.0 / Ms.h[1]), m2 = (T)(D == 3 ? 2.0 / Ms.h[2] : 0.0);
  note_launch();
  volume_q_kernel<D, T, JVP><<<grid, 256, smem, st>>>(Ms.view<T>(), Ms.phys_t<T>(), l1, Ms.qidx, W, V, slots, S,
                                                      sigma, out, Ms.status, Ms.p, Ms.nq1d, pdeg, m0, m1, m2);
  return cudaGetLastError();
}

}  // namespace

template <class T>
cudaError_t launch_volume_q(const Mesh& M, const T* W, const T* V, const T* S, T sigma, bool jvp, T* out,
                            cudaStream_t st) {
  if (M.kind != DG_MESH_STRUCTURED || !M.qidx) return cudaErrorNotSupported;
  if (M.d == 2)
    return jvp ? run_q<2, T, true>(M, W, V, S, sigma, out, st) : run_q<2, T, false>(M, W, V, S, sigma, out, st);
  return jvp ? run_q<3, T, true>(M, W, V, S, sigma, out, st) : run_q<3, T, false>(M, W, V, S, sigma, out, st);
}
template cudaError_t launch_volume_q<double>(const Mesh&, const double*, const double*, const double*, double,
                                             bool, double*, cudaStream_t);
template cudaError_t launch_volume_q<float>(const Mesh&, const float*, const float*, const float*, float, bool,
                                            float*, cudaStream_t);

}  // namespace dgk
