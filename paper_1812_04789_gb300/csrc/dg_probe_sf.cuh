// Diagonal element blocks of 3-D P_p meshes (Sec. 5.1 eq. ODEDG; Sec. 6.3) by
// sum factorisation, in FP32 and FP64 (dg_probe_sf32.cu, dg_probe_sf64.cu).
//
//   D[(v,i'),(w,i)] = sum_p sum_c sum_s Test_c(p,i') J_p[(v,c),(w,s)] Trial_s(p,i)
// over the element's volume points and the points of its faces.  Test and
// trial functions are products of one-dimensional ones, so for every pair (v,
// w) the sum over the points of a line, of a plane and of the element is done
// one direction at a time on the pairs of degrees (a', a):
//   volume  X[a0' a0][q1 q2] = sum_q0, Y[a0'a1' a0a1][q2] = sum_q1, D = sum_q2,
//           where after the first direction the twelve (c, s) have merged into
//           nine kinds (value / derivative in the two others) and after the second
//           into four;
//   faces   three matrices on the tangential pairs, A = value x value (the flux,
//           the lifting, scaled per test pair as in dg_face_sf.cu, the tangential
//           gradients and the tangential dual terms), B = value x normal
//           derivative, C = normal derivative x value, each again direction by
//           direction; the normal direction's end values then spread them
//           over the modes: D += Le' Le A + Le' Le,n B + Le,n' Le C.
// Multiply-adds per element at p = 4: 9 M instead of 53 M for the dense sums,
// at p = 6 50 M instead of 630 M, which outweighs the tensor cores' rate for
// the dense form (probe_tc_kernel, whose operand production was the limit)
// and the FP64 pipe's for probe64_kernel.  A thread takes one test degree (or
// pair) and a row of trial degrees: with a whole degree pair block per thread
// and its total-degree guards inside the loops, or with kinds mixed in a warp,
// the p = 6 kernel took 172 ms.  FP32 is bound by instruction issue (61 % of
// the slots, 30 % of the issued ones multiply-adds, the rest shared-memory
// operands and indices), FP64 by its pipe.  J_p: one dual-number evaluation per
// value seed; a seed of a gradient component enters the viscous flux alone and
// is evaluated directly.
// FP32 (against probe_tc_kernel): 16^3, p = 1: 1.43 -> 0.51 ms; p = 2: 2.5 -> 0.96; p = 4:
// 11.7 -> 5.5; p = 5: 36 -> 12.7; p = 6: 99 -> 24.  FP64 (against probe64_kernel):
// 12^3, p = 4: 198 -> 42 ms.
#pragma once
#include "dg_sf32.cuh"

namespace dgk {

// VG: output variables whose volume Jacobians are held at once (they are formed
// again for the next group); VP: of these, contracted at once (VG or 1); CQ:
// planes q2 contracted at once.  Chosen per type and order for the shared
// memory (two CTAs per SM where that fits).
template <class T, int N1, int VG, int VP, int CQ, bool CACHED>
struct Psf {
  static constexpr int NQ = N1 + 1, NL = NQ * NQ, NV = NL * NQ, NP = sf32_pairs(N1), NM = sf32_modes(N1), M = 5,
                       NB = M * NM, N2 = N1 * N1;
  static constexpr int PAD = CACHED || N1 < 7, XQ = PAD ? NQ | 1 : NQ, YP = PAD ? NP | 1 : NP;   // row strides without bank conflicts
  static constexpr int NT = sizeof(T) == 4 && N1 > 5 ? 512 : 256;    // FP64: registers for the dual numbers
  // volume: [J | X | Y | Dacc | U]; faces: [Jf | F1 | A | traces] over the same space
  static constexpr int nJ = VG * 12 * NV, nX = VP * 9 * N2 * XQ * CQ, nY = VP * 4 * CQ * NP * YP, nD = VP * NM * NM;
  static constexpr int nJf = 6 * M * 8 * NL, nF1 = 6 * 6 * N2 * XQ, nA = 6 * 3 * NP * YP;
  static constexpr int nU = CACHED ? 0 : NV * 20, nP = CACHED ? 0 : 6 * NL * 40;   // traces of the state
  static constexpr size_t nS = sizeof(unsigned short) * (2 * NP + NM + 3 * NM + 4);
  static constexpr bool FT = sizeof(T) * (nJf + nF1 + nA + nP + 7 * NB + 2 * N1 + 2 * N1 * NQ) + nS <= 227 * 1024;   // face traces kept
  static constexpr int vol = nJ + nX + nY + nD + nU, fac = nJf + nF1 + nA + (FT ? nP : 0);
  static constexpr int oW = vol > fac ? vol : fac;                       // W of the element and its neighbours
  static constexpr int oE = oW + (CACHED ? 0 : 7 * NB);                  // end values Le, dLe
  static constexpr int oL = oE + 2 * N1;                                 // L[a][q], dL[a][q]
  static constexpr int total = oL + 2 * N1 * NQ;
  static constexpr size_t bytes = sizeof(T) * total + nS;
};

// acc[a] += sum_q x[q] r[a][q], r the trial values or derivatives.  An item of a
// contraction is one test degree and a row of trial degrees: few registers, many
// items, table entries of the trial side from the constant bank.  A product of
// total-degree pairs uses a < n alone: FP64 leaves the others out (its pipe is the
// limit; n is the same for most of a warp), FP32 computes and drops them.
template <class T, int N1, int NC, bool RD>
__device__ __forceinline__ void psf_row(const SfTab<T, N1>& tb, const T* x, T* acc, int n) {
#pragma unroll
  for (int b = 0; b < NC; ++b)
    if (sizeof(T) == 4 || b < n)
#pragma unroll
      for (int q = 0; q < N1 + 1; ++q) acc[b] += x[q] * (RD ? tb.dL[b][q] : tb.L[b][q]);
}
// x[q] = t[q] y[q S] (ADD: +=)
template <class T, int NQ, int S, bool ADD>
__device__ __forceinline__ void psf_scale(const T* t, const T* y, T* x) {
#pragma unroll
  for (int q = 0; q < NQ; ++q) x[q] = ADD ? x[q] + t[q] * y[q * S] : t[q] * y[q * S];
}

// The state at point q of face f in the face's frame (directions n, t0, t1;
// momenta likewise); sd 0: from the L element's +1 face, sd 1: from R's -1 face.
// sW: the modes of the element, then of its neighbours.
template <class T, int N1>
__device__ __forceinline__ void psf_face_trace(const MeshView<T>& mv, const T* sW, int f, int sd, int q, T* c) {
  constexpr int NQ = N1 + 1, NL = NQ * NQ, NM = sf32_modes(N1), M = 5;
  const int k = f >> 1, t0 = k == 0 ? 1 : 0, t1 = k == 2 ? 1 : 2, qs = q / NQ + NQ * (q % NQ), lf = sd == 0 ? 2 * k + 1 : 2 * k;
  const T* ws = sW + ((sd == 0) == ((f & 1) == 1) ? 0 : 1 + f) * M * NM;
#pragma unroll
  for (int j = 0; j < 20; ++j) c[j] = T(0);
  for (int i = 0; i < NM; ++i) {
    const T p = mv.fphiT[((size_t)lf * NM + i) * NL + qs];
    const T dn = mv.fdphiT[(((size_t)lf * 3 + k) * NM + i) * NL + qs];
    const T d0 = mv.fdphiT[(((size_t)lf * 3 + t0) * NM + i) * NL + qs];
    const T d1 = mv.fdphiT[(((size_t)lf * 3 + t1) * NM + i) * NL + qs];
#pragma unroll
    for (int v = 0; v < M; ++v) {
      const int pv = v == 0 || v == M - 1 ? v : v == 1 ? 1 + k : v == 2 ? 1 + t0 : 1 + t1;
      const T a = ws[pv * NM + i];
      c[v] += a * p;
      c[5 + 3 * v] += a * dn;
      c[6 + 3 * v] += a * d0;
      c[7 + 3 * v] += a * d1;
    }
  }
}

// Derivatives of the outputs of one face point with respect to seed s (0 the
// value, 1 + j the gradient component j of the face's frame) of variable w of
// this element's state (OWN) or the neighbour's, weighted: o[(v 8 + kind) NL],
// v in the face's frame, kinds 0 flux, 1 lifting (s = 0), 2 3 4 flux (s = 1, 2,
// 3), 5 6 7 the own dual tensor's rows n, t0, t1 (s = 0).  side 1: this
// element's +1 face.
template <class T, int N1, bool OWN>
__device__ __forceinline__ void psf_face_jac(const SfTab<T, N1>& tb, const Phys<T>& ph, const T (*c)[20], int k, int side,
                                             int q, int s, int w, T* o) {
  using S = Dual<T>;
  constexpr int NQ = N1 + 1, NL = NQ * NQ, M = 5;
  const int b0 = q / NQ, b1 = q - b0 * NQ, t0 = k == 0 ? 1 : 0;
  const int wf = w == 0 || w == M - 1 ? w : w == 1 + k ? 1 : w == 1 + t0 ? 2 : 3;   // w in the face's frame
  const T mkk = k == 0 ? tb.met[0] : k == 1 ? tb.met[1] : tb.met[2];
  const T mt0 = k == 0 ? tb.met[1] : tb.met[0], mt1 = k == 2 ? tb.met[1] : tb.met[2];
  T wb0 = T(0), wb1 = T(0);
#pragma unroll
  for (int b = 0; b < NQ; ++b) {
    if (b0 == b) wb0 = tb.w[b];
    if (b1 == b) wb1 = tb.w[b];
  }
  const T fw = (k == 0 ? tb.faceJ[0] : k == 1 ? tb.faceJ[1] : tb.faceJ[2]) * wb0 * wb1;
  const T sg = side ? fw : -fw;
  if (s == 0) {
    S u[2][M], g[2][M][3];
#pragma unroll
    for (int sd = 0; sd < 2; ++sd)
#pragma unroll
      for (int v = 0; v < M; ++v) {
        u[sd][v] = S(c[sd][v], (((sd == 0) == (side == 1)) == OWN && v == wf) ? T(1) : T(0));
#pragma unroll
        for (int j = 0; j < 3; ++j) g[sd][v][j] = S(c[sd][5 + 3 * v + j], T(0));
      }
    S fp[M], mL[3], eL[3], mR[3], eR[3];
    face_point_core<3, 0, S, T>(u[0], g[0], u[1], g[1], ph, fp, mL, eL, mR, eR);
    const T lf = sg * ph.eta * mkk * T(0.125);
    T m[3], en[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      m[j] = side ? mL[j].d : mR[j].d;
      en[j] = side ? eL[j].d : eR[j].d;
    }
#pragma unroll
    for (int v = 0; v < M; ++v) {
      const int j = v == 0 || v == M - 1 ? 0 : v - 1;
      o[(v * 8 + 0) * NL] = sg * fp[v].d;
      // normal column of K(uL) jump + K(uR) jump (twice the halves)
      o[(v * 8 + 1) * NL] = v == 0 ? T(0)
                          : v == M - 1 ? lf * T(2) * (eL[0].d + eR[0].d)
                                       : lf * (v == 1 ? T(8) / T(3) : T(2)) * (mL[j].d + mR[j].d);
      // the own dual tensor (visc_rank1): rows n, t0, t1, E
      const T dn = v == 0 ? T(0) : v == 1 ? (T(4) / T(3)) * m[0] : v == 2 ? m[1] : v == 3 ? m[2] : en[0];
      const T d0 = v == 1 ? m[1] : v == 2 ? (T(-2) / T(3)) * m[0] : v == 4 ? en[1] : T(0);
      const T d1 = v == 1 ? m[2] : v == 3 ? (T(-2) / T(3)) * m[0] : v == 4 ? en[2] : T(0);
      o[(v * 8 + 5) * NL] = -fw * mkk * dn;
      o[(v * 8 + 6) * NL] = -fw * mt0 * d0;
      o[(v * 8 + 7) * NL] = -fw * mt1 * d1;
    }
  } else {
    T u[M], g[M][3], F[M];
#pragma unroll
    for (int v = 0; v < M; ++v) {
      u[v] = (side == 1) == OWN ? c[0][v] : c[1][v];
      F[v] = T(0);
#pragma unroll
      for (int j = 0; j < 3; ++j) g[v][j] = (v == wf && j == s - 1) ? T(1) : T(0);
    }
    Prim<3, T> pr;
    primitives<3, T, T>(u, ph, pr);
    add_visc_col<3, 0, T, T>(pr, g, T(0.5), F, ph);
    const T sc = sg * (s == 1 ? mkk : s == 2 ? mt0 : mt1);
#pragma unroll
    for (int v = 0; v < M; ++v) o[(v * 8 + 1 + s) * NL] = sc * F[v];
  }
}

template <class T, int N1, int VG, int VP, int CQ, bool CACHED>
__global__ void __launch_bounds__(Psf<T, N1, VG, VP, CQ, CACHED>::NT, sizeof(T) == 4 && N1 <= 5 ? 2 : 1)
    probe_sf_kernel(const __grid_constant__ SfTab<T, N1> tb, MeshView<T> mv, Phys<T> ph, const int* __restrict__ qidx,
                    const T* __restrict__ W, T sigma, T* __restrict__ Dout, size_t dstride, int* status,
                    const float4* __restrict__ Pv, const float4* __restrict__ Pf) {
  using C = Psf<T, N1, VG, VP, CQ, CACHED>;
  using S = Dual<T>;
  constexpr int NQ = C::NQ, NL = C::NL, NV = C::NV, NP = C::NP, NM = C::NM, M = C::M, NB = C::NB, N2 = C::N2,
                XQ = C::XQ, YP = C::YP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  T* J = sm;                       // [v][c * 4 + s][q0][q1 + NQ q2]
  T* X = J + C::nJ;                // [v][kind][a0' a0][q1 + XQ (q2 - z0)]
  T* Y = X + C::nX;                // [v][kind][q2 - z0][pair' pair]
  T* Da = Y + C::nY;               // [v][position'][position]
  T* Jf = sm;                      // [face][v][8][b1 + NQ b0]
  T* F1 = Jf + C::nJf;             // [face][6][a0' a0][b1]
  T* A = F1 + C::nF1;              // [face][3][pair' pair]
  T* U = Da + C::nD;               // [20][NV]
  T* P = A + C::nA;                // [face][side][20][NL]
  T* sW = sm + C::oW;              // [element, neighbours][NB]
  T* Le = sm + C::oE;              // values at +1, then derivatives
  T *sL = sm + C::oL, *sdL = sL + N1 * NQ;
  unsigned short* ptab = reinterpret_cast<unsigned short*>(sm + C::total);   // pair -> a0 | a1 << 8
  unsigned short* poff = ptab + NP;                                          // pair -> first position
  unsigned short* pmode = poff + NP;                                         // position (direction 2) -> mode
  unsigned short* mk = pmode + NM;                                           // [k][mode]: pair | a_k << 8
  const int tid = threadIdx.x, E = mv.E;
  for (int t = tid; t < N2; t += C::NT) {
    const int a0 = t / N1, a1 = t - a0 * N1;
    if (a0 + a1 < N1) {
      ptab[sf32_pair0(N1, a0) + a1] = (unsigned short)(a0 | a1 << 8);
      poff[sf32_pair0(N1, a0) + a1] = (unsigned short)sf32_run(N1, a0, a1);
    }
  }
  for (int t = tid; t < N1 * N2; t += C::NT) {
    const int i = qidx[t];
    if (i >= 0) {
      const int x0 = t % N1, x1 = t / N1 % N1, x2 = t / N2;
      pmode[sf32_pos<N1>(t, 2)] = (unsigned short)i;
      mk[i] = (unsigned short)((sf32_pair0(N1, x1) + x2) | x0 << 8);
      mk[NM + i] = (unsigned short)((sf32_pair0(N1, x0) + x2) | x1 << 8);
      mk[2 * NM + i] = (unsigned short)((sf32_pair0(N1, x0) + x1) | x2 << 8);
    }
  }
  for (int t = tid; t < 2 * N1; t += C::NT) Le[t] = t < N1 ? tb.Le[t] : tb.dLe[t - N1];
  for (int t = tid; t < N1 * NQ; t += C::NT) {
    sL[t] = tb.L[t / NQ][t % NQ];
    sdL[t] = tb.dL[t / NQ][t % NQ];
  }

  for (int e = blockIdx.x; e < E; e += gridDim.x) {
    T* De = Dout + (size_t)e * dstride;
    __syncthreads();
    if constexpr (!CACHED) {
      for (int t = tid; t < 7 * NB; t += C::NT) {
        const int who = t / NB, j = t - who * NB, el = who == 0 ? e : mv.nbr[e * 6 + who - 1];
        sW[t] = W[(size_t)el * NB + j];
      }
      __syncthreads();
      for (int t = tid; t < NV; t += C::NT) {      // volume traces of the state
        const int q0 = t / NL, l = t - q0 * NL, q = q0 + NQ * l;
        T c[20];
#pragma unroll
        for (int j = 0; j < 20; ++j) c[j] = T(0);
        for (int i = 0; i < NM; ++i) {
          const T p = mv.vphiT[(size_t)i * NV + q], d0 = mv.vdphiT[(size_t)i * NV + q],
                  d1 = mv.vdphiT[((size_t)NM + i) * NV + q], d2 = mv.vdphiT[((size_t)2 * NM + i) * NV + q];
#pragma unroll
          for (int v = 0; v < M; ++v) {
            const T a = sW[v * NM + i];
            c[v] += a * p;
            c[5 + 3 * v] += a * d0;
            c[6 + 3 * v] += a * d1;
            c[7 + 3 * v] += a * d2;
          }
        }
        if (!physical<3>(c, ph.gm1)) atomicOr(status, ST_NONPHYSICAL);
#pragma unroll
        for (int j = 0; j < 20; ++j) U[j * NV + t] = c[j];
      }
      __syncthreads();
    }
    for (int w = 0; w < M; ++w) {
      // ================= volume
      for (int v0 = 0; v0 < M; v0 += VG) {
        const int ng = min(VG, M - v0);
        // J (the seed slowest): seed 0 the value of variable w, 1 + k its derivative d_k
        for (int t = tid; t < 4 * NV; t += C::NT) {
          const int s = t / NV, pt = t - s * NV, q0 = pt / NL, l = pt - q0 * NL, q1 = l % NQ, q2 = l / NQ;
          T c[20];
          if constexpr (CACHED) {
#pragma unroll
            for (int j = 0; j < 5; ++j) {      // the cache's line index is q2 + NQ q1
              const float4 x = __ldg(Pv + sf32_vol_word(e, q0, j, q2 + NQ * q1, NQ));
              c[4 * j] = (T)x.x, c[4 * j + 1] = (T)x.y, c[4 * j + 2] = (T)x.z, c[4 * j + 3] = (T)x.w;
            }
            if (s == 0 && w == 0 && v0 == 0 && !physical<3>(c, ph.gm1)) atomicOr(status, ST_NONPHYSICAL);
          } else {
#pragma unroll
            for (int j = 0; j < 20; ++j) c[j] = U[j * NV + pt];
          }
          T wq = T(0);
          {
            T x0 = T(0), x1 = T(0), x2 = T(0);
#pragma unroll
            for (int b = 0; b < NQ; ++b) {
              if (q0 == b) x0 = tb.w[b];
              if (q1 == b) x1 = tb.w[b];
              if (q2 == b) x2 = tb.w[b];
            }
            wq = -tb.detJ * x0 * x1 * x2;
          }
          T F[M][3];
          if (s == 0) {
            S u[M], g[M][3], Fd[M][3];
#pragma unroll
            for (int v = 0; v < M; ++v) {
              u[v] = S(c[v], v == w ? T(1) : T(0));
#pragma unroll
              for (int k = 0; k < 3; ++k) g[v][k] = S(c[5 + 3 * v + k], T(0));
            }
            flux_total<3, S, T>(u, g, Fd, ph);
#pragma unroll
            for (int v = 0; v < M; ++v)
#pragma unroll
              for (int k = 0; k < 3; ++k) F[v][k] = Fd[v][k].d;
          } else {
            T g[M][3];
#pragma unroll
            for (int v = 0; v < M; ++v)
#pragma unroll
              for (int k = 0; k < 3; ++k) g[v][k] = (v == w && k == s - 1) ? T(1) : T(0);
            Prim<3, T> pr;
            primitives<3, T, T>(c, ph, pr);
            T col[3][M];
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
              for (int v = 0; v < M; ++v) col[k][v] = T(0);
            add_visc_col<3, 0, T, T>(pr, g, T(1), col[0], ph);
            add_visc_col<3, 1, T, T>(pr, g, T(1), col[1], ph);
            add_visc_col<3, 2, T, T>(pr, g, T(1), col[2], ph);
#pragma unroll
            for (int v = 0; v < M; ++v)
#pragma unroll
              for (int k = 0; k < 3; ++k) F[v][k] = col[k][v];
            wq *= s == 1 ? tb.met[0] : s == 2 ? tb.met[1] : tb.met[2];
          }
#pragma unroll
          for (int v = 0; v < M; ++v)
            if (v >= v0 && v < v0 + ng)
#pragma unroll
              for (int k = 0; k < 3; ++k) J[((v - v0) * 12 + k * 4 + s) * NV + pt] = wq * tb.met[k] * F[v][k];
        }
        __syncthreads();
        for (int vb = 0; vb < ng; vb += VP) {
          const int np = min(VP, ng - vb);
          for (int z0 = 0; z0 < NQ; z0 += CQ) {
            const int nz = min(CQ, NQ - z0);
            // X: kinds 3 c + sg, sg = (s = 0, 1), (2), (3); the derivative in direction 0 is
            // test's for c = 0 and trial's for s = 1
            for (int t = tid; t < np * 9 * N1 * NQ * CQ; t += C::NT) {
              const int ra = t / (NQ * CQ), l = t - ra * (NQ * CQ), r = ra / N1, at = ra - r * N1, vp = r / 9, kd = r - vp * 9,
                        c = kd / 3, sg = kd - 3 * c;
              if (l >= NQ * nz) continue;
              const T* j = J + ((vb + vp) * 12 + c * 4 + (sg == 0 ? 0 : sg + 1)) * NV + z0 * NQ + l;
              const T* tt = (c == 0 ? sdL : sL) + at * NQ;
              T x[NQ], acc[N1];
#pragma unroll
              for (int b = 0; b < N1; ++b) acc[b] = T(0);
              psf_scale<T, NQ, NL, false>(tt, j, x);
              psf_row<T, N1, N1, false>(tb, x, acc, N1);
              if (sg == 0) {
                psf_scale<T, NQ, NL, false>(tt, j + NV, x);
                psf_row<T, N1, N1, true>(tb, x, acc, N1);
              }
              T* o = X + ((size_t)r * N2 + at * N1) * XQ * CQ + l / NQ * XQ + l % NQ;
#pragma unroll
              for (int b = 0; b < N1; ++b) o[b * XQ * CQ] = acc[b];
            }
            __syncthreads();
            // Y: kinds (test, trial) in direction 2: 0 value-value, 1 derivative-value, 2
            // value-derivative, 3 derivative-derivative (the kind slowest, then a0: warps of one
            // kind); an item is a test pair, a0 and a plane: its sums over q1 for all a1
            for (int t = tid; t < np * 4 * N1 * NP * CQ; t += C::NT) {
              const int ka = t / (NP * CQ), r = t - ka * (NP * CQ), kv = ka / N1, ar = ka - kv * N1, kd = kv & 3, vp = kv >> 2;
              const int pt = r / CQ, z = r - pt * CQ, at = ptab[pt] & 255, a1t = ptab[pt] >> 8, nr = N1 - ar;
              if (z >= nz) continue;
              constexpr int XS = N2 * XQ * CQ;       // from one X kind to the next
              const T* xb = X + (size_t)vp * 9 * XS + (at * N1 + ar) * XQ * CQ + z * XQ;
              const T *l = sL + a1t * NQ, *dl = sdL + a1t * NQ;
              T x[NQ], acc[N1];
#pragma unroll
              for (int b = 0; b < N1; ++b) acc[b] = T(0);
              if (kd == 0) {          // derivatives in direction 1: X kinds 3 (test), 1 (trial), 4 (both)
                psf_scale<T, NQ, 1, false>(l, xb, x);
                psf_scale<T, NQ, 1, true>(dl, xb + 3 * XS, x);
                psf_row<T, N1, N1, false>(tb, x, acc, nr);
                psf_scale<T, NQ, 1, false>(l, xb + XS, x);
                psf_scale<T, NQ, 1, true>(dl, xb + 4 * XS, x);
                psf_row<T, N1, N1, true>(tb, x, acc, nr);
              } else if (kd == 1) {
                psf_scale<T, NQ, 1, false>(l, xb + 6 * XS, x);
                psf_row<T, N1, N1, false>(tb, x, acc, nr);
                psf_scale<T, NQ, 1, false>(l, xb + 7 * XS, x);
                psf_row<T, N1, N1, true>(tb, x, acc, nr);
              } else {
                psf_scale<T, NQ, 1, false>(l, xb + (kd == 2 ? 2 : 8) * XS, x);
                if (kd == 2) psf_scale<T, NQ, 1, true>(dl, xb + 5 * XS, x);
                psf_row<T, N1, N1, false>(tb, x, acc, nr);
              }
              T* o = Y + ((size_t)(vp * 4 + kd) * CQ + z) * NP * YP + pt * YP + sf32_pair0(N1, ar);
#pragma unroll
              for (int b = 0; b < N1; ++b)
                if (b < nr) o[b] = acc[b];
            }
            __syncthreads();
            // the modes, direction 2
            // (an item: a test mode and a pair of trial degrees, the pair slowest)
            for (int t = tid; t < np * NP * NM; t += C::NT) {
              const int vr = t / NM, it = t - vr * NM, vp = vr / NP, pr = vr - vp * NP;
              const int nr = N1 - (ptab[pr] & 255) - (ptab[pr] >> 8), m2 = mk[2 * NM + pmode[it]], a2t = m2 >> 8;
              const T* y = Y + (size_t)vp * 4 * CQ * NP * YP + (m2 & 255) * YP + pr;
              T acc[N1];
#pragma unroll
              for (int b = 0; b < N1; ++b) acc[b] = T(0);
              for (int z = 0; z < nz; ++z) {
                const T l = sL[a2t * NQ + z0 + z], dl = sdL[a2t * NQ + z0 + z];
                const T p = l * y[z * NP * YP] + dl * y[(CQ + z) * NP * YP];
                const T q = l * y[(2 * CQ + z) * NP * YP] + dl * y[(3 * CQ + z) * NP * YP];
#pragma unroll
                for (int b = 0; b < N1; ++b)
                  if (sizeof(T) == 4 || b < nr) acc[b] += p * tb.L[b][z0 + z] + q * tb.dL[b][z0 + z];
              }
              T* o = Da + ((size_t)vp * NM + it) * NM + poff[pr];
#pragma unroll
              for (int b = 0; b < N1; ++b)
                if (b < nr) o[b] = z0 == 0 ? acc[b] : o[b] + acc[b];
            }
            __syncthreads();
          }
          for (int t = tid; t < np * NM * NM; t += C::NT) {
            const int vp = t / (NM * NM), r = t - vp * NM * NM, a = r / NM, b = r - a * NM;
            De[(size_t)((v0 + vb + vp) * NM + pmode[a]) * NB + w * NM + pmode[b]] = Da[t];
          }
          // (Da is next written two barriers on)
        }
        __syncthreads();
      }
    }
    // ================= faces
    if constexpr (!CACHED && C::FT) {
      for (int t = tid; t < 12 * NL; t += C::NT) {
        const int fs = t / NL, q = t - fs * NL;
        T c[20];
        psf_face_trace<T, N1>(mv, sW, fs >> 1, fs & 1, q, c);
#pragma unroll
        for (int j = 0; j < 20; ++j) P[(fs * 20 + j) * NL + q] = c[j];
      }
      __syncthreads();
    }
    for (int w = 0; w < M; ++w) {
      for (int t = tid; t < 4 * 6 * NL; t += C::NT) {
        const int s = t / (6 * NL), fq = t - s * 6 * NL, f = fq / NL, q = fq - f * NL, k = f >> 1, side = f & 1;
        // the face's L element sees it at its +1 end: side 1 is this element's +1 face
        T c[2][20];
        if constexpr (CACHED) {
          const long fl = (long)k * E + (side ? e : mv.nbr[e * 6 + f]);
#pragma unroll
          for (int sd = 0; sd < 2; ++sd)
#pragma unroll
            for (int j = 0; j < 5; ++j) {
              const float4 x = __ldg(Pf + sf32_face_word(fl, sd, j, q, NL));
              c[sd][4 * j] = (T)x.x, c[sd][4 * j + 1] = (T)x.y, c[sd][4 * j + 2] = (T)x.z, c[sd][4 * j + 3] = (T)x.w;
            }
        } else {
#pragma unroll
          for (int sd = 0; sd < 2; ++sd) {
            if constexpr (C::FT) {
#pragma unroll
              for (int j = 0; j < 20; ++j) c[sd][j] = P[((f * 2 + sd) * 20 + j) * NL + q];
            } else {
              psf_face_trace<T, N1>(mv, sW, f, sd, q, c[sd]);
            }
          }
        }
        if (s == 0 && w == 0 && (!physical<3>(c[0], ph.gm1) || !physical<3>(c[1], ph.gm1)))
          atomicOr(status, ST_NONPHYSICAL);
        psf_face_jac<T, N1, true>(tb, ph, c, k, side, q, s, w, Jf + (size_t)f * M * 8 * NL + q);
      }
      __syncthreads();
      for (int v = 0; v < M; ++v) {      // v in each face's own frame: see the last loop for the rows
        // F1, sums over b0: arrays 0 flux + d_t0 trial + d_t0 test, 1 lifting, 2 normal-derivative
        // trial, 3 d_t1 trial, 4 normal-derivative test, 5 d_t1 test (each value-value in t0)
        for (int t = tid; t < 6 * N1 * 6 * NQ; t += C::NT) {
          const int aa = t / (6 * NQ), r = t - aa * 6 * NQ, arr = aa / N1, at = aa - arr * N1, f = r / NQ, b1 = r - f * NQ,
                    k = f >> 1;
          // row variable v (physical) in the face's frame
          const int t0 = k == 0 ? 1 : 0, vf = v == 0 || v == M - 1 ? v : v == 1 + k ? 1 : v == 1 + t0 ? 2 : 3;
          const T* j = Jf + ((size_t)(f * M + vf) * 8) * NL + b1;
          const int kind = arr == 0 ? 0 : arr == 1 ? 1 : arr == 2 ? 2 : arr == 3 ? 4 : arr == 4 ? 5 : 7;
          const T *l = sL + at * NQ, *dl = sdL + at * NQ;
          T x[NQ], acc[N1];
#pragma unroll
          for (int b = 0; b < N1; ++b) acc[b] = T(0);
          psf_scale<T, NQ, NQ, false>(l, j + kind * NL, x);
          if (arr == 0) psf_scale<T, NQ, NQ, true>(dl, j + 6 * NL, x);
          psf_row<T, N1, N1, false>(tb, x, acc, N1);
          if (arr == 0) {
            psf_scale<T, NQ, NQ, false>(l, j + 3 * NL, x);
            psf_row<T, N1, N1, true>(tb, x, acc, N1);
          }
          T* o = F1 + ((size_t)(f * 6 + arr) * N2 + at * N1) * XQ + b1;
#pragma unroll
          for (int b = 0; b < N1; ++b) o[b * XQ] = acc[b];
        }
        __syncthreads();
        // A, B, C: sums over b1, an item a test pair, a0 and a face (the matrix slowest)
        for (int t = tid; t < 3 * N1 * NP * 6; t += C::NT) {
          const int oa = t / (NP * 6), r = t - oa * (NP * 6), out = oa / N1, ar = oa - out * N1, f = r / NP, pt = r - f * NP;
          const int at = ptab[pt] & 255, a1t = ptab[pt] >> 8, nr = N1 - ar;
          constexpr int FS = N2 * XQ;                // from one array to the next
          const T* fb = F1 + (size_t)f * 6 * FS + (at * N1 + ar) * XQ;
          const T *l = sL + a1t * NQ, *dl = sdL + a1t * NQ;
          T x[NQ], acc[N1];
#pragma unroll
          for (int b = 0; b < N1; ++b) acc[b] = T(0);
          if (out == 0) {
            const T n = (T)(N1 - at - a1t);          // the lifting's factor n^2 / 2, n values of the normal degree
#pragma unroll
            for (int q = 0; q < NQ; ++q) x[q] = l[q] * (fb[q] + n * n * fb[FS + q]);
            psf_scale<T, NQ, 1, true>(dl, fb + 5 * FS, x);
            psf_row<T, N1, N1, false>(tb, x, acc, nr);
            psf_scale<T, NQ, 1, false>(l, fb + 3 * FS, x);
            psf_row<T, N1, N1, true>(tb, x, acc, nr);
          } else {
            psf_scale<T, NQ, 1, false>(l, fb + (out == 1 ? 2 : 4) * FS, x);
            psf_row<T, N1, N1, false>(tb, x, acc, nr);
          }
          T* o = A + (size_t)(f * 3 + out) * NP * YP + pt * YP + sf32_pair0(N1, ar);
#pragma unroll
          for (int b = 0; b < N1; ++b)
            if (b < nr) o[b] = acc[b];
        }
        __syncthreads();
        // over the modes: D += Le' Le A + Le' dLe B + dLe' Le C, both ends of three directions
        // (a batch of entries loaded at once)
        for (int tb0 = tid; tb0 < NM * NM; tb0 += 4 * C::NT) {
          T dv[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int t = min(tb0 + u * C::NT, NM * NM - 1), it = t / NM, ir = t - it * NM;
            dv[u] = De[(size_t)(v * NM + it) * NB + w * NM + ir];
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int t = tb0 + u * C::NT, it = t / NM, ir = t - it * NM;
            if (t >= NM * NM) break;
            T acc = dv[u];
            if (v == w && it == ir) acc += sigma * tb.detJ;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const int mt = mk[k * NM + it], mr = mk[k * NM + ir], at = mt >> 8, ar = mr >> 8;
              const T lt = Le[at], dt = Le[N1 + at], lr = Le[ar], dr = Le[N1 + ar];
              const T* a = A + (size_t)(2 * k) * 3 * NP * YP + (mt & 255) * YP + (mr & 255);   // the face at -1
              const T* b = a + 3 * NP * YP;                                                    // the face at +1
              // at -1 each value of odd degree and each derivative of even degree changes sign
              const T ps = (at + ar) & 1 ? T(-1) : T(1);
              acc += lt * lr * (b[0] + ps * a[0]);
              acc += lt * dr * (b[NP * YP] - ps * a[NP * YP]);
              acc += dt * lr * (b[2 * NP * YP] - ps * a[2 * NP * YP]);
            }
            De[(size_t)(v * NM + it) * NB + w * NM + ir] = acc;
          }
        }
        // (F1 is next written after this loop's reads of A only; A two barriers on)
      }
      __syncthreads();
    }
  }
}

template <class T, int N1, int VG, int VP, int CQ, bool CACHED>
cudaError_t run_probe_sf(const Mesh& Ms, const T* W, T sigma, T* D, size_t dstride, const float4* Pv, const float4* Pf,
                         cudaStream_t st) {
  using C = Psf<T, N1, VG, VP, CQ, CACHED>;
  static_assert(C::bytes <= 227 * 1024, "shared memory");
  auto kern = probe_sf_kernel<T, N1, VG, VP, CQ, CACHED>;
  cudaError_t e = allow_max_smem(kern);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, C::NT, C::bytes);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorNotSupported;
  note_launch();
  kern<<<std::min(Ms.E, occ * sm_count()), C::NT, C::bytes, st>>>(
      sf_tab<T, N1>(Ms), Ms.view<T>(), Ms.phys_t<T>(), Ms.qidx, W, sigma, D, dstride, Ms.status, Pv, Pf);
  return cudaGetLastError();
}

}  // namespace dgk
