// Neighbour blocks of 3-D P_p meshes on the first coarse order (Sec. 6.3: the
// inherited block-sparse operator's off-diagonal part, dR_e/dW_nbr restricted to
// the modes of order NC - 1) by sum factorisation, in FP32 and FP64
// (dg_nbr_sf32.cu, dg_nbr_sf64.cu): the face part of dg_probe_sf.cuh with the
// neighbour's state seeded and pairs of the coarse degrees,
//   O = lt lr A + lt dr B + dt lr C,
// lt, dt the own test end value and derivative in the face's normal direction,
// lr, dr the neighbour's (which sees the face at its other end).  One CTA takes
// an element's six faces; per seed variable w one dual-number evaluation per
// point gives the value seed and three direct ones the gradient seeds (the
// kernels before, probe_nbr_kernel and probe64_kernel's neighbour part, spend a
// dual evaluation or a dense sum of point Jacobians on all four).  Bound by
// instruction issue (FP32) and the FP64 pipe.
// To coarse order 0, FP32, 16^3 elements: p = 4 2.15 -> 0.43 ms, p = 6 4.3 -> 0.63
// ms; FP64, 12^3, p = 4: 9.0 -> 4.0 ms.
#pragma once
#include "dg_probe_sf.cuh"

namespace dgk {

template <class T, int N1, int NC>
struct Nsf {
  static constexpr bool CACHED = sizeof(T) == 4;
  static constexpr int NT = 256, NQ = N1 + 1, NL = NQ * NQ, NP = sf32_pairs(NC), NM = sf32_modes(NC), M = 5,
                       NB = M * sf32_modes(N1), XQ = NQ | 1, YP = NP | 1;
  // [Jf | F1 | A | traces | W], F1 and A of VB output variables at once
  static constexpr int nJf = 6 * M * 8 * NL, f1 = 36 * NC * NC * XQ, a1 = 18 * NP * YP;
  static constexpr int nP = CACHED ? 0 : 6 * NL * 40, nW = CACHED ? 0 : 7 * NB, tail = 2 * N1 + 2 * NC * NQ;
  static constexpr size_t nS = sizeof(unsigned short) * (NP + 3 * NM + 4);
  static constexpr size_t of(int vb) { return sizeof(T) * (nJf + vb * (f1 + a1) + nP + nW + tail) + nS; }
  // all five together (fewer barriers) where that leaves room for two CTAs (FP32) or one
  static constexpr int VB = of(M) <= (CACHED ? 113 : 227) * 1024 ? M : 1;
  static constexpr size_t bytes = of(VB);
};

template <class T, int N1, int NC>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1)
    nbr_sf_kernel(const __grid_constant__ SfTab<T, N1> tb, MeshView<T> mv, Phys<T> ph, const int* __restrict__ qidx,
                  const T* __restrict__ W, T* __restrict__ O, size_t ostride, int ldo, const float4* __restrict__ Pf) {
  using C = Nsf<T, N1, NC>;
  constexpr int NQ = C::NQ, NL = C::NL, NP = C::NP, NM = C::NM, M = C::M, NB = C::NB, XQ = C::XQ, YP = C::YP, VB = C::VB,
                N2 = NC * NC;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Jf = reinterpret_cast<T*>(smem_raw);   // [face][v][8][b1 + NQ b0]
  T* F1 = Jf + C::nJf;                      // [v][face][6][a0' a0][b1]
  T* A = F1 + VB * C::f1;                   // [v][face][3][pair' pair]
  T* P = A + VB * C::a1;                    // [face][side][20][NL]
  T* sW = P + C::nP;                        // [element, neighbours][NB]
  T* Le = sW + C::nW;                       // values at +1, then derivatives
  T *sL = Le + 2 * N1, *sdL = sL + NC * NQ;
  unsigned short* ptab = reinterpret_cast<unsigned short*>(sdL + NC * NQ);   // pair -> a0 | a1 << 8
  unsigned short* mk = ptab + NP;                                            // [k][mode]: pair | a_k << 8
  const int tid = threadIdx.x, E = mv.E;
  for (int t = tid; t < N2; t += C::NT) {
    const int a0 = t / NC, a1 = t - a0 * NC;
    if (a0 + a1 < NC) ptab[sf32_pair0(NC, a0) + a1] = (unsigned short)(a0 | a1 << 8);
  }
  for (int t = tid; t < NC * N2; t += C::NT) {
    const int x0 = t % NC, x1 = t / NC % NC, x2 = t / N2;
    if (x0 + x1 + x2 < NC) {      // the coarse modes are the first NM of the fine order's
      const int i = qidx[x0 + N1 * (x1 + N1 * x2)];
      mk[i] = (unsigned short)((sf32_pair0(NC, x1) + x2) | x0 << 8);
      mk[NM + i] = (unsigned short)((sf32_pair0(NC, x0) + x2) | x1 << 8);
      mk[2 * NM + i] = (unsigned short)((sf32_pair0(NC, x0) + x1) | x2 << 8);
    }
  }
  for (int t = tid; t < 2 * N1; t += C::NT) Le[t] = t < N1 ? tb.Le[t] : tb.dLe[t - N1];
  for (int t = tid; t < NC * NQ; t += C::NT) {
    sL[t] = tb.L[t / NQ][t % NQ];
    sdL[t] = tb.dL[t / NQ][t % NQ];
  }
  for (int e = blockIdx.x; e < E; e += gridDim.x) {
    if constexpr (!C::CACHED) {
      __syncthreads();
      for (int t = tid; t < 7 * NB; t += C::NT) {
        const int who = t / NB, j = t - who * NB, el = who == 0 ? e : mv.nbr[e * 6 + who - 1];
        sW[t] = W[(size_t)el * NB + j];
      }
      __syncthreads();
      for (int t = tid; t < 12 * NL; t += C::NT) {
        const int fs = t / NL, q = t - fs * NL;
        T c[20];
        psf_face_trace<T, N1>(mv, sW, fs >> 1, fs & 1, q, c);
#pragma unroll
        for (int j = 0; j < 20; ++j) P[(fs * 20 + j) * NL + q] = c[j];
      }
    }
    __syncthreads();
    for (int w = 0; w < M; ++w) {
      // (Jf is last read before the barrier that precedes A's last use)
      for (int t = tid; t < 4 * 6 * NL; t += C::NT) {
        const int s = t / (6 * NL), fq = t - s * 6 * NL, f = fq / NL, q = fq - f * NL, k = f >> 1, side = f & 1;
        T c[2][20];
        if constexpr (C::CACHED) {
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
          for (int sd = 0; sd < 2; ++sd)
#pragma unroll
            for (int j = 0; j < 20; ++j) c[sd][j] = P[((f * 2 + sd) * 20 + j) * NL + q];
        }
        psf_face_jac<T, N1, false>(tb, ph, c, k, side, q, s, w, Jf + (size_t)f * M * 8 * NL + q);
      }
      __syncthreads();
      for (int v0 = 0; v0 < M; v0 += VB) {
        // sums over b0 and over b1, arrays and matrices as in probe_sf_kernel
        for (int t = tid; t < VB * 36 * NC * NQ; t += C::NT) {
          const int va = t / (36 * NC * NQ), aa_ = t - va * (36 * NC * NQ), aa = aa_ / (6 * NQ), r = aa_ - aa * 6 * NQ,
                    arr = aa / NC, at = aa - arr * NC, f = r / NQ, b1 = r - f * NQ, k = f >> 1, v = v0 + va;
          const int t0 = k == 0 ? 1 : 0, vf = v == 0 || v == M - 1 ? v : v == 1 + k ? 1 : v == 1 + t0 ? 2 : 3;
          const T* j = Jf + ((size_t)(f * M + vf) * 8) * NL + b1;
          const int kind = arr == 0 ? 0 : arr == 1 ? 1 : arr == 2 ? 2 : arr == 3 ? 4 : arr == 4 ? 5 : 7;
          const T *l = sL + at * NQ, *dl = sdL + at * NQ;
          T x[NQ], acc[NC];
#pragma unroll
          for (int b = 0; b < NC; ++b) acc[b] = T(0);
          psf_scale<T, NQ, NQ, false>(l, j + kind * NL, x);
          if (arr == 0) psf_scale<T, NQ, NQ, true>(dl, j + 6 * NL, x);
          psf_row<T, N1, NC, false>(tb, x, acc, NC);
          if (arr == 0) {
            psf_scale<T, NQ, NQ, false>(l, j + 3 * NL, x);
            psf_row<T, N1, NC, true>(tb, x, acc, NC);
          }
          T* o = F1 + ((size_t)((va * 6 + f) * 6 + arr) * N2 + at * NC) * XQ + b1;
#pragma unroll
          for (int b = 0; b < NC; ++b) o[b * XQ] = acc[b];
        }
        __syncthreads();
        for (int t = tid; t < VB * 18 * NC * NP; t += C::NT) {
          const int va = t / (18 * NC * NP), oa_ = t - va * (18 * NC * NP), oa = oa_ / (NP * 6), r = oa_ - oa * (NP * 6),
                    out = oa / NC, ar = oa - out * NC, f = r / NP, pt = r - f * NP;
          const int at = ptab[pt] & 255, a1t = ptab[pt] >> 8, nr = NC - ar;
          constexpr int FS = N2 * XQ;
          const T* fb = F1 + (size_t)(va * 6 + f) * 6 * FS + (at * NC + ar) * XQ;
          const T *l = sL + a1t * NQ, *dl = sdL + a1t * NQ;
          T x[NQ], acc[NC];
#pragma unroll
          for (int b = 0; b < NC; ++b) acc[b] = T(0);
          if (out == 0) {
            const T n = (T)(N1 - at - a1t);          // the lifting is the fine order's
#pragma unroll
            for (int q = 0; q < NQ; ++q) x[q] = l[q] * (fb[q] + n * n * fb[FS + q]);
            psf_scale<T, NQ, 1, true>(dl, fb + 5 * FS, x);
            psf_row<T, N1, NC, false>(tb, x, acc, nr);
            psf_scale<T, NQ, 1, false>(l, fb + 3 * FS, x);
            psf_row<T, N1, NC, true>(tb, x, acc, nr);
          } else {
            psf_scale<T, NQ, 1, false>(l, fb + (out == 1 ? 2 : 4) * FS, x);
            psf_row<T, N1, NC, false>(tb, x, acc, nr);
          }
          T* o = A + (size_t)((va * 6 + f) * 3 + out) * NP * YP + pt * YP + sf32_pair0(NC, ar);
#pragma unroll
          for (int b = 0; b < NC; ++b)
            if (b < nr) o[b] = acc[b];
        }
        __syncthreads();
        // over the modes; the index that is contiguous in memory fastest
        for (int t = tid; t < VB * 6 * NM * NM; t += C::NT) {
          const int vf = t / (NM * NM), r = t - vf * NM * NM, f = vf % 6, va = vf / 6, x1 = r / NM, x0 = r - x1 * NM;
          const int it = ldo > 0 ? x0 : x1, ir = ldo > 0 ? x1 : x0, k = f >> 1, v = v0 + va;
          const int mt = mk[k * NM + it], mr = mk[k * NM + ir], at = mt >> 8, ar = mr >> 8;
          // side 1: test functions at +1, the neighbour's at -1; side 0: the other way round (at -1 each
          // value of odd degree and each derivative of even degree changes sign)
          const T sv = ((f & 1 ? ar : at) & 1) ? T(-1) : T(1);
          const T lt = Le[at], dt = Le[N1 + at], lr = Le[ar], dr = Le[N1 + ar];
          const T* a = A + (size_t)(va * 6 + f) * 3 * NP * YP + (mt & 255) * YP + (mr & 255);
          const T o = f & 1 ? sv * (lr * (lt * a[0] + dt * a[2 * NP * YP]) - lt * dr * a[NP * YP])
                            : sv * (lt * (lr * a[0] + dr * a[NP * YP]) - dt * lr * a[2 * NP * YP]);
          T* Os = O + ((size_t)e * 6 + f) * ostride;
          const int row = v * NM + it, col = w * NM + ir;
          Os[ldo > 0 ? (size_t)col * ldo + row : (size_t)row * (M * NM) + col] = o;
        }
      }
    }
  }
}

template <class T, int N1, int NC>
cudaError_t run_nbr_sf(const Mesh& Ms, const T* W, T* O, int colmajor, const float4* Pf, cudaStream_t st) {
  using C = Nsf<T, N1, NC>;
  static_assert(C::bytes <= 227 * 1024, "shared memory");
  auto kern = nbr_sf_kernel<T, N1, NC>;
  cudaError_t e = allow_max_smem(kern);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, C::NT, C::bytes);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorNotSupported;
  const int nbc = C::M * C::NM, ldo = colmajor ? inv_ld<T>(nbc) : 0;
  note_launch();
  kern<<<std::min(Ms.E, occ * sm_count()), C::NT, C::bytes, st>>>(sf_tab<T, N1>(Ms), Ms.view<T>(), Ms.phys_t<T>(), Ms.qidx, W,
                                                                  O, (size_t)nbc * (ldo ? ldo : nbc), ldo, Pf);
  return cudaGetLastError();
}

template <class T, int N1>
cudaError_t run_nbr_sf(const Mesh& Ms, const T* W, T* O, int nmc, int colmajor, const float4* Pf, cudaStream_t st) {
  if (nmc == sf32_modes(1)) return run_nbr_sf<T, N1, 1>(Ms, W, O, colmajor, Pf, st);
  if constexpr (N1 > 2)
    if (nmc == sf32_modes(2)) return run_nbr_sf<T, N1, 2>(Ms, W, O, colmajor, Pf, st);
  if constexpr (N1 > 3)
    if (nmc == sf32_modes(3)) return run_nbr_sf<T, N1, 3>(Ms, W, O, colmajor, Pf, st);
  if constexpr (N1 > 4)
    if (nmc == sf32_modes(4)) return run_nbr_sf<T, N1, 4>(Ms, W, O, colmajor, Pf, st);
  if constexpr (N1 > 5)
    if (nmc == sf32_modes(5)) return run_nbr_sf<T, N1, 5>(Ms, W, O, colmajor, Pf, st);
  if constexpr (N1 > 6)
    if (nmc == sf32_modes(6)) return run_nbr_sf<T, N1, 6>(Ms, W, O, colmajor, Pf, st);
  return cudaErrorNotSupported;
}

}  // namespace dgk
