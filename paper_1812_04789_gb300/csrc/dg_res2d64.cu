// FP64 face and volume terms of 2-D structured meshes (Sec. 3-4: Roe flux, BR2
// lifting, dual-consistent viscous term, volume fluxes), residual and
// Jacobian-vector product.
//
// An FP64 instruction occupies its warp for 64 clocks and its SM for 19 (four
// warps keep the pipe busy; measured), whatever the number of active lanes.  A
// small mesh is therefore bound by the longest chain of FP64 instructions of
// one thread, a large one by the number of warp instructions.  With a thread
// per point doing everything, 16^2 quads at p = 2 took 38 us for a JVP's face
// terms: 750 instructions in a row.  Hence
//  * interpolation: an item per (state or direction, side, value or derivative,
//    point), M values of n_m multiply-adds each;
//  * the point physics in three roles on three warps (Roe flux; each side's
//    viscous flux and dual tensor) where a CTA has at most 32 points, which
//    leaves three of four issue slots idle otherwise; two primitive states
//    more, so a thread per point where there are more points;
//  * lifting per (point, variable) on the three independent integrands, and
//    projection per (side, mode, variable): the tensor's factors 4/3, -2/3 are
//    taken out of the sums over the points.
// 16^2 quads, p = 2: JVP, face 37 -> 18 us, volume 17 -> 12 us; residual 25 -> 13
// and 13 -> 9 us.  Large meshes: the lines below.
#include <algorithm>

#include "dg_internal.h"

namespace dgk {

namespace {

constexpr int R2_THREADS = 128;
constexpr int M2 = 4;     // variables

// value and tangent at point pt of array entry c of a side's 12 (u[4], d_0 u[4], d_1 u[4])
template <bool JVP, class S>
__device__ __forceinline__ void r2_state(const double* sU, int np, int pt, S* u, S (*g)[2]) {
#pragma unroll
  for (int v = 0; v < M2; ++v) {
    if constexpr (JVP) {
      u[v] = S(sU[v * np + pt], sU[(12 + v) * np + pt]);
      g[v][0] = S(sU[(4 + v) * np + pt], sU[(16 + v) * np + pt]);
      g[v][1] = S(sU[(8 + v) * np + pt], sU[(20 + v) * np + pt]);
    } else {
      u[v] = sU[v * np + pt];
      g[v][0] = sU[(4 + v) * np + pt];
      g[v][1] = sU[(8 + v) * np + pt];
    }
  }
}
template <bool JVP, class S>
__device__ __forceinline__ double r2_out(const S& x) {
  if constexpr (JVP)
    return tan_part(x);
  else
    return val(x);
}

// one side's viscous flux (half of it) and rank-one tensor; k the face's direction
template <int k, bool JVP, class S>
__device__ __forceinline__ void r2_visc(const S* u, const S (*g)[2], const S* jump, const Phys<double>& ph, double* X,
                                        double* Dm, int np) {
  Prim<2, S> P;
  primitives<2, S, double>(u, ph, P);
  S F[M2], m[2], e[2];
#pragma unroll
  for (int v = 0; v < M2; ++v) F[v] = 0.0;
  add_visc_col<2, k, S, double>(P, g, 0.5, F, ph);
  visc_rank1<2, k, S, double>(P, jump, 0.5, m, e, ph);
#pragma unroll
  for (int v = 1; v < M2; ++v) X[v * np] = r2_out<JVP>(F[v]);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    Dm[j * np] = r2_out<JVP>(m[j]);
    Dm[(2 + j) * np] = r2_out<JVP>(e[j]);
  }
}
template <int k, bool JVP, class S>
__device__ __forceinline__ void r2_roe(const S* uL, const S* uR, const Phys<double>& ph, double* F, int np) {
  S f[M2];
  roe_flux<2, k, S, double>(uL, uR, f, ph);
#pragma unroll
  for (int v = 0; v < M2; ++v) F[v * np] = r2_out<JVP>(f[v]);
}

// doubles of shared memory per face
inline size_t r2_face_doubles(int nm, int nqf, bool jvp, bool split) {
  const int K = jvp ? 2 : 1;
  return (size_t)K * 2 * nm * M2 + (size_t)nqf * (24 * K + M2 + 8 + (split ? 2 * M2 : 0));
}

template <bool JVP, bool SPLIT>
__global__ void __launch_bounds__(R2_THREADS, 2) face2d64_kernel(MeshView<double> mv, Phys<double> ph,
                                                                 const double* __restrict__ W,
                                                                 const double* __restrict__ V,
                                                                 double* __restrict__ slots, int* status, int fpc) {
  using S = typename std::conditional<JVP, Dual<double>, double>::type;
  constexpr int K = JVP ? 2 : 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nb = mv.nb, nm = mv.nm, nqf = mv.nqf, E = mv.E, tid = threadIdx.x;
  const int f0 = blockIdx.x * fpc, nl = min(fpc, 2 * E - f0), np = fpc * nqf, npl = nl * nqf;
  if (nl <= 0) return;
  double* sW = reinterpret_cast<double*>(smem_raw);   // [K][face][side][mode][4]
  double* sU = sW + (size_t)K * fpc * 2 * nm * M2;    // [side][K][12][point]
  double* sF = sU + (size_t)24 * K * np;              // [4][point]
  double* sD = sF + (size_t)M2 * np;                  // [side][m_0, m_1, e_0, e_1][point]
  double* sX = sD + (size_t)8 * np;                   // SPLIT: [side][4][point]
  for (int t = tid; t < nl * 2 * nb; t += R2_THREADS) {
    const int fl = t / (2 * nb), r = t - fl * 2 * nb, side = r / nb, j = r - side * nb, v = j / nm, i = j - v * nm;
    const int f = f0 + fl, k = f / E, e = f - k * E, el = side == 0 ? e : mv.nbr[(e * 2 + k) * 2 + 1];
    const size_t o = ((size_t)(fl * 2 + side) * nm + i) * M2 + v;
    sW[o] = W[(size_t)el * nb + j];
    if (JVP) sW[(size_t)fpc * 2 * nm * M2 + o] = V[(size_t)el * nb + j];
  }
  __syncthreads();
  for (int t = tid; t < 6 * K * npl; t += R2_THREADS) {
    const int a = t / npl, pt = t - a * npl, c = a % 3, ks = a / 3, side = ks & 1, kc = ks >> 1;
    const int fl = pt / nqf, q = pt - fl * nqf, k = (f0 + fl) / E, lf = side == 0 ? 2 * k + 1 : 2 * k;
    const double* w = sW + ((size_t)((kc * fpc + fl) * 2 + side) * nm) * M2;
    const double* b = mv.fpk + ((size_t)lf * nm * nqf + q) * 4 + c;
    double acc[M2] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int i = 0; i < nm; ++i) {
      const double p = __ldg(b + (size_t)i * nqf * 4);
      double x[M2];
      ld_vec<double, M2>(w + (size_t)i * M2, x);
#pragma unroll
      for (int v = 0; v < M2; ++v) acc[v] += x[v] * p;
    }
    double* o = sU + (size_t)((side * K + kc) * 12 + c * 4) * np + pt;
#pragma unroll
    for (int v = 0; v < M2; ++v) o[v * np] = acc[v];
  }
  __syncthreads();
  const double* UL = sU;
  const double* UR = sU + (size_t)12 * K * np;
  if constexpr (SPLIT) {
    const int npr = (npl + 31) / 32 * 32;             // roles on warps of their own
    for (int t = tid; t < 3 * npr; t += R2_THREADS) {
      const int role = t / npr, pt = t - role * npr;
      if (pt >= npl) continue;
      const int k = (f0 + pt / nqf) / E;
      S uL[M2], uR[M2], gL[M2][2], gR[M2][2];
      r2_state<JVP>(UL, np, pt, uL, gL);
      r2_state<JVP>(UR, np, pt, uR, gR);
      if (role == 0) {
        if (!physical<2>(uL, ph.gm1) || !physical<2>(uR, ph.gm1)) atomicOr(status, ST_NONPHYSICAL);
        if (k == 0)
          r2_roe<0, JVP>(uL, uR, ph, sF + pt, np);
        else
          r2_roe<1, JVP>(uL, uR, ph, sF + pt, np);
      } else {
        const int side = role - 1;
        S u[M2], g[M2][2], jump[M2];
#pragma unroll
        for (int v = 0; v < M2; ++v) {
          jump[v] = uL[v] - uR[v];
          u[v] = side ? uR[v] : uL[v];
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) g[v][kk] = side ? gR[v][kk] : gL[v][kk];
        }
        double *X = sX + (size_t)side * M2 * np + pt, *Dm = sD + (size_t)side * 4 * np + pt;
        if (k == 0)
          r2_visc<0, JVP>(u, g, jump, ph, X, Dm, np);
        else
          r2_visc<1, JVP>(u, g, jump, ph, X, Dm, np);
      }
    }
  } else {
    for (int pt = tid; pt < npl; pt += R2_THREADS) {
      const int k = (f0 + pt / nqf) / E;
      S uL[M2], uR[M2], gL[M2][2], gR[M2][2], fp[M2], mL[2], eL[2], mR[2], eR[2];
      r2_state<JVP>(UL, np, pt, uL, gL);
      r2_state<JVP>(UR, np, pt, uR, gR);
      if (!physical<2>(uL, ph.gm1) || !physical<2>(uR, ph.gm1)) atomicOr(status, ST_NONPHYSICAL);
      face_point_core_k<2, S, double>(k, uL, gL, uR, gR, ph, fp, mL, eL, mR, eR);
#pragma unroll
      for (int v = 0; v < M2; ++v) sF[v * np + pt] = r2_out<JVP>(fp[v]);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        sD[j * np + pt] = r2_out<JVP>(mL[j]);
        sD[(2 + j) * np + pt] = r2_out<JVP>(eL[j]);
        sD[(4 + j) * np + pt] = r2_out<JVP>(mR[j]);
        sD[(6 + j) * np + pt] = r2_out<JVP>(eR[j]);
      }
    }
  }
  __syncthreads();
  // lifting on both sides: the integrand of variable v is twice the normal column of its tensor
  for (int t = tid; t < 3 * npl; t += R2_THREADS) {
    const int v = 1 + t / npl, pt = t - (v - 1) * npl, fl = pt / nqf, q = pt - fl * nqf, k = (f0 + fl) / E;
    const int idx = v == 3 ? 2 + k : v - 1;           // e_k or m_j
    const double cf = v - 1 == k ? 8.0 / 3.0 : 2.0;
    const double* PL = mv.lift + (size_t)(2 * k + 1) * nqf * nqf + q;
    const double* PR = mv.lift + (size_t)(2 * k) * nqf * nqf + q;
    const double *a = sD + (size_t)idx * np + fl * nqf, *b = a + 4 * np;
    double dl = 0.0, dr = 0.0;
#pragma unroll 4
    for (int q2 = 0; q2 < nqf; ++q2) {
      dl += __ldg(PL + (size_t)q2 * nqf) * a[q2];
      dr += __ldg(PR + (size_t)q2 * nqf) * b[q2];
    }
    double f = sF[v * np + pt];
    if (SPLIT) f += sX[v * np + pt] + sX[(M2 + v) * np + pt];
    sF[v * np + pt] = f + (ph.eta * 0.5 * cf) * (dl + dr);
  }
  __syncthreads();
  for (int t = tid; t < nl * 2 * nb; t += R2_THREADS) {
    const int fs = t / nb, j = t - fs * nb, v = j / nm, i = j - v * nm, fl = fs >> 1, side = fs & 1;
    const int f = f0 + fl, k = f / E, e = f - k * E, lf = side == 0 ? 2 * k + 1 : 2 * k;
    // G[v][kk] = cf[kk] x entry id[kk] of (m, e): see visc_rank1
    int id0 = 0, id1 = 0;
    double cf0 = 0.0, cf1 = 0.0;
    if (v == 3) {
      id0 = 2, id1 = 3;
      cf0 = cf1 = 1.0;
    } else if (v == 1) {      // j = 0
      id0 = 0, cf0 = k == 0 ? 4.0 / 3.0 : -2.0 / 3.0;     // kk = 0: normal 4/3 m_0; tangential -2/3 m_k
      id1 = k == 0 ? 1 : 0, cf1 = 1.0;                    // kk = 1: tangential m_1; normal m_0
      if (k == 1) id0 = 1;
    } else if (v == 2) {      // j = 1
      id1 = 1, cf1 = k == 1 ? 4.0 / 3.0 : -2.0 / 3.0;
      id0 = k == 1 ? 0 : 1, cf0 = 1.0;
      if (k == 0) id1 = 0;
    }
    const double* pw = mv.fpw + ((size_t)lf * nqf * nm + i) * 4;
    const double* F = sF + (size_t)v * np + fl * nqf;
    const double *d0 = sD + (size_t)(side * 4 + id0) * np + fl * nqf, *d1 = sD + (size_t)(side * 4 + id1) * np + fl * nqf;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll 4
    for (int q = 0; q < nqf; ++q) {
      double w[4];
      ld_vec<double, 4>(pw + (size_t)q * nm * 4, w);
      s0 += w[0] * F[q];
      s1 += w[1] * d0[q];
      s2 += w[2] * d1[q];
    }
    const double fn = side == 0 ? s0 : -s0;
    slots[(((size_t)e * 2 + k) * 2 + side) * nb + j] = v == 0 ? fn : fn - cf0 * s1 - cf1 * s2;
  }
}

template <bool JVP>
__global__ void __launch_bounds__(R2_THREADS, 2) vol2d64_kernel(MeshView<double> mv, Phys<double> ph,
                                                                const double* __restrict__ W,
                                                                const double* __restrict__ V,
                                                                const double* __restrict__ slots,
                                                                const double* __restrict__ Src, double sigma,
                                                                double* __restrict__ out, int* status, int epc) {
  using S = typename std::conditional<JVP, Dual<double>, double>::type;
  constexpr int K = JVP ? 2 : 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nb = mv.nb, nm = mv.nm, nq = mv.nq, E = mv.E, tid = threadIdx.x;
  const int e0 = blockIdx.x * epc, nl = min(epc, E - e0), np = epc * nq, npl = nl * nq;
  if (nl <= 0) return;
  double* sW = reinterpret_cast<double*>(smem_raw);   // [K][element][mode][4]
  double* sU = sW + (size_t)K * epc * nm * M2;        // [K][12][point]
  double* sF = sU + (size_t)12 * K * np;              // [v][k][point], weighted
  for (int t = tid; t < nl * nb; t += R2_THREADS) {
    const int el = t / nb, j = t - el * nb, v = j / nm, i = j - v * nm;
    const size_t o = ((size_t)el * nm + i) * M2 + v;
    sW[o] = W[(size_t)e0 * nb + t];
    if (JVP) sW[(size_t)epc * nm * M2 + o] = V[(size_t)e0 * nb + t];
  }
  __syncthreads();
  for (int t = tid; t < 3 * K * npl; t += R2_THREADS) {
    const int a = t / npl, pt = t - a * npl, c = a % 3, kc = a / 3, el = pt / nq, q = pt - el * nq;
    const double* w = sW + (size_t)(kc * epc + el) * nm * M2;
    const double* b = (c == 0 ? mv.vphiT : mv.vdphiT + (size_t)(c - 1) * nm * nq) + q;
    double acc[M2] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int i = 0; i < nm; ++i) {
      const double p = __ldg(b + (size_t)i * nq);
      double x[M2];
      ld_vec<double, M2>(w + (size_t)i * M2, x);
#pragma unroll
      for (int v = 0; v < M2; ++v) acc[v] += x[v] * p;
    }
    double* o = sU + (size_t)(kc * 12 + c * 4) * np + pt;
#pragma unroll
    for (int v = 0; v < M2; ++v) o[v * np] = acc[v];
  }
  __syncthreads();
  for (int pt = tid; pt < npl; pt += R2_THREADS) {
    S u[M2], g[M2][2], F[M2][2];
    r2_state<JVP>(sU, np, pt, u, g);
    if (!physical<2>(u, ph.gm1)) atomicOr(status, ST_NONPHYSICAL);
    flux_total<2, S, double>(u, g, F, ph);
    const double wq = mv.vw[pt % nq];
#pragma unroll
    for (int v = 0; v < M2; ++v)
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) sF[(v * 2 + kk) * np + pt] = wq * r2_out<JVP>(F[v][kk]);
  }
  __syncthreads();
  for (int t = tid; t < nl * nb; t += R2_THREADS) {
    const int el = t / nb, j = t - el * nb, v = j / nm, i = j - v * nm, e = e0 + el;
    const double *f = sF + (size_t)v * 2 * np + el * nq, *d0 = mv.vdphi + i, *d1 = d0 + (size_t)nq * nm;
    double a0 = 0.0, a1 = 0.0;
#pragma unroll 4
    for (int q = 0; q < nq; ++q) {
      a0 -= __ldg(d0 + (size_t)q * nm) * f[q];
      a1 -= __ldg(d1 + (size_t)q * nm) * f[np + q];
    }
    double acc = a0 + a1;
    // face contributions in fixed order: for each direction, own +k face then -k face
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int em = mv.nbr[(e * 2 + k) * 2 + 0];
      acc += slots[(((size_t)e * 2 + k) * 2 + 0) * nb + j];
      acc += slots[(((size_t)em * 2 + k) * 2 + 1) * nb + j];
    }
    if (JVP)
      acc += sigma * mv.detJ * sW[(size_t)(epc + el) * nm * M2 + (size_t)i * M2 + v];
    else if (Src)
      acc -= Src[(size_t)e * nb + j];
    out[(size_t)e * nb + j] = acc;
  }
}

template <bool JVP>
cudaError_t run_face(const Mesh& M, const double* W, const double* V, double* slots, cudaStream_t st) {
  const int nfaces = 2 * M.E;
  // a CTA per SM while the faces allow, and up to a thread per point
  int fpc = std::max(1, std::min((nfaces + sm_count() - 1) / sm_count(), R2_THREADS / M.nqf));
  const bool split = fpc * M.nqf <= 32;
  size_t smem = 0;
  for (;; --fpc) {
    smem = sizeof(double) * fpc * r2_face_doubles(M.nm, M.nqf, JVP, split);
    if (smem <= 100 * 1024 || fpc == 1) break;
  }
  const int grid = (nfaces + fpc - 1) / fpc;
  cudaError_t e = split ? allow_max_smem(face2d64_kernel<JVP, true>) : allow_max_smem(face2d64_kernel<JVP, false>);
  if (e != cudaSuccess) return e;
  note_launch();
  if (split)
    face2d64_kernel<JVP, true><<<grid, R2_THREADS, smem, st>>>(M.view<double>(), M.phys_t<double>(), W, V, slots,
                                                               M.status, fpc);
  else
    face2d64_kernel<JVP, false><<<grid, R2_THREADS, smem, st>>>(M.view<double>(), M.phys_t<double>(), W, V, slots,
                                                                M.status, fpc);
  return cudaGetLastError();
}

template <bool JVP>
cudaError_t run_vol(const Mesh& M, const double* W, const double* V, const double* slots, const double* Src,
                    double sigma, double* out, cudaStream_t st) {
  const int K = JVP ? 2 : 1;
  int epc = std::max(1, std::min((M.E + sm_count() - 1) / sm_count(), R2_THREADS / M.nq));
  const size_t per = sizeof(double) * ((size_t)K * M.nm * M2 + (size_t)M.nq * (12 * K + 8));
  while (epc > 1 && epc * per > 100 * 1024) --epc;
  const cudaError_t e = allow_max_smem(vol2d64_kernel<JVP>);
  if (e != cudaSuccess) return e;
  note_launch();
  vol2d64_kernel<JVP><<<(M.E + epc - 1) / epc, R2_THREADS, epc * per, st>>>(M.view<double>(), M.phys_t<double>(), W, V,
                                                                           slots, Src, sigma, out, M.status, epc);
  return cudaGetLastError();
}

}  // namespace

// The lines, measured against the thread-per-point kernels (us, those / these):
// face terms of the residual 25 / 13 (16^2, p = 2), 129 / 121 (100 x 75, p = 3),
// 1,053 / 982 (256^2, p = 3): always; of a JVP 37 / 18, 55 / 47 (32^2, p = 2), 103
// / 106 (48^2, p = 3, 151 points per SM), 251 / 270 (128^2, p = 2); volume terms of
// a JVP 17 / 12, 18 / 19 (32^2, p = 2, 108 points per SM), 151 / 166 (100 x 75).
bool face2d64_ok(const Mesh& M, bool jvp) { return !jvp || 2L * M.E * M.nqf <= 128L * sm_count(); }
bool vol2d64_ok(const Mesh& M) { return (long)M.E * M.nq <= 64L * sm_count(); }

cudaError_t launch_face2d64(const Mesh& M, const double* W, const double* V, double* slots, bool jvp, cudaStream_t st) {
  return jvp ? run_face<true>(M, W, V, slots, st) : run_face<false>(M, W, V, slots, st);
}
cudaError_t launch_vol2d64(const Mesh& M, const double* W, const double* V, const double* slots, const double* Src,
                           double sigma, double* out, bool jvp, cudaStream_t st) {
  return jvp ? run_vol<true>(M, W, V, slots, Src, sigma, out, st) : run_vol<false>(M, W, V, slots, Src, sigma, out, st);
}

}  // namespace dgk
