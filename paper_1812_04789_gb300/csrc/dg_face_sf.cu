// Face term of the residual / exact JVP on 3-D meshes by sum factorisation
// (Sec. 3.1 eq. dg_ns face terms, eq. visc_flux and the lifting of eq. re).
//
// On the face k of an element the basis functions are products
// L_a(xi_k = +-1) L_b(xi_t0) L_c(xi_t1) (t0 < t1 the two other directions) and
// the face points a tensor grid (b0, b1) of the same Gauss-Legendre points,
// q = b0 + nq b1.  Everything is done in the face's frame: directions (n, t0,
// t1), variables (rho, the momenta along n, t0, t1, rho e0); the physics is
// invariant under that permutation, so one copy of it (normal = first
// direction) serves all faces.  Traces of a field and of its gradient:
//   S1  c0[a0][a1] = sum_ak w L_ak(+-1),  c1[a0][a1] = sum_ak w L'_ak(+-1)
//   S2  d0[a0][b1] = sum_a1 c0 L_a1(b1),  d1 = sum_a1 c0 L'_a1(b1),  d2 = sum_a1 c1 L_a1(b1)
//   per point: u = sum_a0 d0 L_a0(b0), du/dt0 = sum d0 L'_a0(b0), du/dt1 = sum d1 L_a0(b0),
//              du/dn = sum d2 L_a0(b0)   (each derivative times its metric 2/h)
// and the projection onto both elements' test functions is the transposed
// sequence (X over b0, Y over b1, then the end values).  The total-degree
// space P_p is the subset a_k + a0 + a1 <= p of these products, Q_p all of
// them; the sums run over that subset only.
//
// In FP64 the kernel is bound by the FP64 pipe (two lanes per clock and SM), so
// the work is what counts, shared-memory traffic and index arithmetic are free:
//  * the fluxes of the two sides differ in sign only: one projection for both;
//  * the dual-consistency tensors have six independent entries per side
//    (visc_rank1), of which eight tangential contractions are needed;
//  * the BR2 lifting of eq. re is never formed at the points.  Both sides lift
//    with the same operator, delta = sum_a C_a psi_a (sum_q w psi_a G) / (2 |J|)
//    over the tangential products psi_a, C_a = sum_ak L_ak(+-1)^2 (n^2 / 2 for n
//    values of ak), and its projection onto psi_a' is exact (Gauss-Legendre,
//    nq >= p + 1), so in the projected flux it is a factor per (a0, a1):
//    Y_a += eta/2 C_a (1/h_k) (sum_q w psi_a (G_L + G_R)).
// FP64 operations per face at p = 4, JVP: 154 k -> 64 k (with the point
// physics of dg_common.cuh).  JVP, FP64, faces: 32^3 p = 6 79.7 -> 29 ms, 16^3 p =
// 4 3.64 -> 1.50 ms (FP64 pipe 72 % busy when each thread ran one sum at a time).
#include <algorithm>
#include <type_traits>

#include "dg_internal.h"

namespace dgk {

namespace {

constexpr int FSF_NP = 21;   // point values: flux 5, lifting integrand 4, two sides' tensors 6 each
constexpr int FSF_NX = 25;   // X arrays: flux 5, lifting 4, per side 5 with L and 3 with L'
constexpr int FSF_NY = 25;   // Y arrays: flux 5, per side 4 value and 4 normal-derivative parts, lifting 4

// shared-memory plan (elements of T); NC = interpolated real fields per side
struct FsfPlan {
  int n1, nq, nqf, NC, npair;
  size_t oV, oS, oT, per_face, total;
};

__host__ __device__ inline FsfPlan fsf_plan(int p, int nq, int nb, int M, bool total_degree, bool jvp, bool cached,
                                            int fpc) {
  FsfPlan P;
  P.n1 = p + 1;
  P.nq = nq;
  P.nqf = nq * nq;
  P.npair = total_degree ? P.n1 * (P.n1 + 1) / 2 : P.n1 * P.n1;
  const bool haveW = !(jvp && cached);
  P.NC = (haveW ? 1 : 0) + (jvp ? 1 : 0);
  // region 0: the coefficients (read by S1 only), then the point values (written
  // after S2), then the projected modes
  P.oV = haveW ? (size_t)fpc * 2 * nb : 0;
  const size_t coef = P.oV + (jvp ? (size_t)fpc * 2 * nb : 0), pts = (size_t)fpc * FSF_NP * P.nqf;
  size_t o = coef > pts ? coef : pts;
  const size_t modes = (size_t)fpc * 2 * nb;
  o = o > modes ? o : modes;
  // region 1, per face: the interpolation's stages, then the projection's
  const size_t interp = (size_t)2 * P.NC * M * (2 * P.npair + 3 * P.n1 * nq);
  const size_t proj = (size_t)FSF_NX * P.n1 * nq + FSF_NY * P.npair;
  P.per_face = interp > proj ? interp : proj;
  P.oS = o;
  o += (size_t)fpc * P.per_face;
  P.oT = o;                                            // L[n1][nq] dL[n1][nq] Le[2][n1] dLe[2][n1]
  o += (size_t)2 * P.n1 * nq + 4 * P.n1;
  P.total = o;
  return P;
}

// component d of a triple held in scalars (no run-time indexing of local arrays)
template <class T>
__device__ __forceinline__ T pick3(int d, T x0, T x1, T x2) {
  return d == 0 ? x0 : (d == 1 ? x1 : x2);
}

}  // namespace

template <class T, bool JVP>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 4 : 2)
    face_sf_kernel(MeshView<T> mv, Phys<T> ph, const T* __restrict__ W, const T* __restrict__ V,
                   T* __restrict__ slots, int* status, int fpc, const T* __restrict__ Pf, const T* __restrict__ l1g,
                   const int* __restrict__ qidx, int p, int nq, int total_degree, T m0, T m1, T m2) {
  using S = typename std::conditional<JVP, Dual<T>, T>::type;
  constexpr int D = 3, M = D + 2, PU = M * (1 + D);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  __shared__ unsigned short ptab[256];   // pair -> a0 | a1 << 8, a0-major
  const int nb = mv.nb, nm = mv.nm, nqf = mv.nqf, E = mv.E;
  const bool cached = JVP && Pf != nullptr;
  const FsfPlan P = fsf_plan(p, nq, nb, M, total_degree, JVP, cached, fpc);
  const int n1 = P.n1, NC = P.NC, npair = P.npair, n1s = n1 * n1;
  const bool haveW = !cached;
  const int nfaces = D * E, f0 = blockIdx.x * fpc, nloc = min(fpc, nfaces - f0);
  if (nloc <= 0) return;
  T* sW = sm;                      // [fpc][2][nb]  state (not with cached traces), until S1
  T* sV = sm + P.oV;               // [fpc][2][nb]  direction (JVP), until S1
  T* sP = sm;                      // [fpc][FSF_NP][nqf] point values times the face weight
  T* sS = sm + P.oS;               // [fpc][per_face]: contraction stages
  T* tab = sm + P.oT;
  const T* L = tab;                // L[a][b]
  const T* dL = tab + n1 * nq;     // dL[a][b] (reference derivative)
  const T* Le = dL + n1 * nq;      // Le[end][a], end 0 at -1, 1 at +1
  const T* dLe = Le + 2 * n1;
  for (int t = threadIdx.x; t < 2 * n1 * nq; t += blockDim.x) tab[t] = l1g[t];
  for (int t = threadIdx.x; t < 4 * n1; t += blockDim.x) tab[2 * n1 * nq + t] = l1g[2 * n1 * nq + nq + t];
  // first pair of a0: a0 n1 - a0 (a0 - 1) / 2 (P_p) or a0 n1 (Q_p)
  auto pair0 = [&](int a0) { return total_degree ? a0 * n1 - a0 * (a0 - 1) / 2 : a0 * n1; };
  for (int t = threadIdx.x; t < n1s; t += blockDim.x) {
    const int a0 = t / n1, a1 = t - a0 * n1;
    if (!total_degree || a0 + a1 <= p) ptab[pair0(a0) + a1] = (unsigned short)(a0 | a1 << 8);
  }
  // phase 0: the modal coefficients of both elements of every face
  for (int t = threadIdx.x; t < nloc * 2 * nb; t += blockDim.x) {
    const int fl = t / (2 * nb), r = t % (2 * nb), side = r / nb, j = r % nb;
    const int f = f0 + fl, k = f / E, e = f % E;
    const int el = side == 0 ? e : mv.nbr[(e * D + k) * 2 + 1];
    if (haveW) sW[t] = W[(size_t)el * nb + j];
    if (JVP) sV[t] = V[(size_t)el * nb + j];
  }
  __syncthreads();
  // S1: collapse the normal direction with the end values (L and L'); the pair
  // slowest, so that the lanes of a warp run sums of one length
  const int n_s1 = 2 * NC * M, s1sz = 2 * n_s1 * npair;
  for (int t = threadIdx.x; t < nloc * n_s1 * npair; t += blockDim.x) {
    const int pr = t / (nloc * n_s1);
    int r = t - pr * (nloc * n_s1);
    const int fl = r / n_s1;
    r -= fl * n_s1;
    const int row = r, v = r % M;
    r /= M;
    const int c = r % NC, side = r / NC;
    const int a0 = ptab[pr] & 255, a1 = ptab[pr] >> 8;
    const int k = (f0 + fl) / E, t0 = k == 0 ? 1 : 0, t1 = k == 2 ? 1 : 2;
    const int pv = v == 0 || v == M - 1 ? v : 1 + pick3(v - 1, k, t0, t1);   // the frame's variable v
    const int end = side == 0 ? 1 : 0;       // the element on side 0 meets the face at xi_k = +1
    const T* Ev = Le + end * n1;
    const T* dEv = dLe + end * n1;
    const T* fld = ((haveW && c == 0) ? sW : sV) + ((size_t)fl * 2 + side) * nb + pv * nm;
    T acc = T(0), dacc = T(0);
    const int sk = pick3(k, 1, n1, n1s), base = a0 * pick3(t0, 1, n1, n1s) + a1 * pick3(t1, 1, n1, n1s);
    const int nak = total_degree ? n1 - a0 - a1 : n1;
#pragma unroll 4
    for (int ak = 0; ak < nak; ++ak) {
      const T x = fld[qidx[base + ak * sk]];
      acc += x * Ev[ak];
      dacc += x * dEv[ak];
    }
    T* o = sS + (size_t)fl * P.per_face + (size_t)row * 2 * npair + pr;
    o[0] = acc;
    o[npair] = dacc;
  }
  __syncthreads();
  // S2: contract the second tangential direction: d0 = c0 L, d1 = c0 L', d2 = c1 L;
  // a0 slowest, as S1's pair
  const int n_s2 = 2 * NC * M * nq;
  for (int t = threadIdx.x; t < nloc * n_s2 * n1; t += blockDim.x) {
    const int a0 = t / (nloc * n_s2);
    int r = t - a0 * (nloc * n_s2);
    const int fl = r / n_s2;
    r -= fl * n_s2;
    const int b1 = r % nq, scv = r / nq;                            // scv = (side, c, v)
    const T* s1 = sS + (size_t)fl * P.per_face + (size_t)scv * 2 * npair + pair0(a0);
    const int na1 = total_degree ? n1 - a0 : n1;
    T d0 = T(0), d1 = T(0), d2 = T(0);
#pragma unroll 4
    for (int a1 = 0; a1 < na1; ++a1) {
      const T la = L[a1 * nq + b1], x = s1[a1];
      d0 += x * la;
      d1 += x * dL[a1 * nq + b1];
      d2 += s1[npair + a1] * la;
    }
    T* o = sS + (size_t)fl * P.per_face + s1sz + ((size_t)scv * 3 * n1 + a0) * nq + b1;
    o[0] = d0;
    o[(size_t)n1 * nq] = d1;
    o[(size_t)2 * n1 * nq] = d2;
  }
  __syncthreads();
  // phase 1: traces at the face points from the S2 stage, pointwise physics
  // (with cached traces a JVP takes the state's from the cache)
  for (int t = threadIdx.x; t < nloc * nqf; t += blockDim.x) {
    const int fl = t / nqf, q = t % nqf, b0 = q % nq, b1 = q / nq;
    const int f = f0 + fl, k = f / E, t0 = k == 0 ? 1 : 0, t1 = k == 2 ? 1 : 2;
    const T mk = pick3(k, m0, m1, m2), mt0 = pick3(t0, m0, m1, m2), mt1 = pick3(t1, m0, m1, m2);
    const T* s2 = sS + (size_t)fl * P.per_face + s1sz;
    S uS[2][M], gS[2][M][D];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
#pragma unroll
      for (int v = 0; v < M; ++v) {
        T val[2] = {T(0), T(0)}, gn[2] = {T(0), T(0)}, g0[2] = {T(0), T(0)}, g1[2] = {T(0), T(0)};
        const T* d = s2 + ((size_t)(side * NC * M + v) * 3) * n1 * nq + b1;   // [ty][a0][b1]
        const size_t dc = (size_t)M * 3 * n1 * nq;                            // to the second field
        for (int a0 = 0; a0 < n1; ++a0) {
          const T la = L[a0 * nq + b0], da = dL[a0 * nq + b0];
#pragma unroll
          for (int c = 0; c < (JVP ? 2 : 1); ++c) {
            if (c >= NC) continue;
            const T* x = d + c * dc + (size_t)a0 * nq;
            const T d0 = x[0], d1 = x[(size_t)n1 * nq], d2 = x[(size_t)2 * n1 * nq];
            val[c] += d0 * la;
            g0[c] += d0 * da;
            g1[c] += d1 * la;
            gn[c] += d2 * la;
          }
        }
#pragma unroll
        for (int c = 0; c < (JVP ? 2 : 1); ++c) {
          gn[c] *= mk;
          g0[c] *= mt0;
          g1[c] *= mt1;
        }
        if constexpr (JVP) {
          if (cached) {
            const int pv = v == 0 || v == M - 1 ? v : 1 + pick3(v - 1, k, t0, t1);
            const T* cc = Pf + ((size_t)(f0 + fl) * nqf + q) * 2 * PU + side * PU;
            uS[side][v] = S(cc[pv], val[0]);
            gS[side][v][0] = S(cc[M + pv * D + k], gn[0]);
            gS[side][v][1] = S(cc[M + pv * D + t0], g0[0]);
            gS[side][v][2] = S(cc[M + pv * D + t1], g1[0]);
          } else {
            uS[side][v] = S(val[0], val[1]);
            gS[side][v][0] = S(gn[0], gn[1]);
            gS[side][v][1] = S(g0[0], g0[1]);
            gS[side][v][2] = S(g1[0], g1[1]);
          }
        } else {
          uS[side][v] = val[0];
          gS[side][v][0] = gn[0];
          gS[side][v][1] = g0[0];
          gS[side][v][2] = g1[0];
        }
      }
    }
    if (!physical<D>(uS[0], ph.gm1) || !physical<D>(uS[1], ph.gm1)) atomicOr(status, ST_NONPHYSICAL);
    S fp[M], mL[D], eL[D], mR[D], eR[D];
    face_point_core<D, 0, S, T>(uS[0], gS[0], uS[1], gS[1], ph, fp, mL, eL, mR, eR);
    const T fw = mv.fw[(size_t)k * nqf + q];
    T* o = sP + (size_t)fl * FSF_NP * nqf + q;
#define PART(x) (JVP ? tan_part(x) : val(x))
#pragma unroll
    for (int v = 0; v < M; ++v) o[(size_t)v * nqf] = fw * PART(fp[v]);
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const T ml = fw * PART(mL[j]), mr = fw * PART(mR[j]), el = fw * PART(eL[j]), er = fw * PART(eR[j]);
      // normal column of K(uL) jump + K(uR) jump (twice the halves)
      o[(size_t)(5 + j) * nqf] = (j == 0 ? T(8) / T(3) : T(2)) * (ml + mr);
      if (j == 0) o[(size_t)8 * nqf] = T(2) * (el + er);
      o[(size_t)(9 + j) * nqf] = ml;
      o[(size_t)(12 + j) * nqf] = el;
      o[(size_t)(15 + j) * nqf] = mr;
      o[(size_t)(18 + j) * nqf] = er;
    }
#undef PART
  }
  __syncthreads();
  // X: sums over b0.  Arrays 0-4 the flux, 5-8 the lifting integrand, then per
  // side m_n, m_t0, m_t1, e_n, e_t1 with L and m_t0, m_n, e_t0 with L'
  // (a thread takes the arrays of one kind together: independent sums of one
  // test function, which keep the FP64 pipe fed from few warps)
  const int xrow = n1 * nq, xsz = FSF_NX * xrow;
  for (int t = threadIdx.x; t < nloc * 6 * xrow; t += blockDim.x) {
    const int g = t / (nloc * xrow);                                // flux, lifting, then (side, L / L')
    int r = t - g * (nloc * xrow);
    const int fl = r / xrow;
    r -= fl * xrow;
    const int b1 = r % nq, a0 = r / nq, side = g >= 4 ? 1 : 0;
    const T* src = sP + (size_t)fl * FSF_NP * nqf + (size_t)nq * b1;
    const bool der = g == 3 || g == 5;
    const T* La = (der ? dL : L) + a0 * nq;
    int c0, c1, c2, c3, c4, n, to;                                  // components, how many, first array
    if (g == 0) {
      c0 = 0, c1 = 1, c2 = 2, c3 = 3, c4 = 4, n = 5, to = 0;
    } else if (g == 1) {
      c0 = 5, c1 = 6, c2 = 7, c3 = 8, c4 = 8, n = 4, to = 5;
    } else {
      const int b = 9 + 6 * side;
      if (!der) {
        c0 = b, c1 = b + 1, c2 = b + 2, c3 = b + 3, c4 = b + 5, n = 5, to = 9 + 8 * side;
      } else {
        c0 = b + 1, c1 = b, c2 = b + 4, c3 = b + 4, c4 = b + 4, n = 3, to = 14 + 8 * side;
      }
    }
    const T *p0 = src + (size_t)c0 * nqf, *p1 = src + (size_t)c1 * nqf, *p2 = src + (size_t)c2 * nqf,
            *p3 = src + (size_t)c3 * nqf, *p4 = src + (size_t)c4 * nqf;
    T s0 = T(0), s1 = T(0), s2 = T(0), s3 = T(0), s4 = T(0);
    if (n == 3) {
#pragma unroll 2
      for (int b0 = 0; b0 < nq; ++b0) {
        const T la = La[b0];
        s0 += p0[b0] * la;
        s1 += p1[b0] * la;
        s2 += p2[b0] * la;
      }
    } else if (n == 4) {
      for (int b0 = 0; b0 < nq; ++b0) {
        const T la = La[b0];
        s0 += p0[b0] * la;
        s1 += p1[b0] * la;
        s2 += p2[b0] * la;
        s3 += p3[b0] * la;
      }
    } else {
      for (int b0 = 0; b0 < nq; ++b0) {
        const T la = La[b0];
        s0 += p0[b0] * la;
        s1 += p1[b0] * la;
        s2 += p2[b0] * la;
        s3 += p3[b0] * la;
        s4 += p4[b0] * la;
      }
    }
    T* o = sS + (size_t)fl * P.per_face + (size_t)to * xrow + a0 * nq + b1;
    o[0] = s0;
    o[xrow] = s1;
    o[2 * xrow] = s2;
    if (n > 3) o[3 * xrow] = s3;
    if (n > 4) o[4 * xrow] = s4;
  }
  __syncthreads();
  // Y: sums over b1, per pair.  Arrays 0-4 the flux, then per side the
  // dual-consistency terms' value part (n, t0, t1, E) and normal derivative
  // part, then the lifting (n, t0, t1, E)
  for (int t = threadIdx.x; t < nloc * 6 * npair; t += blockDim.x) {
    const int g = t / (nloc * npair);                               // flux, lifting, then (side, value / normal part)
    int r = t - g * (nloc * npair);
    const int fl = r / npair, pr = r - fl * npair;
    const int a0 = ptab[pr] & 255, a1 = ptab[pr] >> 8, side = g >= 4 ? 1 : 0;
    const int k = (f0 + fl) / E, t0 = k == 0 ? 1 : 0, t1 = k == 2 ? 1 : 2;
    const T mk = pick3(k, m0, m1, m2);
    const T* X = sS + (size_t)fl * P.per_face + a0 * nq;       // array i at + i * xrow
    T* o = sS + (size_t)fl * P.per_face + xsz + pr;            // array i at + i * npair
    const T* L1 = L + a1 * nq;
    const T* D1 = dL + a1 * nq;
    if (g == 0) {
      T s[M] = {};
      for (int b = 0; b < nq; ++b)
#pragma unroll
        for (int v = 0; v < M; ++v) s[v] += X[(size_t)v * xrow + b] * L1[b];
#pragma unroll
      for (int v = 0; v < M; ++v) o[(size_t)v * npair] = s[v];
    } else if (g == 1) {
      T s[M - 1] = {};
      for (int b = 0; b < nq; ++b)
#pragma unroll
        for (int v = 0; v < M - 1; ++v) s[v] += X[(size_t)(5 + v) * xrow + b] * L1[b];
      const int n = total_degree ? n1 - a0 - a1 : n1;          // C_a = n^2 / 2
      const T sc = ph.eta * mk * (T(0.125) * (T)(n * n));
#pragma unroll
      for (int v = 0; v < M - 1; ++v) o[(size_t)(M + 16 + v) * npair] = sc * s[v];
    } else {
      const T* xs = X + (size_t)(9 + 8 * side) * xrow;         // m_n m_t0 m_t1 e_n e_t1 | m_t0' m_n' e_t0'
      T* os = o + (size_t)(M + 8 * side) * npair;
      if (g == 3 || g == 5) {
        T s[4] = {};
        for (int b = 0; b < nq; ++b)
#pragma unroll
          for (int v = 0; v < 4; ++v) s[v] += xs[(size_t)v * xrow + b] * L1[b];
        os[(size_t)4 * npair] = -mk * (T(4) / T(3)) * s[0];
#pragma unroll
        for (int v = 1; v < 4; ++v) os[(size_t)(4 + v) * npair] = -mk * s[v];
      } else {
        // rows n, E: m_t0 d_t0 + m_t1 d_t1, e_t0 d_t0 + e_t1 d_t1; t0, t1: -2/3 m_n d_t0, d_t1
        T s[6] = {};
        for (int b = 0; b < nq; ++b) {
          const T l = L1[b], dl = D1[b];
          s[0] += xs[(size_t)5 * xrow + b] * l;
          s[1] += xs[(size_t)6 * xrow + b] * l;
          s[2] += xs[(size_t)7 * xrow + b] * l;
          s[3] += xs[(size_t)2 * xrow + b] * dl;
          s[4] += xs[b] * dl;
          s[5] += xs[(size_t)4 * xrow + b] * dl;
        }
        const T mt0 = pick3(t0, m0, m1, m2), mt1 = pick3(t1, m0, m1, m2);
        os[0] = -(mt0 * s[0] + mt1 * s[3]);
        os[npair] = (T(2) / T(3)) * mt0 * s[1];
        os[(size_t)2 * npair] = (T(2) / T(3)) * mt1 * s[4];
        os[(size_t)3 * npair] = -(mt0 * s[2] + mt1 * s[5]);
      }
    }
  }
  __syncthreads();
  // the normal direction's end values: modes of both elements, in shared memory
  const int osz = 2 * M * npair;
  for (int t = threadIdx.x; t < nloc * osz; t += blockDim.x) {
    const int fl = t / osz;
    int r = t - fl * osz;
    const int pr = r % npair;
    r /= npair;
    const int v = r % M, side = r / M;
    const int a0 = ptab[pr] & 255, a1 = ptab[pr] >> 8;
    const int k = (f0 + fl) / E, t0 = k == 0 ? 1 : 0, t1 = k == 2 ? 1 : 2;
    const int pv = v == 0 || v == M - 1 ? v : 1 + pick3(v - 1, k, t0, t1);
    const int end = side == 0 ? 1 : 0;
    const T* Y = sS + (size_t)fl * P.per_face + xsz + pr;
    const T yf = v > 0 ? Y[(size_t)v * npair] + Y[(size_t)(M + 16 + v - 1) * npair] : Y[0];
    T ya = side == 0 ? yf : -yf, yn = T(0);
    if (v > 0) {
      ya += Y[(size_t)(M + 8 * side + v - 1) * npair];
      yn = Y[(size_t)(M + 8 * side + 4 + v - 1) * npair];
    }
    const int sk = pick3(k, 1, n1, n1s), base = a0 * pick3(t0, 1, n1, n1s) + a1 * pick3(t1, 1, n1, n1s);
    const int nak = total_degree ? n1 - a0 - a1 : n1;
    T* o = sm + ((size_t)fl * 2 + side) * nb + pv * nm;      // over the point values (dead since X)
    for (int ak = 0; ak < nak; ++ak) o[qidx[base + ak * sk]] = Le[end * n1 + ak] * ya + dLe[end * n1 + ak] * yn;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nloc * 2 * nb; t += blockDim.x) {
    const int fl = t / (2 * nb), r = t - fl * 2 * nb, f = f0 + fl, k = f / E, e = f % E;
    slots[((size_t)e * D + k) * 2 * nb + r] = sm[t];
  }
}

template <class T, bool JVP>
static cudaError_t run_face_sf(const Mesh& Ms, const T* W, const T* V, T* slots, const T* Pf, cudaStream_t st) {
  const bool cached = JVP && Pf != nullptr;
  const int pdeg = Ms.desc.space == DG_SPACE_Q ? 0 : 1;
  if (Ms.p + 1 > 15) return cudaErrorNotSupported;   // the pair table
  int threads = 128;
  int fpc = items_per_cta(3L * Ms.E, std::max(1, 128 / Ms.nqf), Ms.nqf, 128, &threads);
  int dev = 0, smax = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  auto bytes = [&](int f) { return fsf_plan(Ms.p, Ms.nq1d, Ms.nb, Ms.m, pdeg, JVP, cached, f).total * sizeof(T); };
  size_t smem = bytes(fpc);
  while (smem > (size_t)smax - 1536 && fpc > 1) smem = bytes(--fpc);
  if (smem > (size_t)smax - 1536) return cudaErrorNotSupported;
  if (smem > 48 * 1024) {
    cudaError_t e = allow_max_smem(face_sf_kernel<T, JVP>);
    if (e != cudaSuccess) return e;
  }
  const T* l1 = std::is_same<T, double>::value ? (const T*)Ms.t64.l1d : (const T*)Ms.t32.l1d;
  const T m0 = (T)(2.0 / Ms.h[0]), m1 = (T)(2.0 / Ms.h[1]), m2 = (T)(2.0 / Ms.h[2]);
  const int nfaces = 3 * Ms.E;
  note_launch();
  face_sf_kernel<T, JVP><<<(nfaces + fpc - 1) / fpc, threads, smem, st>>>(Ms.view<T>(), Ms.phys_t<T>(), W, V, slots,
                                                                     Ms.status, fpc, cached ? Pf : nullptr, l1,
                                                                     Ms.qidx, Ms.p, Ms.nq1d, pdeg, m0, m1, m2);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_face_sf(const Mesh& M, const T* W, const T* V, T* slots, bool jvp, const T* Pf,
                           cudaStream_t st) {
  if (M.kind != DG_MESH_STRUCTURED || M.d != 3 || !M.qidx) return cudaErrorNotSupported;
  return jvp ? run_face_sf<T, true>(M, W, V, slots, Pf, st) : run_face_sf<T, false>(M, W, V, slots, nullptr, st);
}
template cudaError_t launch_face_sf<double>(const Mesh&, const double*, const double*, double*, bool, const double*,
                                            cudaStream_t);
template cudaError_t launch_face_sf<float>(const Mesh&, const float*, const float*, float*, bool, const float*,
                                           cudaStream_t);

}  // namespace dgk
