// Face term of the FP32 Jacobian-vector product on 3-D P_p meshes (Sec. 3.1 eq.
// dg_ns face terms, eq. visc_flux, eq. re) by sum factorisation, p = 1 .. 6 with
// p + 2 points per direction: the stages, the face's frame and the treatment
// of the flux, of the lifting and of the dual-consistency tensors are those of
// face_sf_kernel (dg_face_sf.cu).  In FP32 the limit is not the arithmetic but
// instruction issue (face_kernel's dense contractions: 800 k operations per
// element at p = 4; factorised 130 k), so, as in dg_vol32.cu, a thread contracts
// a whole line at once with unrolled loops and constant-bank tables:
//   S1  (side, v, pair): the normal direction's end values
//   S2  (side, v, a0): all b1 of d0, d1, d2
//   S3  (side, v, b1): all b0 of u and its three derivatives, to shared memory
//   pt  a thread per point: the linearised physics
//   X   (array, b1): all a0;   Y  (array, a0): all a1;   then the modes
// 16^3 elements, p = 4 with cached traces: 231 -> 86 us; 16^3, p = 6: 769 -> 175 us.
#include "dg_sf32.cuh"

namespace dgk {

namespace {

constexpr int F32_THREADS = 128;

template <int N1, bool CACHED>
struct F32 {
  static constexpr int NQ = N1 + 1, NL = NQ * NQ, NP = sf32_pairs(N1), NM = sf32_modes(N1), M = 5, NB = M * NM;
  static constexpr int NC = CACHED ? 1 : 2;
  static constexpr int FPC = F32_THREADS / NL > 0 ? F32_THREADS / NL : 1;
  static constexpr int mx(int a, int b) { return a > b ? a : b; }
  // region 0: coefficients, then point values, then the projected modes;
  // region 1: S1 and S2, then X and Y; region 2: the traces at the points
  static constexpr int n0 = mx(mx(2 * NC * NB, 21 * NL), 2 * NB);
  static constexpr int nS1 = 2 * NC * M * 2 * NP, nS2 = 2 * NC * M * 3 * N1 * NQ;
  static constexpr int nX = 25 * N1 * NQ, nY = 25 * NP, n1 = mx(nS1 + nS2, nX + nY);
  static constexpr int n2 = 2 * NC * M * 4 * NL;
  static constexpr int o1 = FPC * n0, o2 = o1 + FPC * n1, oI = o2 + FPC * n2;
  static constexpr size_t bytes = sizeof(float) * oI + sizeof(int) * 3 * FPC +
                                  sizeof(unsigned short) * (3 * NM + 2 * NP + 2);
  static constexpr int nld = (FPC * 2 * NB + F32_THREADS - 1) / F32_THREADS;   // coefficient loads of a thread
};

template <int N1, bool CACHED>
__global__ void __launch_bounds__(F32_THREADS, 4) face32_kernel(const __grid_constant__ Sf32Tab<N1> tb, Phys<float> ph,
                                                                const int* __restrict__ nbr,
                                                                const int* __restrict__ qidx, int E,
                                                                const float* __restrict__ W,
                                                                const float* __restrict__ V,
                                                                float* __restrict__ slots, int* status,
                                                                const float4* __restrict__ Pf) {
  using C = F32<N1, CACHED>;
  using S = Dual<float>;
  constexpr int NQ = C::NQ, NL = C::NL, NP = C::NP, NM = C::NM, M = C::M, NB = C::NB, NC = C::NC, FPC = C::FPC;
  constexpr int XR = N1 * NQ;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* sm = reinterpret_cast<float*>(smem_raw);
  int* fk = reinterpret_cast<int*>(sm + C::oI);                           // per face: direction, elements L and R
  unsigned short* pos = reinterpret_cast<unsigned short*>(fk + 3 * FPC);  // [k][mode]: sf32_pos
  unsigned short* ptab = pos + 3 * NM;                                    // pair -> a0 | a1 << 8
  unsigned short* poff = ptab + NP;                                       // pair -> sf32_run
  const int tid = threadIdx.x, f0 = blockIdx.x * FPC, nf = min(FPC, 3 * E - f0);
  if (tid < FPC) {
    const int f = min(f0 + tid, 3 * E - 1), k = f / E, e = f - k * E;
    fk[3 * tid] = k;
    fk[3 * tid + 1] = e;
    fk[3 * tid + 2] = nbr[(e * 3 + k) * 2 + 1];
  }
  for (int t = tid; t < N1 * N1 * N1; t += F32_THREADS) {
    const int i = qidx[t];
    if (i >= 0)
#pragma unroll
      for (int k = 0; k < 3; ++k) pos[k * NM + i] = (unsigned short)sf32_pos<N1>(t, k);
  }
  for (int t = tid; t < N1 * N1; t += F32_THREADS) {
    const int a0 = t / N1, a1 = t - a0 * N1;
    if (a0 + a1 < N1) {
      ptab[sf32_pair0(N1, a0) + a1] = (unsigned short)(a0 | a1 << 8);
      poff[sf32_pair0(N1, a0) + a1] = (unsigned short)sf32_run(N1, a0, a1);
    }
  }
  __syncthreads();
  // (the loops below run over all FPC faces, also where the last CTA has fewer:
  // the index divisions are then by constants)
  // coefficients of both elements of every face, [fl][side][c][v][position],
  // all of a thread's loads in flight together
  {
    float xw[CACHED ? 1 : C::nld], xv[C::nld];
#pragma unroll
    for (int u = 0; u < C::nld; ++u) {
      const int t = min(tid + u * F32_THREADS, FPC * 2 * NB - 1);
      const int fs = t / NB, j = t - fs * NB, el = fk[3 * (fs >> 1) + 1 + (fs & 1)];
      xv[u] = V[(size_t)el * NB + j];
      if constexpr (!CACHED) xw[u] = W[(size_t)el * NB + j];
    }
#pragma unroll
    for (int u = 0; u < C::nld; ++u) {
      const int t = min(tid + u * F32_THREADS, FPC * 2 * NB - 1);
      const int fs = t / NB, j = t - fs * NB, fl = fs >> 1, side = fs & 1, v = j / NM, i = j - v * NM;
      float* o = sm + fl * C::n0 + side * NC * NB + v * NM + pos[fk[3 * fl] * NM + i];
      if constexpr (!CACHED) o[0] = xw[u];
      o[(NC - 1) * NB] = xv[u];
    }
  }
  __syncthreads();
  // S1 (the pair slowest)
  for (int t = tid; t < NP * FPC * 2 * NC * M; t += F32_THREADS) {
    const int pr = t / (FPC * 2 * NC * M), r = t - pr * (FPC * 2 * NC * M), fl = r / (2 * NC * M);
    const int scv = r - fl * (2 * NC * M), v = scv % M, sc = scv / M, side = sc / NC;
    const int na = N1 - (ptab[pr] & 255) - (ptab[pr] >> 8);
    const int k = fk[3 * fl], t0 = k == 0 ? 1 : 0, t1 = k == 2 ? 1 : 2;
    const int pv = v == 0 || v == M - 1 ? v : v == 1 ? 1 + k : v == 2 ? 1 + t0 : 1 + t1;
    const float* w = sm + fl * C::n0 + sc * NB + pv * NM + poff[pr];
    // even and odd ak apart: the values at -1 differ in the odd ones' sign
    float ev = 0.f, od = 0.f, dev = 0.f, dod = 0.f;
#pragma unroll
    for (int ak = 0; ak < N1; ++ak) {
      if (ak < na) {
        const float x = w[ak];
        if (ak % 2 == 0) {
          ev = fmaf(x, tb.Le[ak], ev);
          dev = fmaf(x, tb.dLe[ak], dev);
        } else {
          od = fmaf(x, tb.Le[ak], od);
          dod = fmaf(x, tb.dLe[ak], dod);
        }
      }
    }
    // side 0 meets the face at xi_k = +1, side 1 at -1
    float* o = sm + C::o1 + fl * C::n1 + scv * 2 * NP + pr;
    o[0] = side == 0 ? ev + od : ev - od;
    o[NP] = side == 0 ? dev + dod : dod - dev;
  }
  __syncthreads();
  // S2 (a0 slowest)
  for (int t = tid; t < N1 * FPC * 2 * NC * M; t += F32_THREADS) {
    const int a0 = t / (FPC * 2 * NC * M), r = t - a0 * (FPC * 2 * NC * M), fl = r / (2 * NC * M);
    const int scv = r - fl * (2 * NC * M), na = N1 - a0;
    const float* c = sm + C::o1 + fl * C::n1 + scv * 2 * NP + sf32_pair0(N1, a0);
    float d0[NQ], d1[NQ], d2[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) d0[q] = d1[q] = d2[q] = 0.f;
#pragma unroll
    for (int a1 = 0; a1 < N1; ++a1) {
      if (a1 < na) {
        const float x = c[a1], y = c[NP + a1];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          d0[q] = fmaf(x, tb.L[a1][q], d0[q]);
          d1[q] = fmaf(x, tb.dL[a1][q], d1[q]);
          d2[q] = fmaf(y, tb.L[a1][q], d2[q]);
        }
      }
    }
    float* o = sm + C::o1 + fl * C::n1 + C::nS1 + (scv * 3 * N1 + a0) * NQ;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      o[q] = d0[q];
      o[XR + q] = d1[q];
      o[2 * XR + q] = d2[q];
    }
  }
  __syncthreads();
  // S3: u, d/dn, d/dt0, d/dt1 at (b0, b1), point index b1 + NQ b0
  for (int t = tid; t < FPC * 2 * NC * M * NQ; t += F32_THREADS) {
    const int fscv = t / NQ, b1 = t - fscv * NQ, fl = fscv / (2 * NC * M), scv = fscv - fl * (2 * NC * M);
    const int k = fk[3 * fl];
    const float mk = k == 0 ? tb.met[0] : k == 1 ? tb.met[1] : tb.met[2];
    const float mt0 = k == 0 ? tb.met[1] : tb.met[0], mt1 = k == 2 ? tb.met[1] : tb.met[2];
    const float* d = sm + C::o1 + fl * C::n1 + C::nS1 + scv * 3 * XR + b1;
    float u[NQ], g0[NQ], g1[NQ], gn[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) u[q] = g0[q] = g1[q] = gn[q] = 0.f;
#pragma unroll
    for (int a = 0; a < N1; ++a) {
      const float x = d[a * NQ], y = d[XR + a * NQ], z = d[2 * XR + a * NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        u[q] = fmaf(x, tb.L[a][q], u[q]);
        g0[q] = fmaf(x, tb.dL[a][q], g0[q]);
        g1[q] = fmaf(y, tb.L[a][q], g1[q]);
        gn[q] = fmaf(z, tb.L[a][q], gn[q]);
      }
    }
    float* o = sm + C::o2 + fl * C::n2 + scv * 4 * NL + b1;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      o[q * NQ] = u[q];
      o[NL + q * NQ] = mk * gn[q];
      o[2 * NL + q * NQ] = mt0 * g0[q];
      o[3 * NL + q * NQ] = mt1 * g1[q];
    }
  }
  __syncthreads();
  // points
  if (tid < nf * NL) {
    const int fl = tid / NL, q = tid - fl * NL, f = f0 + fl, k = fk[3 * fl];
    const float* G = sm + C::o2 + fl * C::n2 + q;
    S u[2][M], g[2][M][3];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      if constexpr (CACHED) {
        float c[20];
#pragma unroll
        for (int w = 0; w < 5; ++w) {
          const float4 x = __ldg(Pf + sf32_face_word(f, side, w, q, NL));
          c[4 * w] = x.x, c[4 * w + 1] = x.y, c[4 * w + 2] = x.z, c[4 * w + 3] = x.w;
        }
#pragma unroll
        for (int v = 0; v < M; ++v) {
          const float* t = G + (side * M + v) * 4 * NL;
          u[side][v] = S(c[v], t[0]);
#pragma unroll
          for (int j = 0; j < 3; ++j) g[side][v][j] = S(c[5 + 3 * v + j], t[(1 + j) * NL]);
        }
      } else {
#pragma unroll
        for (int v = 0; v < M; ++v) {
          const float* s = G + ((side * 2) * M + v) * 4 * NL;
          const float* t = G + ((side * 2 + 1) * M + v) * 4 * NL;
          u[side][v] = S(s[0], t[0]);
#pragma unroll
          for (int j = 0; j < 3; ++j) g[side][v][j] = S(s[(1 + j) * NL], t[(1 + j) * NL]);
        }
      }
    }
    if (!physical<3>(u[0], ph.gm1) || !physical<3>(u[1], ph.gm1)) atomicOr(status, ST_NONPHYSICAL);
    S fp[M], mL[3], eL[3], mR[3], eR[3];
    face_point_core<3, 0, S, float>(u[0], g[0], u[1], g[1], ph, fp, mL, eL, mR, eR);
    const float fj = k == 0 ? tb.faceJ[0] : k == 1 ? tb.faceJ[1] : tb.faceJ[2];
    float wb0 = 0.f, wb1 = 0.f;
#pragma unroll
    for (int b = 0; b < NQ; ++b) {
      if (q / NQ == b) wb0 = tb.w[b];
      if (q % NQ == b) wb1 = tb.w[b];
    }
    const float fw = fj * wb0 * wb1;
    float* o = sm + fl * C::n0 + q;
#pragma unroll
    for (int v = 0; v < M; ++v) o[v * NL] = fw * fp[v].d;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float ml = fw * mL[j].d, mr = fw * mR[j].d, el = fw * eL[j].d, er = fw * eR[j].d;
      // normal column of K(uL) jump + K(uR) jump (twice the halves)
      o[(5 + j) * NL] = (j == 0 ? 8.f / 3.f : 2.f) * (ml + mr);
      if (j == 0) o[8 * NL] = 2.f * (el + er);
      o[(9 + j) * NL] = ml;
      o[(12 + j) * NL] = el;
      o[(15 + j) * NL] = mr;
      o[(18 + j) * NL] = er;
    }
  }
  __syncthreads();
  // X: arrays 0-4 the flux, 5-8 the lifting integrand, then per side m_n, m_t0,
  // m_t1, e_n, e_t1 with L, then per side m_t0, m_n, e_t0 with L' (the array
  // slowest: warps of one kind)
  for (int t = tid; t < 25 * FPC * NQ; t += F32_THREADS) {
    const int arr = t / (FPC * NQ), r = t - arr * (FPC * NQ), fl = r / NQ, b1 = r - fl * NQ;
    int comp = arr;
    if (arr >= 19) {
      const int w = arr - 19, side = w >= 3 ? 1 : 0, i = w - 3 * side;
      comp = 9 + 6 * side + (i == 0 ? 1 : i == 1 ? 0 : 4);
    } else if (arr >= 9) {
      const int w = arr - 9, side = w >= 5 ? 1 : 0, i = w - 5 * side;
      comp = 9 + 6 * side + (i < 4 ? i : 5);
    }
    const float* s = sm + fl * C::n0 + comp * NL + b1;
    float* d = sm + C::o1 + fl * C::n1 + arr * XR + b1;
    float x[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) x[q] = s[q * NQ];
    if (arr < 19) {
#pragma unroll
      for (int a = 0; a < N1; ++a) {
        float o = 0.f;
#pragma unroll
        for (int q = 0; q < NQ; ++q) o = fmaf(x[q], tb.L[a][q], o);
        d[a * NQ] = o;
      }
    } else {
#pragma unroll
      for (int a = 0; a < N1; ++a) {
        float o = 0.f;
#pragma unroll
        for (int q = 0; q < NQ; ++q) o = fmaf(x[q], tb.dL[a][q], o);
        d[a * NQ] = o;
      }
    }
  }
  __syncthreads();
  // Y (the kind of array, then a0 slowest): arrays 0-4 the flux with the lifting, 5-8 and
  // 9-12 the sides' dual terms (n, t0, t1, E), 13-16 and 17-20 their
  // normal-derivative parts
  for (int t = tid; t < N1 * 21 * FPC; t += F32_THREADS) {
    constexpr int K1 = 5 * N1 * FPC, K2 = 8 * N1 * FPC;
    const int kind = t < K1 ? 0 : t < K1 + K2 ? 1 : 2, r0 = kind == 0 ? t : kind == 1 ? t - K1 : t - K1 - K2;
    const int nk = kind == 0 ? 5 : 8, a0 = kind == 0 ? r0 / (5 * FPC) : r0 / (8 * FPC);
    const int r = r0 - a0 * nk * FPC, ai = r / FPC, fl = r - ai * FPC, na = N1 - a0;
    const int arr = kind == 0 ? ai : kind == 1 ? 5 + ai : 13 + ai;
    const int k = fk[3 * fl];
    const float mk = k == 0 ? tb.met[0] : k == 1 ? tb.met[1] : tb.met[2];
    const float mt0 = k == 0 ? tb.met[1] : tb.met[0], mt1 = k == 2 ? tb.met[1] : tb.met[2];
    const float* X = sm + C::o1 + fl * C::n1 + a0 * NQ;
    float* o = sm + C::o1 + fl * C::n1 + C::nX + arr * NP + sf32_pair0(N1, a0);
    float xa[NQ], xb[NQ];
    if (kind == 0) {
      const float fb = ph.eta * mk * 0.125f;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        xa[q] = X[arr * XR + q];
        xb[q] = arr > 0 ? fb * X[(4 + arr) * XR + q] : 0.f;
      }
#pragma unroll
      for (int a1 = 0; a1 < N1; ++a1) {
        if (a1 < na) {
          float s = 0.f, d = 0.f;
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            s = fmaf(xa[q], tb.L[a1][q], s);
            d = fmaf(xb[q], tb.L[a1][q], d);
          }
          const float n = (float)(na - a1);            // C_a = n^2 / 2, n values of ak
          o[a1] = fmaf(n * n, d, s);
        }
      }
    } else if (kind == 1) {
      // rows n, E: m_t0 d_t0 + m_t1 d_t1, e_t0 d_t0 + e_t1 d_t1; t0, t1: -2/3 m_n d_t0, d_t1
      const int side = arr >= 9 ? 1 : 0, w = arr - 5 - 4 * side;
      const int ia = 19 + 3 * side + (w == 0 ? 0 : w == 3 ? 2 : 1), ib = 9 + 5 * side + (w == 0 ? 2 : w == 3 ? 4 : 0);
      const float sc = w == 1 || w == 2 ? 2.f / 3.f : -1.f, fa = w == 2 ? 0.f : sc * mt0, fb = w == 1 ? 0.f : sc * mt1;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        xa[q] = fa * X[ia * XR + q];
        xb[q] = fb * X[ib * XR + q];
      }
#pragma unroll
      for (int a1 = 0; a1 < N1; ++a1) {
        if (a1 < na) {
          float s = 0.f;
#pragma unroll
          for (int q = 0; q < NQ; ++q) s = fmaf(xa[q], tb.L[a1][q], fmaf(xb[q], tb.dL[a1][q], s));
          o[a1] = s;
        }
      }
    } else {
      const int side = arr >= 17 ? 1 : 0, w = arr - 13 - 4 * side;
      const float fa = -mk * (w == 0 ? 4.f / 3.f : 1.f);
#pragma unroll
      for (int q = 0; q < NQ; ++q) xa[q] = fa * X[(9 + 5 * side + w) * XR + q];
#pragma unroll
      for (int a1 = 0; a1 < N1; ++a1) {
        if (a1 < na) {
          float s = 0.f;
#pragma unroll
          for (int q = 0; q < NQ; ++q) s = fmaf(xa[q], tb.L[a1][q], s);
          o[a1] = s;
        }
      }
    }
  }
  __syncthreads();
  // the normal direction's end values: modes of both elements, in shared memory
  for (int t = tid; t < NP * FPC * 2 * M; t += F32_THREADS) {
    const int pr = t / (FPC * 2 * M), r = t - pr * (FPC * 2 * M), fl = r / (2 * M), sv = r - fl * (2 * M);
    const int side = sv / M, v = sv - side * M;
    const int na = N1 - (ptab[pr] & 255) - (ptab[pr] >> 8);
    const int k = fk[3 * fl], t0 = k == 0 ? 1 : 0, t1 = k == 2 ? 1 : 2;
    const int pv = v == 0 || v == M - 1 ? v : v == 1 ? 1 + k : v == 2 ? 1 + t0 : 1 + t1;
    const float* y = sm + C::o1 + fl * C::n1 + C::nX + pr;
    float ya = side == 0 ? y[v * NP] : -y[v * NP], yn = 0.f;
    if (v > 0) {
      ya += y[(5 + 4 * side + v - 1) * NP];
      yn = y[(13 + 4 * side + v - 1) * NP];
    }
    const float sg = side == 0 ? 1.f : -1.f;         // parity of the end values at -1
    float* o = sm + fl * C::n0 + side * NB + pv * NM + poff[pr];
#pragma unroll
    for (int ak = 0; ak < N1; ++ak)
      if (ak < na) {
        const float x = ak % 2 ? fmaf(sg * tb.Le[ak], ya, tb.dLe[ak] * yn) : fmaf(tb.Le[ak], ya, sg * tb.dLe[ak] * yn);
        o[ak] = x;
      }
  }
  __syncthreads();
  for (int t = tid; t < nf * 2 * NB; t += F32_THREADS) {
    const int fl = t / (2 * NB), r = t - fl * 2 * NB, k = fk[3 * fl], e = fk[3 * fl + 1];
    const int sv = r / NM;
    slots[((size_t)e * 3 + k) * 2 * NB + r] = sm[fl * C::n0 + sv * NM + pos[k * NM + r - sv * NM]];
  }
}

template <int N1, bool CACHED>
cudaError_t run_face32(const Mesh& Ms, const float* W, const float* V, float* slots, const float4* Pf, cudaStream_t st) {
  using C = F32<N1, CACHED>;
  cudaError_t e = allow_max_smem(face32_kernel<N1, CACHED>);
  if (e != cudaSuccess) return e;
  note_launch();
  face32_kernel<N1, CACHED><<<(3 * Ms.E + C::FPC - 1) / C::FPC, F32_THREADS, C::bytes, st>>>(
      sf_tab<float, N1>(Ms), Ms.phys_t<float>(), Ms.nbr, Ms.qidx, Ms.E, W, V, slots, Ms.status, Pf);
  return cudaGetLastError();
}

// Primal traces of the FP32 state in the layout of dg_sf32.cuh, by the dense
// tables (once per preconditioner refresh).
__global__ void primal_cache_sf_kernel(MeshView<float> mv, const float* __restrict__ W, float4* __restrict__ Pv,
                                       float4* __restrict__ Pf, int n1d) {
  constexpr int M = 5;
  const int nb = mv.nb, nm = mv.nm, nq = mv.nq, nqf = mv.nqf, E = mv.E;
  const long nvol = (long)E * nq, nface = (long)3 * E * nqf * 2;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < nvol + nface; t += (long)gridDim.x * blockDim.x) {
    float c[20];
#pragma unroll
    for (int j = 0; j < 20; ++j) c[j] = 0.f;
    if (t < nvol) {
      const long e = t / nq;
      const int r = (int)(t - e * nq), q0 = r / nqf, line = r - q0 * nqf, q2 = line % n1d, q1 = line / n1d;
      const int q = q0 + n1d * (q1 + n1d * q2);
      const float* w = W + (size_t)e * nb;
      for (int i = 0; i < nm; ++i) {
        const float p = mv.vphiT[(size_t)i * nq + q];
        float dp[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) dp[k] = mv.vdphiT[((size_t)k * nm + i) * nq + q];
#pragma unroll
        for (int v = 0; v < M; ++v) {
          const float a = w[v * nm + i];
          c[v] += a * p;
#pragma unroll
          for (int k = 0; k < 3; ++k) c[5 + 3 * v + k] += a * dp[k];
        }
      }
#pragma unroll
      for (int j = 0; j < 5; ++j)
        Pv[sf32_vol_word(e, q0, j, line, n1d)] = make_float4(c[4 * j], c[4 * j + 1], c[4 * j + 2], c[4 * j + 3]);
    } else {
      const long r = t - nvol;
      const long fs = r / nqf, f = fs >> 1;
      const int qi = (int)(r - fs * nqf), side = (int)(fs & 1), k = (int)(f / E);
      const int q = qi / n1d + n1d * (qi % n1d);   // b0 + nq b1
      const long e = f - (long)k * E;
      const long el = side == 0 ? e : mv.nbr[(e * 3 + k) * 2 + 1];
      const int lf = side == 0 ? 2 * k + 1 : 2 * k, t0 = k == 0 ? 1 : 0, t1 = k == 2 ? 1 : 2;
      const float* w = W + (size_t)el * nb;
      for (int i = 0; i < nm; ++i) {
        const float p = mv.fphiT[((size_t)lf * nm + i) * nqf + q];
        const float dn = mv.fdphiT[(((size_t)lf * 3 + k) * nm + i) * nqf + q];
        const float d0 = mv.fdphiT[(((size_t)lf * 3 + t0) * nm + i) * nqf + q];
        const float d1 = mv.fdphiT[(((size_t)lf * 3 + t1) * nm + i) * nqf + q];
#pragma unroll
        for (int v = 0; v < M; ++v) {
          const int pv = v == 0 || v == M - 1 ? v : v == 1 ? 1 + k : v == 2 ? 1 + t0 : 1 + t1;
          const float a = w[pv * nm + i];
          c[v] += a * p;
          c[5 + 3 * v] += a * dn;
          c[6 + 3 * v] += a * d0;
          c[7 + 3 * v] += a * d1;
        }
      }
#pragma unroll
      for (int j = 0; j < 5; ++j)
        Pf[sf32_face_word(f, side, j, qi, nqf)] = make_float4(c[4 * j], c[4 * j + 1], c[4 * j + 2], c[4 * j + 3]);
    }
  }
}

}  // namespace

bool sf32_ok(const Mesh& M) {
  return M.kind == DG_MESH_STRUCTURED && M.d == 3 && M.desc.space == DG_SPACE_P && M.p >= 1 && M.p <= 6 &&
         M.nq1d == M.p + 2 && M.qidx != nullptr;
}

cudaError_t launch_face32(const Mesh& M, const float* W, const float* V, const float* Pf, cudaStream_t st) {
  if (!sf32_ok(M)) return cudaErrorNotSupported;
  float* slots = M.t32.slots;
  const float4* P4 = reinterpret_cast<const float4*>(Pf);
  switch (M.p + 1) {
#define CASE(n)                                                                                                     \
  case n:                                                                                                           \
    return Pf ? run_face32<n, true>(M, W, V, slots, P4, st) : run_face32<n, false>(M, W, V, slots, nullptr, st);
    CASE(2)
    CASE(3)
    CASE(4)
    CASE(5)
    CASE(6)
    CASE(7)
#undef CASE
  }
  return cudaErrorNotSupported;
}

cudaError_t launch_primal_cache_sf(const Mesh& M, const float* W, float* Pv, float* Pf, cudaStream_t st) {
  const long tot = (long)M.E * M.nq + (long)3 * M.E * M.nqf * 2;
  const int grid = (int)std::min<long>((tot + 255) / 256, 65535L * 4);
  note_launch();
  primal_cache_sf_kernel<<<grid, 256, 0, st>>>(M.view<float>(), W, reinterpret_cast<float4*>(Pv),
                                               reinterpret_cast<float4*>(Pf), M.nq1d);
  return cudaGetLastError();
}

}  // namespace dgk
