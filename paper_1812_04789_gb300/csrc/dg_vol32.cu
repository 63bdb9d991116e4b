// Volume term of the FP32 Jacobian-vector product on 3-D P_p meshes (the mixed
// preconditioner's fine-level operator and the FP32 product mode; Sec. 3.1 eq.
// dg_ns, Sec. 5.1) by sum factorisation, p = 1 .. 6 with p + 2 points.
//
// Against the dense contractions of volume_kernel_st (600 k FP32 operations per
// element at p = 4) the factorised ones take about 60 k, and the point physics
// becomes the larger part; what then limits the kernel is instruction issue,
// so the stages are built to spend few instructions per operation: a thread
// contracts a whole line at once (n values in, n + 1 points out), its loops are
// unrolled and its tables are constant-bank operands.  Stages, per element
// (a0, a1, a2 mode degrees, q0, q1, q2 points):
//   A   Z_s[v][a0 a1][q2] = sum_a2 V L^s_a2(q2), s = value, derivative
//   B   Y_t[v][a0][q1 q2] = sum_a1 (Z L, Z L', Z' L)
//   pt  a thread per line (q1, q2): for each q0 the traces from Y (sum over a0),
//       the tangent of the flux, and at once its projection over q0, summed in
//       registers: P_j[v][a0] += w L_a0(q0) F_j
//   B^T, A^T the transposed contractions to the modes
//   then the face slots in a fixed order and sigma |J| v.
// The state's traces come from the cache of the preconditioner (CACHED) or are
// interpolated along with the direction's.  16^3 elements, p = 4 with cached
// traces: 165 -> 51 us; 16^3, p = 6: 1,015 -> 169 us.
#include "dg_sf32.cuh"

namespace dgk {

namespace {

constexpr int V32_THREADS = 128;

// Tangent of F_c + F_v (flux_total) at the state (u, g) along (tu, tg); whether the
// state is physical (physical(), from the pressure at hand).
__device__ __forceinline__ bool flux_tangent(const float* u, const float (*g)[3], const float* tu, const float (*tg)[3],
                                             const Phys<float>& ph, float (*F)[3]) {
  const float ir = 1.f / u[0];
  float vel[3], dv[3];
  const float dr = tu[0] * ir;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    vel[j] = u[1 + j] * ir;
    dv[j] = tu[1 + j] * ir - vel[j] * dr;
  }
  float mv = 0.f, dmv = 0.f;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    mv = fmaf(u[1 + j], vel[j], mv);
    dmv = fmaf(tu[1 + j], vel[j], fmaf(u[1 + j], dv[j], dmv));
  }
  const float p = ph.gm1 * fmaf(-0.5f, mv, u[4]), dp = ph.gm1 * fmaf(-0.5f, dmv, tu[4]);
  const float e0 = u[4] * ir, h0 = fmaf(p, ir, e0);
  const float de0 = tu[4] * ir - e0 * dr, dh0 = (tu[4] + dp) * ir - h0 * dr;
  float a[3][3], da[3][3], b[3], db[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float g0 = g[0][k], t0 = tg[0][k];
    b[k] = fmaf(-e0, g0, g[4][k]);
    db[k] = fmaf(-e0, t0, fmaf(-de0, g0, tg[4][k]));
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      a[j][k] = fmaf(-vel[j], g0, g[1 + j][k]);
      da[j][k] = fmaf(-vel[j], t0, fmaf(-dv[j], g0, tg[1 + j][k]));
      b[k] = fmaf(-vel[j], a[j][k], b[k]);
      db[k] = fmaf(-vel[j], da[j][k], fmaf(-dv[j], a[j][k], db[k]));
    }
  }
  const float mi = ph.mu * ir, ki = ph.kq * ir;
  const float div = (2.f / 3.f) * (a[0][0] + a[1][1] + a[2][2]);
  const float ddiv = (2.f / 3.f) * (da[0][0] + da[1][1] + da[2][2]);
  float tau[3][3], dt[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j <= k; ++j) {
      const float s = j == k ? fmaf(2.f, a[k][k], -div) : a[j][k] + a[k][j];
      const float ds = j == k ? fmaf(2.f, da[k][k], -ddiv) : da[j][k] + da[k][j];
      tau[j][k] = tau[k][j] = mi * s;
      dt[j][k] = dt[k][j] = fmaf(mi, ds, -dr * tau[j][k]);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    F[0][k] = tu[1 + k];
#pragma unroll
    for (int j = 0; j <= k; ++j) {
      float f = fmaf(tu[1 + j], vel[k], fmaf(u[1 + j], dv[k], -dt[j][k]));
      if (j == k) f += dp;
      F[1 + j][k] = F[1 + k][j] = f;
    }
    float q = ki * fmaf(-dr, b[k], db[k]);
#pragma unroll
    for (int j = 0; j < 3; ++j) q = fmaf(vel[j], dt[j][k], fmaf(dv[j], tau[j][k], q));
    F[4][k] = fmaf(tu[1 + k], h0, fmaf(u[1 + k], dh0, -q));
  }
  return u[0] > 0.f && p > 0.f;
}

template <int N1, bool CACHED>
struct V32 {
  static constexpr int NQ = N1 + 1, NL = NQ * NQ, NP = sf32_pairs(N1), NM = sf32_modes(N1), M = 5, NB = M * NM;
  static constexpr int NC = CACHED ? 1 : 2;                      // fields interpolated: (state,) direction
  static constexpr int EPC = V32_THREADS / NL > 0 ? V32_THREADS / NL : 1;
  static constexpr int TS = (2 * N1 + 1 + 3) / 4 * 4;            // table row per q0: L, met0 dL, w
  static constexpr int nV = NC * NB, nZ = NC * 2 * M * NP * NQ, nY = NC * 3 * M * N1 * NL;   // per element
  static constexpr int oZ = (EPC * nV + 3) / 4 * 4, oY = oZ + (EPC * nZ + 3) / 4 * 4, oT = oY + (EPC * nY + 3) / 4 * 4,
                       oI = oT + NQ * TS;
  static constexpr size_t bytes = sizeof(float) * oI + sizeof(unsigned short) * (NM + 2 * NP + 2);
  static constexpr int nld = (EPC * NB + V32_THREADS - 1) / V32_THREADS;   // coefficient loads of a thread
};

template <int N1, bool CACHED>
__global__ void __launch_bounds__(V32_THREADS) vol32_kernel(const __grid_constant__ Sf32Tab<N1> tb, Phys<float> ph,
                                                            const int* __restrict__ nbr, const int* __restrict__ qidx,
                                                            int E, const float* __restrict__ W,
                                                            const float* __restrict__ V,
                                                            const float* __restrict__ slots, float sigma,
                                                            float* __restrict__ out, int* status,
                                                            const float4* __restrict__ Pv) {
  using C = V32<N1, CACHED>;
  constexpr int NQ = C::NQ, NL = C::NL, NP = C::NP, NM = C::NM, M = C::M, NB = C::NB, NC = C::NC, EPC = C::EPC;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* sm = reinterpret_cast<float*>(smem_raw);
  float* sV = sm;                  // [el][c][NB], later the modes' sums [el][NB]
  float* Z = sm + C::oZ;           // [el][c][s][v][pair][q2], later [el][A, B][v][pair][q2]
  float* Y = sm + C::oY;           // [el][c][t][v][a0][q2 + NQ q1], later the projections P in c = 0
  float* sT = sm + C::oT;
  unsigned short* pos = reinterpret_cast<unsigned short*>(sm + C::oI);    // mode -> sf32_pos, a2 contiguous
  unsigned short* ptab = pos + NM;                                        // pair -> a0 | a1 << 8
  unsigned short* poff = ptab + NP;                                       // pair -> sf32_run
  const int tid = threadIdx.x, e0 = blockIdx.x * EPC, ne = min(EPC, E - e0);
  float xw[CACHED ? 1 : C::nld], xv[C::nld];   // (all of a thread's coefficient loads in flight together)
#pragma unroll
  for (int u = 0; u < C::nld; ++u) {
    const int t = min(tid + u * V32_THREADS, ne * NB - 1);
    xv[u] = V[(size_t)e0 * NB + t];
    if constexpr (!CACHED) xw[u] = W[(size_t)e0 * NB + t];
  }
  for (int t = tid; t < N1 * N1 * N1; t += V32_THREADS) {
    const int i = qidx[t];
    if (i >= 0) pos[i] = (unsigned short)sf32_pos<N1>(t, 2);
  }
  for (int t = tid; t < N1 * N1; t += V32_THREADS) {
    const int a0 = t / N1, a1 = t - a0 * N1;
    if (a0 + a1 < N1) {
      ptab[sf32_pair0(N1, a0) + a1] = (unsigned short)(a0 | a1 << 8);
      poff[sf32_pair0(N1, a0) + a1] = (unsigned short)sf32_run(N1, a0, a1);
    }
  }
  for (int t = tid; t < NQ * C::TS; t += V32_THREADS) {
    const int q = t / C::TS, a = t - q * C::TS;
    sT[t] = a < N1 ? tb.L[a][q] : a < 2 * N1 ? tb.met[0] * tb.dL[a - N1][q] : a == 2 * N1 ? tb.w[q] : 0.f;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < C::nld; ++u) {
    const int t = min(tid + u * V32_THREADS, ne * NB - 1);
    const int el = t / NB, j = t - el * NB, v = j / NM, p = v * NM + pos[j - v * NM];
    if constexpr (!CACHED) sV[el * NC * NB + p] = xw[u];
    sV[(el * NC + NC - 1) * NB + p] = xv[u];
  }
  __syncthreads();
  // A (the pair slowest: the lanes of a warp run sums of one length)
  // (these loops run over all EPC elements, also where the last CTA has fewer: the
  // index divisions are then by constants)
  for (int t = tid; t < NP * EPC * NC * M; t += V32_THREADS) {
    const int pr = t / (EPC * NC * M), r = t - pr * (EPC * NC * M), ec = r / M, v = r - ec * M;
    const int na = N1 - (ptab[pr] & 255) - (ptab[pr] >> 8);
    const float* w = sV + ec * NB + v * NM + poff[pr];
    float z0[NQ], z1[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) z0[q] = z1[q] = 0.f;
#pragma unroll
    for (int a2 = 0; a2 < N1; ++a2) {
      if (a2 < na) {
        const float x = w[a2];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          z0[q] = fmaf(x, tb.L[a2][q], z0[q]);
          z1[q] = fmaf(x, tb.dL[a2][q], z1[q]);
        }
      }
    }
    float* o = Z + ((ec * 2 * M + v) * NP + pr) * NQ;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      o[q] = z0[q];
      o[M * NP * NQ + q] = z1[q];
    }
  }
  __syncthreads();
  // B (a0 slowest)
  for (int t = tid; t < N1 * EPC * NC * M * NQ; t += V32_THREADS) {
    const int a0 = t / (EPC * NC * M * NQ), r = t - a0 * (EPC * NC * M * NQ), ecv = r / NQ, q2 = r - ecv * NQ;
    const int ec = ecv / M, v = ecv - ec * M, na = N1 - a0;
    const float* z = Z + ((ec * 2 * M + v) * NP + sf32_pair0(N1, a0)) * NQ + q2;
    float y0[NQ], y1[NQ], y2[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) y0[q] = y1[q] = y2[q] = 0.f;
#pragma unroll
    for (int a1 = 0; a1 < N1; ++a1) {
      if (a1 < na) {
        const float x0 = z[a1 * NQ], x1 = z[M * NP * NQ + a1 * NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          y0[q] = fmaf(x0, tb.L[a1][q], y0[q]);
          y1[q] = fmaf(x0, tb.dL[a1][q], y1[q]);
          y2[q] = fmaf(x1, tb.L[a1][q], y2[q]);
        }
      }
    }
    float* o = Y + ((ec * 3 * M + v) * N1 + a0) * NL + q2;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      o[q * NQ] = y0[q];
      o[M * N1 * NL + q * NQ] = tb.met[1] * y1[q];
      o[2 * M * N1 * NL + q * NQ] = tb.met[2] * y2[q];
    }
  }
  __syncthreads();
  // points, a line (q1, q2) per thread
  if (tid < ne * NL) {
    const int el = tid / NL, line = tid - el * NL;
    const float* ye = Y + el * C::nY + line;
    float P[3][M][N1];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int v = 0; v < M; ++v)
#pragma unroll
        for (int a = 0; a < N1; ++a) P[j][v][a] = 0.f;
    const float w12 = tb.detJ * sT[(line / NQ) * C::TS + 2 * N1] * sT[(line % NQ) * C::TS + 2 * N1];
    bool ok = true;
#pragma unroll 1
    for (int q0 = 0; q0 < NQ; ++q0) {
      float la[C::TS];
#pragma unroll
      for (int a = 0; a < C::TS; a += 4) {
        const float4 x = *reinterpret_cast<const float4*>(sT + q0 * C::TS + a);
        la[a] = x.x, la[a + 1] = x.y, la[a + 2] = x.z, la[a + 3] = x.w;
      }
      float u[M], g[M][3], tu[M], tg[M][3];
      if constexpr (CACHED) {
        float c[20];
#pragma unroll
        for (int w = 0; w < 5; ++w) {
          const float4 x = __ldg(Pv + sf32_vol_word(e0 + el, q0, w, line, NQ));
          c[4 * w] = x.x, c[4 * w + 1] = x.y, c[4 * w + 2] = x.z, c[4 * w + 3] = x.w;
        }
#pragma unroll
        for (int v = 0; v < M; ++v) {
          u[v] = c[v];
#pragma unroll
          for (int k = 0; k < 3; ++k) g[v][k] = c[5 + 3 * v + k];
        }
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float* uu = (!CACHED && c == 0) ? u : tu;
        float(*gg)[3] = (!CACHED && c == 0) ? g : tg;
#pragma unroll
        for (int v = 0; v < M; ++v) {
          float s = 0.f, d0 = 0.f, d1 = 0.f, d2 = 0.f;
#pragma unroll
          for (int a = 0; a < N1; ++a) {
            const float* y = ye + ((c * 3 * M + v) * N1 + a) * NL;
            const float y0 = y[0];
            s = fmaf(y0, la[a], s);
            d0 = fmaf(y0, la[N1 + a], d0);
            d1 = fmaf(y[M * N1 * NL], la[a], d1);
            d2 = fmaf(y[2 * M * N1 * NL], la[a], d2);
          }
          uu[v] = s;
          gg[v][0] = d0;
          gg[v][1] = d1;
          gg[v][2] = d2;
        }
      }
      float F[M][3];
      const bool phys = flux_tangent(u, g, tu, tg, ph, F);
      ok = ok && phys;
      const float w = w12 * la[2 * N1], w1 = w * tb.met[1], w2 = w * tb.met[2];
#pragma unroll
      for (int v = 0; v < M; ++v) {
        const float f0 = w * F[v][0], f1 = w1 * F[v][1], f2 = w2 * F[v][2];
#pragma unroll
        for (int a = 0; a < N1; ++a) {
          P[0][v][a] = fmaf(f0, la[N1 + a], P[0][v][a]);
          P[1][v][a] = fmaf(f1, la[a], P[1][v][a]);
          P[2][v][a] = fmaf(f2, la[a], P[2][v][a]);
        }
      }
    }
    if (!ok) atomicOr(status, ST_NONPHYSICAL);
    float* po = Y + el * C::nY + line;       // over this line's own Y values
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int v = 0; v < M; ++v)
#pragma unroll
        for (int a = 0; a < N1; ++a) po[((j * M + v) * N1 + a) * NL] = P[j][v][a];
  }
  __syncthreads();
  // B^T
  for (int t = tid; t < N1 * EPC * M * NQ; t += V32_THREADS) {
    const int a0 = t / (EPC * M * NQ), r = t - a0 * (EPC * M * NQ), ev = r / NQ, q2 = r - ev * NQ;
    const int el = ev / M, v = ev - el * M, na = N1 - a0;
    const float* p = Y + el * C::nY + (v * N1 + a0) * NL + q2;
    float p0[NQ], p1[NQ], p2[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      p0[q] = p[q * NQ];
      p1[q] = p[M * N1 * NL + q * NQ];
      p2[q] = p[2 * M * N1 * NL + q * NQ];
    }
    float* o = Z + ((el * 2 * M + v) * NP + sf32_pair0(N1, a0)) * NQ + q2;
#pragma unroll
    for (int a1 = 0; a1 < N1; ++a1) {
      if (a1 < na) {
        float s = 0.f, d = 0.f;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          s = fmaf(tb.L[a1][q], p0[q], fmaf(tb.dL[a1][q], p1[q], s));
          d = fmaf(tb.L[a1][q], p2[q], d);
        }
        o[a1 * NQ] = s;
        o[M * NP * NQ + a1 * NQ] = d;
      }
    }
  }
  __syncthreads();
  // A^T
  for (int t = tid; t < NP * EPC * M; t += V32_THREADS) {
    const int pr = t / (EPC * M), ev = t - pr * (EPC * M), el = ev / M, v = ev - el * M;
    const int na = N1 - (ptab[pr] & 255) - (ptab[pr] >> 8);
    const float* z = Z + ((el * 2 * M + v) * NP + pr) * NQ;
    float za[NQ], zb[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      za[q] = z[q];
      zb[q] = z[M * NP * NQ + q];
    }
    float* o = sV + el * NB + v * NM + poff[pr];
#pragma unroll
    for (int a2 = 0; a2 < N1; ++a2) {
      if (a2 < na) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < NQ; ++q) s = fmaf(tb.L[a2][q], za[q], fmaf(tb.dL[a2][q], zb[q], s));
        o[a2] = s;
      }
    }
  }
  __syncthreads();
  // face contributions in fixed order: for each direction, own +k face then -k face
  for (int t = tid; t < ne * NB; t += V32_THREADS) {
    const int el = t / NB, j = t - el * NB, e = e0 + el;
    const int v = j / NM;
    float a = -sV[el * NB + v * NM + pos[j - v * NM]];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int em = nbr[(e * 3 + k) * 2];
      a += slots[(((size_t)e * 3 + k) * 2 + 0) * NB + j];
      a += slots[(((size_t)em * 3 + k) * 2 + 1) * NB + j];
    }
    out[(size_t)e0 * NB + t] = fmaf(sigma * tb.detJ, V[(size_t)e0 * NB + t], a);
  }
}

template <int N1, bool CACHED>
cudaError_t run_vol32(const Mesh& Ms, const float* W, const float* V, const float* slots, float sigma, float* out,
                      const float4* Pv, cudaStream_t st) {
  using C = V32<N1, CACHED>;
  cudaError_t e = allow_max_smem(vol32_kernel<N1, CACHED>);
  if (e != cudaSuccess) return e;
  note_launch();
  vol32_kernel<N1, CACHED><<<(Ms.E + C::EPC - 1) / C::EPC, V32_THREADS, C::bytes, st>>>(
      sf_tab<float, N1>(Ms), Ms.phys_t<float>(), Ms.nbr, Ms.qidx, Ms.E, W, V, slots, sigma, out, Ms.status, Pv);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_vol32(const Mesh& M, const float* W, const float* V, float sigma, float* out, const float* Pv,
                         cudaStream_t st) {
  if (!sf32_ok(M)) return cudaErrorNotSupported;
  const float* slots = M.t32.slots;
  const float4* P4 = reinterpret_cast<const float4*>(Pv);
  switch (M.p + 1) {
#define CASE(n)                                                              \
  case n:                                                                    \
    return Pv ? run_vol32<n, true>(M, W, V, slots, sigma, out, P4, st)       \
              : run_vol32<n, false>(M, W, V, slots, sigma, out, nullptr, st);
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

}  // namespace dgk
