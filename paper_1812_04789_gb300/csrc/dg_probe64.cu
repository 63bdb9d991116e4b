// FP64 element Jacobian blocks (Sec. 5.1 eq. ODEDG; Sec. 6.3): the diagonal
// blocks at the fine order and the neighbour blocks at the first coarse order,
// structured meshes without a direction of one element (there probe_kernel of
// dg_blocks.cu, whose faces then feed the diagonal block twice).
//
//   D[(v,i'),(w,i)] = sum_p sum_c sum_s Test_c(p,i') J_p[(v,c),(w,s)] Trial_s(p,i)
// over the element's volume points and the points of its own faces, J_p the
// derivative of the point outputs c (volume: the flux tensor; face: numerical
// flux, the two lifting integrands, the own dual tensor) with respect to the
// inputs s (value, d gradient components) of variable w.
//
// GB300 issues two FP64 lanes per clock and SM, so the kernel is bound by the
// number of FP64 instructions and by nothing else: shared-memory traffic, index
// arithmetic and barriers hide behind them.  Hence
//  * the test side first, Z_s[(w,v,i')] = sum_c Test_c J[(v,c),(w,s)], then
//    D += Z_s Trial_s: four multiply-adds per point and block entry whatever the
//    number of outputs c (probe_kernel, trial side first, takes 2d for a face);
//  * every block entry is summed in a register over all points (a thread's
//    entries are tid, tid + 256, ..: no padded tiles) and written once;
//  * J_p: a dual-number evaluation only for the seeds of the values; a seed of
//    a gradient component enters the viscous flux alone, which is linear in it
//    and is evaluated directly (the lifting and dual outputs do not see it).
// Blocks of more entries than 256 threads hold are taken in passes over the
// rows (w, v, i'), each a CTA of its own, as is an element's set of neighbour
// blocks.  9 x 10 x 12 elements, p = 3: 137 -> 34 ms (17 M multiply-adds per element at the FP64 pipe's rate: 29 ms);
// 16^2 quads, p = 2 (diagonal blocks alone): 1.63 -> 0.2 ms.  The diagonal
// blocks of 3-D P_p meshes up to p = 4 come from dg_probe_sf.cuh instead (12^3, p = 4: 198 -> 42 ms).
#include <algorithm>

#include "dg_probe.cuh"

namespace dgk {

namespace {

constexpr int P64_THREADS = 256;
constexpr int P64_ZQ = 4;     // points per contraction sub-chunk

struct P64Plan {
  int ok = 0, jq = 0, nacc = 0, passes = 0, rows = 0;   // rows of the diagonal block per pass
  int oU = 0, oJ = 0, oT = 0, oN = 0, oZ = 0, smem = 0;
};

// J entries per point and seed variable: volume (1 + d) m d, face m (3 + d) + d m
__host__ __device__ constexpr int p64_jw(int d) {
  return (1 + d) * (d + 2) * d > (d + 2) * (3 + 2 * d) ? (1 + d) * (d + 2) * d : (d + 2) * (3 + 2 * d);
}

P64Plan p64_plan(int d, int nm, int nmc, int smax) {
  P64Plan P;
  const int M = d + 2, NF = 2 * d, PU = M * (1 + d), nb = M * nm, R = M * M * nm;
  const long out = (long)R * nm, outc = (long)M * M * nmc * nmc;
  P.nacc = std::max(out, outc) <= 10L * P64_THREADS ? 10 : 40;
  const long cap = (long)P.nacc * P64_THREADS;
  if (outc > cap || nm > cap) return P;
  P.passes = (int)((out + cap - 1) / cap);
  P.rows = (R + P.passes - 1) / P.passes;
  while ((long)P.rows * nm > cap) P.rows = (R + ++P.passes - 1) / P.passes;
  const int wspan = std::min(M, (P.rows + nb - 1) / nb + 1);         // seed variables a pass can touch
  const int zr = std::max(P.rows, M * M * nmc);
  for (int jq = 48; jq >= P64_ZQ; jq -= P64_ZQ) {
    long o = 0;
    auto take = [&](long n) {
      const long r = o;
      o = (o + n + 1) / 2 * 2;      // 16-byte aligned
      return (int)r;
    };
    take((long)(1 + NF) * nb);                                   // W of the element and its neighbours
    P.oU = take((long)jq * 2 * PU);
    P.oJ = take((long)jq * (nmc > 0 ? M : wspan) * p64_jw(d));
    P.oT = take((long)P64_ZQ * (3 + d) * nm);
    P.oN = take((long)P64_ZQ * 4 * nm);
    P.oZ = take((long)P64_ZQ * zr * 4);
    if (o * (long)sizeof(double) <= smax) {
      P.jq = jq;
      P.smem = (int)(o * sizeof(double));
      P.ok = 1;
      return P;
    }
  }
  return P;
}

// column k of the viscous flux, the direction at run time
template <int D>
__device__ __forceinline__ void visc_col(int k, const double* u, const double (*g)[D], double* F, const Phys<double>& ph) {
  if (k == 0)
    flux_visc_col<D, 0, double, double>(u, g, F, ph);
  else if (k == 1)
    flux_visc_col<D, 1, double, double>(u, g, F, ph);
  else if constexpr (D == 3)
    flux_visc_col<D, 2, double, double>(u, g, F, ph);
}

// One sweep over the points [0, npts): the volume points (FACE = false) or
// points of the element's faces, s = s0 + pt / nqf.  OWN: seeds on the element's
// own trace, else on the neighbour's.  Adds to acc[u] the entry tid + u
// blockDim of the rows [r0, r1) of the (M M nmo) x nmo block, row = (w, v, i').
template <int D, int NACC, bool FACE, bool OWN>
__device__ __forceinline__ void p64_sweep(const MeshView<double>& mv, const Phys<double>& ph, const P64Plan& P,
                                          double* sm, int s0, int npts, int r0, int r1, int nmo, double* acc,
                                          int* status) {
  constexpr int M = D + 2, NS = 1 + D, KM = 3 + D, PU = M * (1 + D), JW = p64_jw(D);
  constexpr int NK = FACE ? KM : D;
  const int tid = threadIdx.x, nm = mv.nm, nb = mv.nb, nq = mv.nq, nqf = mv.nqf;
  const double* cW = sm;
  double* U = sm + P.oU;       // [jq][own, neighbour][PU]
  double* J = sm + P.oJ;       // [jq][w - w0][JW]
  double* Ts = sm + P.oT;      // [zq][NK][nmo]
  double* Tn = sm + P.oN;      // [zq][nmo][4]
  double* Z = sm + P.oZ;       // [zq][row - r0][4]
  const int w0 = r0 / (M * nmo), nw = (r1 - 1) / (M * nmo) + 1 - w0, nr = r1 - r0;
  for (int c0 = 0; c0 < npts; c0 += P.jq) {
    const int nc = min(P.jq, npts - c0);
    // traces of the state at the chunk's points
    for (int t = tid; t < nc * (FACE ? 2 : 1); t += P64_THREADS) {
      const int pl = FACE ? t >> 1 : t, side = FACE ? t & 1 : 0, pt = c0 + pl;
      const int s = FACE ? s0 + pt / nqf : 0, q = FACE ? pt % nqf : pt, lf = side ? s ^ 1 : s;
      const double* w = cW + (size_t)(side ? 1 + s : 0) * nb;
      double u[M], g[M][D];
#pragma unroll
      for (int v = 0; v < M; ++v) {
        u[v] = 0.0;
#pragma unroll
        for (int kk = 0; kk < D; ++kk) g[v][kk] = 0.0;
      }
      for (int i = 0; i < nm; ++i) {
        const double p = FACE ? mv.fphiT[((size_t)lf * nm + i) * nqf + q] : mv.vphiT[(size_t)i * nq + q];
        double dp[D];
#pragma unroll
        for (int kk = 0; kk < D; ++kk)
          dp[kk] = FACE ? mv.fdphiT[(((size_t)lf * D + kk) * nm + i) * nqf + q] : mv.vdphiT[((size_t)kk * nm + i) * nq + q];
#pragma unroll
        for (int v = 0; v < M; ++v) {
          const double a = w[v * nm + i];
          u[v] += a * p;
#pragma unroll
          for (int kk = 0; kk < D; ++kk) g[v][kk] += a * dp[kk];
        }
      }
      if (!physical<D>(u, ph.gm1)) atomicOr(status, ST_NONPHYSICAL);
      double* o = U + ((size_t)pl * 2 + side) * PU;
#pragma unroll
      for (int v = 0; v < M; ++v) {
        o[v] = u[v];
#pragma unroll
        for (int kk = 0; kk < D; ++kk) o[M + v * D + kk] = g[v][kk];
      }
    }
    __syncthreads();
    // J, value seeds: dual numbers
    for (int t = tid; t < nc * nw; t += P64_THREADS) {
      const int pl = t / nw, wl = t - pl * nw, w = w0 + wl;
      const double* pu = U + (size_t)pl * 2 * PU;
      double* jo = J + ((size_t)pl * nw + wl) * JW;
      if constexpr (FACE) {
        const int s = s0 + (c0 + pl) / nqf;
        double zero[D];
#pragma unroll
        for (int kk = 0; kk < D; ++kk) zero[kk] = 0.0;
        double oGL[M], oGR[M], oFp[M], oDo[M * D];
        face_point_tangent<D, double>(pu, pu + PU, s / 2, s % 2, w, OWN ? 1.0 : 0.0, zero, OWN ? 0.0 : 1.0, zero, ph,
                                      oGL, oGR, oFp, oDo);
#pragma unroll
        for (int v = 0; v < M; ++v) {
          jo[v * KM + 0] = oFp[v];
          jo[v * KM + 1] = oGL[v];
          jo[v * KM + 2] = oGR[v];
#pragma unroll
          for (int kk = 0; kk < D; ++kk) jo[v * KM + 3 + kk] = oDo[v * D + kk];
        }
      } else {
        using S = Dual<double>;
        S u[M], g[M][D], F[M][D];
#pragma unroll
        for (int v = 0; v < M; ++v) {
          u[v] = S(pu[v], v == w ? 1.0 : 0.0);
#pragma unroll
          for (int kk = 0; kk < D; ++kk) g[v][kk] = S(pu[M + v * D + kk], 0.0);
        }
        flux_total<D, S, double>(u, g, F, ph);
#pragma unroll
        for (int v = 0; v < M; ++v)
#pragma unroll
          for (int kk = 0; kk < D; ++kk) jo[v * D + kk] = F[v][kk].d;
      }
    }
    // J, gradient seeds: the viscous flux of a unit gradient
    for (int t = tid; t < nc * nw * D; t += P64_THREADS) {
      const int kk0 = t % D, r = t / D, pl = r / nw, wl = r - pl * nw, w = w0 + wl;
      const double* pu = U + ((size_t)pl * 2 + (FACE && !OWN ? 1 : 0)) * PU;
      double* jo = J + ((size_t)pl * nw + wl) * JW;
      double u[M], g[M][D], F[M];
#pragma unroll
      for (int v = 0; v < M; ++v) {
        u[v] = pu[v];
#pragma unroll
        for (int kk = 0; kk < D; ++kk) g[v][kk] = (v == w && kk == kk0) ? 1.0 : 0.0;
      }
      if constexpr (FACE) {
        const int s = s0 + (c0 + pl) / nqf;
        visc_col<D>(s / 2, u, g, F, ph);
#pragma unroll
        for (int v = 0; v < M; ++v) jo[M * KM + kk0 * M + v] = 0.5 * F[v];
      } else {
#pragma unroll
        for (int k = 0; k < D; ++k) {
          visc_col<D>(k, u, g, F, ph);
#pragma unroll
          for (int v = 0; v < M; ++v) jo[(1 + kk0) * M * D + v * D + k] = F[v];
        }
      }
    }
    __syncthreads();
    for (int z0 = 0; z0 < nc; z0 += P64_ZQ) {
      const int nz = min(P64_ZQ, nc - z0);
      // test and trial functions of the sub-chunk's points
      for (int t = tid; t < nz * (NK + 4) * nmo; t += P64_THREADS) {
        const int i = t % nmo, r = t / nmo, c = r % (NK + 4), pl = r / (NK + 4), pt = c0 + z0 + pl;
        if constexpr (FACE) {
          const int s = s0 + pt / nqf, q = pt % nqf, lf = OWN ? s : s ^ 1;
          const double sg = (s % 2) ? 1.0 : -1.0, fw = mv.fw[(size_t)(s / 2) * nqf + q];
          if (c == 0)
            Ts[((size_t)pl * NK + c) * nmo + i] = sg * fw * mv.fphi[((size_t)s * nqf + q) * nm + i];
          else if (c < 3)
            Ts[((size_t)pl * NK + c) * nmo + i] =
                sg * (0.5 * ph.eta) * mv.liftT[(((size_t)s * 2 + (c - 1)) * nqf + q) * nm + i];
          else if (c < NK)
            Ts[((size_t)pl * NK + c) * nmo + i] = -fw * mv.fdphi[(((size_t)s * D + (c - 3)) * nqf + q) * nm + i];
          else {
            const int sd = c - NK;
            Tn[((size_t)pl * nmo + i) * 4 + sd] =
                sd == 0 ? mv.fphi[((size_t)lf * nqf + q) * nm + i]
                        : sd < NS ? mv.fdphi[(((size_t)lf * D + (sd - 1)) * nqf + q) * nm + i] : 0.0;
          }
        } else {
          if (c < NK)
            Ts[((size_t)pl * NK + c) * nmo + i] = -mv.vw[pt] * mv.vdphi[((size_t)c * nq + pt) * nm + i];
          else {
            const int sd = c - NK;
            Tn[((size_t)pl * nmo + i) * 4 + sd] =
                sd == 0 ? mv.vphi[(size_t)pt * nm + i] : sd < NS ? mv.vdphi[((size_t)(sd - 1) * nq + pt) * nm + i] : 0.0;
          }
        }
      }
      __syncthreads();
      // Z: test side first
      for (int t = tid; t < nz * nr; t += P64_THREADS) {
        const int pl = t / nr, rl = t - pl * nr, row = r0 + rl;
        const int w = row / (M * nmo), v = (row / nmo) % M, ip = row % nmo;
        const double* jr = J + ((size_t)(z0 + pl) * nw + (w - w0)) * JW;
        const double* tr = Ts + (size_t)pl * NK * nmo + ip;
        double z[4] = {0.0, 0.0, 0.0, 0.0};
        if constexpr (FACE) {
#pragma unroll
          for (int c = 0; c < KM; ++c) z[0] += tr[c * nmo] * jr[v * KM + c];
#pragma unroll
          for (int kk = 0; kk < D; ++kk) z[1 + kk] = tr[0] * jr[M * KM + kk * M + v];
        } else {
#pragma unroll
          for (int sd = 0; sd < NS; ++sd)
#pragma unroll
            for (int c = 0; c < D; ++c) z[sd] += tr[c * nmo] * jr[sd * M * D + v * D + c];
        }
        double2* zo = reinterpret_cast<double2*>(Z + (size_t)t * 4);
        zo[0] = make_double2(z[0], z[1]);
        zo[1] = make_double2(z[2], z[3]);
      }
      __syncthreads();
      // the block entries
      const int tot = nr * nmo, di = P64_THREADS % nmo, dr = P64_THREADS / nmo;
      for (int pl = 0; pl < nz; ++pl) {
        const double* zp = Z + (size_t)pl * nr * 4;
        const double* tp = Tn + (size_t)pl * nmo * 4;
        int t = tid, row = tid / nmo, i = tid - row * nmo;
#pragma unroll
        for (int u = 0; u < NACC; ++u) {
          if (t < tot) {
            const double2 za = reinterpret_cast<const double2*>(zp + (size_t)row * 4)[0];
            const double2 zb = reinterpret_cast<const double2*>(zp + (size_t)row * 4)[1];
            const double2 ta = reinterpret_cast<const double2*>(tp + (size_t)i * 4)[0];
            const double2 tb = reinterpret_cast<const double2*>(tp + (size_t)i * 4)[1];
            double a = acc[u];
            a = fma(za.x, ta.x, a);
            a = fma(za.y, ta.y, a);
            a = fma(zb.x, tb.x, a);
            if constexpr (D == 3) a = fma(zb.y, tb.y, a);
            acc[u] = a;
          }
          t += P64_THREADS;
          row += dr;
          i += di;
          if (i >= nmo) {
            i -= nmo;
            ++row;
          }
        }
      }
      __syncthreads();
    }
  }
}

// CTA (e, job): jobs 0 .. passes - 1 the rows of element e's diagonal block, job
// passes (when Oout) its neighbour blocks.
template <int D, int NACC>
__global__ void __launch_bounds__(P64_THREADS, 1)
    probe64_kernel(MeshView<double> mv, Phys<double> ph, const double* __restrict__ W, double sigma,
                   double* __restrict__ Dout, size_t dstride, double* __restrict__ Oout, size_t ostride, int ldo,
                   int nmc, P64Plan P, int* status) {
  constexpr int M = D + 2, NF = 2 * D;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sm = reinterpret_cast<double*>(smem_raw);
  const int nm = mv.nm, nb = mv.nb, nqf = mv.nqf, tid = threadIdx.x;
  const int e = blockIdx.x, job = blockIdx.y;
  for (int t = tid; t < (1 + NF) * nb; t += P64_THREADS) {
    const int who = t / nb, j = t - who * nb, el = who == 0 ? e : mv.nbr[e * NF + who - 1];
    sm[t] = W[(size_t)el * nb + j];
  }
  __syncthreads();
  double acc[NACC];
  if (job < P.passes) {
    const int r0 = job * P.rows, r1 = min(M * M * nm, r0 + P.rows);
    if (r0 >= r1) return;
#pragma unroll
    for (int u = 0; u < NACC; ++u) acc[u] = 0.0;
    p64_sweep<D, NACC, false, true>(mv, ph, P, sm, 0, mv.nq, r0, r1, nm, acc, status);
    p64_sweep<D, NACC, true, true>(mv, ph, P, sm, 0, NF * nqf, r0, r1, nm, acc, status);
    double* De = Dout + (size_t)e * dstride;
#pragma unroll
    for (int u = 0; u < NACC; ++u) {
      const int t = tid + u * P64_THREADS;
      if (t < (r1 - r0) * nm) {
        const int row = r0 + t / nm, i = t % nm, w = row / (M * nm), j = row - w * M * nm, col = w * nm + i;
        De[(size_t)j * nb + col] = acc[u] + (j == col ? sigma * mv.detJ : 0.0);
      }
    }
    return;
  }
  const int nbc = M * nmc, R = M * nbc;
  for (int s = 0; s < NF; ++s) {
#pragma unroll
    for (int u = 0; u < NACC; ++u) acc[u] = 0.0;
    p64_sweep<D, NACC, true, false>(mv, ph, P, sm, s, nqf, 0, R, nmc, acc, status);
    double* Os = Oout + ((size_t)e * NF + s) * ostride;
#pragma unroll
    for (int u = 0; u < NACC; ++u) {
      const int t = tid + u * P64_THREADS;
      if (t < R * nmc) {
        const int row = t / nmc, i = t - row * nmc, w = row / nbc, j = row - w * nbc, col = w * nmc + i;
        Os[ldo > 0 ? (size_t)col * ldo + j : (size_t)j * nbc + col] = acc[u];
      }
    }
  }
}

template <int D, int NACC>
cudaError_t run_probe64(const Mesh& Ms, const double* W, double sigma, double* Dout, size_t dstride, double* O,
                        size_t ostride, int ldo, int nmc, const P64Plan& P, cudaStream_t st) {
  cudaError_t e = allow_max_smem(probe64_kernel<D, NACC>);
  if (e != cudaSuccess) return e;
  note_launch();
  probe64_kernel<D, NACC><<<dim3(Ms.E, P.passes + (O ? 1 : 0)), P64_THREADS, P.smem, st>>>(
      Ms.view<double>(), Ms.phys_t<double>(), W, sigma, Dout, dstride, O, ostride, ldo, nmc, P, Ms.status);
  return cudaGetLastError();
}

bool probe64_plan(const Mesh& M, int nmc, P64Plan* P) {
  if (M.kind != DG_MESH_STRUCTURED || nmc > M.nm) return false;
  for (int k = 0; k < M.d; ++k)
    if (M.desc.n[k] == 1) return false;
  int dev = 0, smax = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  *P = p64_plan(M.d, M.nm, nmc, smax - 1024);
  return P->ok != 0 && P->passes < 65535;
}

}  // namespace

bool probe64_fits(const Mesh& M, int nmc) {
  P64Plan P;
  return probe64_plan(M, nmc, &P);
}

cudaError_t launch_probe64(const Mesh& M, const double* W, double sigma, double* D, size_t dstride, double* O,
                           int nmc, int colmajor, cudaStream_t st) {
  P64Plan P;
  if (!O) nmc = 0;
  if (!probe64_plan(M, nmc, &P)) return cudaErrorInvalidValue;
  const int nbc = M.m * nmc, ldo = colmajor ? inv_ld<double>(nbc) : 0;
  const size_t ostride = (size_t)nbc * (ldo ? ldo : nbc);
  if (M.d == 2)
    return P.nacc == 10 ? run_probe64<2, 10>(M, W, sigma, D, dstride, O, ostride, ldo, nmc, P, st)
                        : run_probe64<2, 40>(M, W, sigma, D, dstride, O, ostride, ldo, nmc, P, st);
  return P.nacc == 10 ? run_probe64<3, 10>(M, W, sigma, D, dstride, O, ostride, ldo, nmc, P, st)
                      : run_probe64<3, 40>(M, W, sigma, D, dstride, O, ostride, ldo, nmc, P, st);
}

}  // namespace dgk
