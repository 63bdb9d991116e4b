// One step of the Arnoldi process (classical Gram-Schmidt twice, the new basis
// vector, the Hessenberg column through its Givens rotations) as one
// cooperative kernel, for vectors of which every CTA holds its part of w in
// shared memory.
//
// A kernel per operation takes ten launches of 2 to 6 us a step, whatever the
// size: on 16^2 quads at p = 2 (6,144 unknowns) 32 of an FGMRES iteration's 90
// us.  Here the CTAs exchange the sums of the two passes by polled values
// (dg_exchange.cuh, two exchanges of 3 to 4 us; the norm comes with the second
// pass, |w - V h|^2 = w.w - h.h, and from a third exchange where that cancels: an
// exhausted Krylov space), and w stays in shared memory.  The sums are those of mdot_kernel: FP64 vectors in FP64;
// FP32 vectors with at most 16 products per FP64 addition, a CTA's lanes in
// FP32, the CTAs in FP64.  Fixed order: results do not depend on timing.
// us per step, kernels per operation / here: FP64, 16^2, p = 2 (up to 45 vectors): 32
// / 20; FP32, 100 x 75, p = 3 (up to 10): 31 / 20; 16^3, p = 4: 37 / 31; 16^3, p = 6:
// 58 / 51.  Bound by the two exchanges and the launch, at 16^3 by the reads of V.
// Every wait is bounded as in dg_smoother.cu: ST_TIMEOUT in the status word, and
// the step's outputs are then unwritten: the caller stops (fgm_check_kernel).
#include <algorithm>

#include "dg_exchange.cuh"

namespace dgk {

namespace {

constexpr int ARN_THREADS = 512, ARN_WARPS = ARN_THREADS / 32;

template <class T>
struct ArnArgs {
  T* V;                 // [nmax + 1][N]
  const T* w;
  double *H, *cs, *sn, *g, *res;   // H: column j
  int* kdim;
  Pair64* px;           // [2][nmax + 2][G + 1] partial sums
  Pair64* sums;         // [2][nmax + 2][SUM_STRIDE]
  double* Q;            // [nmax + 2][nmax + 2] the q_i
  unsigned* epoch;
  int* status;
  long N, chunk;
  int j, ni, extra;     // extra: CTAs that the exchanges wait for and that do not exist (a test's)
};

// a warp's sum of a[r] b[r] over its lanes' rows r = lane, lane + 32, .. < n
__device__ __forceinline__ double warp_dot(const double* a, const double* b, int n) {
  double s = 0.0;
#pragma unroll 4
  for (int r = threadIdx.x & 31; r < n; r += 32) s = fma(a[r], b[r], s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
__device__ __forceinline__ double warp_dot(const float* a, const float* b, int n) {
  double s = 0.0;
  for (int r0 = threadIdx.x & 31; r0 < n; r0 += 16 * 32) {
    float f = 0.f;
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (r0 + 32 * u < n) f = fmaf(a[r0 + 32 * u], b[r0 + 32 * u], f);
    s += (double)f;
  }
  float t = (float)s;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return (double)t;
}

// the norm and its reciprocal from its square; 0 and 0 where that is zero or not finite
__device__ __forceinline__ void set_norm(double s, double* nrm, double* inv, int* bad) {
  const bool fin = isfinite(s);
  const double i = s > 0.0 && fin ? rsqrt(s) : 0.0;
  *inv = i;
  *nrm = s > 0.0 && fin ? s * i : 0.0;
  *bad = !fin;
}

// w -= V h, four rows of a thread together (their loads in flight); few rows:
// groups of threads take every gr-th vector each (ps: their sums)
template <class T>
__device__ __forceinline__ void subtract(const T* V, long N, const double2* h, int nv, int n, T* w, T* ps) {
  constexpr int U = 4;
  const int n32 = (n + 31) & ~31, gr = n32 > 0 ? min(16, ARN_THREADS / n32) : 1;
  if (gr > 1) {
    const int g = threadIdx.x / n32, r = threadIdx.x - g * n32;
    if (g < gr && r < n) {
      T x = T(0);
#pragma unroll 4
      for (int i = g; i < nv; i += gr) x = fma((T)h[i].x, V[(size_t)i * N + r], x);
      ps[threadIdx.x] = x;
    }
    __syncthreads();
    if (threadIdx.x < n) {
      T x = w[threadIdx.x];
      for (int k = 0; k < gr; ++k) x -= ps[k * n32 + threadIdx.x];
      w[threadIdx.x] = x;
    }
    return;
  }
  for (int r0 = threadIdx.x; r0 < n; r0 += U * ARN_THREADS) {
    T x[U];
    const T* v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = min(r0 + u * ARN_THREADS, n - 1);     // (past the end: the last row again, not stored)
      v[u] = V + r;
      x[u] = w[r];
    }
#pragma unroll 4
    for (int i = 0; i < nv; ++i) {
      const T c = -(T)h[i].x;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (u == 0 || r0 + u * ARN_THREADS < n) x[u] = fma(c, v[u][(size_t)i * N], x[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (r0 + u * ARN_THREADS < n) w[r0 + u * ARN_THREADS] = x[u];
  }
}

template <class T>
__global__ void __launch_bounds__(ARN_THREADS, 1) arnoldi_kernel(ArnArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, G = gridDim.x, j = a.j, nv = j + 1;
  double2* st = reinterpret_cast<double2*>(smem_raw);   // [ni]
  double* hs = reinterpret_cast<double*>(st + a.ni);    // [ni] the new column
  double* rot = hs + a.ni;                              // [2 ni] old rotations (CTA 0)
  double* red = rot + 2 * a.ni;                         // [max(ni, warps)] partial sums
  T* ps = reinterpret_cast<T*>(red + a.ni + ARN_WARPS); // [threads]
  T* ws = ps + ARN_THREADS;                             // [chunk]
  __shared__ int timed_out;
  __shared__ double s_nrm, s_inv;
  __shared__ int s_expl, s_bad;
  const long beg = min(a.N, blockIdx.x * a.chunk);
  const int n = (int)(min(a.N, beg + a.chunk) - beg);
  if (tid == 0) timed_out = (*(volatile int*)a.status & ST_TIMEOUT) ? 1 : 0;
  const unsigned base = *(volatile unsigned*)a.epoch;
  for (int r = tid; r < n; r += ARN_THREADS) ws[r] = a.w[beg + r];
  if (blockIdx.x == 0) {
    if (tid == 0 && j == 0) a.Q[0] = 1.0;
    for (int i = tid; i < j; i += ARN_THREADS) {
      rot[i] = a.cs[i];
      rot[a.ni + i] = a.sn[i];
    }
  }
  __syncthreads();
  if (timed_out) return;
  const T* Vc = a.V + beg;
  // pass 0: h = V^T w, w -= V h; pass 1: the same again, with w.w beside it
  for (int pass = 0; pass < 2; ++pass) {
    const unsigned ep = base + 1u + (unsigned)pass;
    const int items = nv + pass, sp = max(1, ARN_WARPS / items);   // warps per inner product
    Pair64* px = a.px + (size_t)pass * a.ni * (G + 1);
    const int per = (n + sp - 1) / sp;
    for (int k = warp; k < items * sp; k += ARN_WARPS) {
      const int i = k / sp, r0 = min(n, (k - i * sp) * per), m = min(n, r0 + per) - r0;
      const T* v = i < nv ? Vc + (size_t)i * a.N : ws;
      const double s = warp_dot(v + r0, ws + r0, m);
      if (lane == 0) red[k] = s;
    }
    __syncthreads();
    for (int i = tid; i < items; i += ARN_THREADS) {
      double s = 0.0;
      if (sizeof(T) == 4) {      // (a CTA's sum in FP32, as mdot_kernel's)
        float f = 0.f;
        for (int k = 0; k < sp; ++k) f += (float)red[i * sp + k];
        s = (double)f;
      } else {
        for (int k = 0; k < sp; ++k) s += red[i * sp + k];
      }
      Xch<double>::stp(px + (size_t)i * (G + 1) + blockIdx.x, s, 0.0, ep);
    }
    const bool ok =
        gather_dots<double, ARN_WARPS>(px, G + 1, items, G + a.extra, a.sums + (size_t)pass * a.ni * SUM_STRIDE, ep, a.status, st);
    if (__syncthreads_or(ok ? 0 : 1)) {
      if (tid == 0) atomicMax(a.epoch, base + 8u);
      return;
    }
    if (pass == 1) break;
    subtract(Vc, a.N, st, nv, n, ws, ps);
    for (int i = tid; i < nv; i += ARN_THREADS) hs[i] = st[i].x;
    __syncthreads();
  }
  // |w - V h2|^2 = w.w - h2.h2 (h2 is the rounding of the first pass along V),
  // unless h2 carries half of w: then w is little but rounding, and the
  // difference too, and the norm is summed over what is left
  if (warp == 0) {
    double h2 = 0.0;
    for (int i = lane; i < nv; i += 32) h2 = fma(st[i].x, st[i].x, h2);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) h2 += __shfl_xor_sync(0xffffffffu, h2, o);
    const double ww = st[nv].x, s = ww - h2;
    if (lane == 0) {
      s_expl = s < 0.5 * ww;
      set_norm(s, &s_nrm, &s_inv, &s_bad);
    }
  } else if (blockIdx.x == 0) {
    // the old rotations on the new column: entry i < j becomes c_i (q_i . h[0..i]) +
    // s_i h[i + 1] and the last one q_j . h, q_i the last row of the product of the
    // rotations before i (a serial sweep of 4 j FP64 operations otherwise); a warp per entry
    for (int i = warp - 1; i <= j; i += ARN_WARPS - 1) {
      double s = 0.0;
      for (int k = lane; k <= i; k += 32) s = fma(a.Q[(size_t)i * a.ni + k], hs[k] + st[k].x, s);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) {
        if (i < j)
          a.H[i] = rot[i] * s + rot[a.ni + i] * (hs[i + 1] + st[i + 1].x);
        else
          red[0] = s;
      }
    }
  }
  subtract(Vc, a.N, st, nv, n, ws, ps);
  __syncthreads();
  if (s_expl) {      // (the same in every CTA; every CTA is done with the first pass' buffers)
    const unsigned ep = base + 3u;
    const int per = (n + ARN_WARPS - 1) / ARN_WARPS, r0 = min(n, warp * per), m = min(n, r0 + per) - r0;
    const double s = warp_dot(ws + r0, ws + r0, m);
    if (lane == 0) red[1 + warp] = s;      // (red[0]: the rotations' last entry)
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int k = 0; k < ARN_WARPS; ++k) t += red[1 + k];
      Xch<double>::stp(a.px + blockIdx.x, t, 0.0, ep);
    }
    const bool ok = gather_dots<double, ARN_WARPS>(a.px, G + 1, 1, G + a.extra, a.sums, ep, a.status, st);
    if (__syncthreads_or(ok ? 0 : 1)) {
      if (tid == 0) atomicMax(a.epoch, base + 8u);
      return;
    }
    if (tid == 0) set_norm(st[0].x, &s_nrm, &s_inv, &s_bad);
    __syncthreads();
  }
  if (blockIdx.x == 0 && tid == 0) {
    if (s_bad) atomicOr(a.kdim + 1, ST_NONFINITE);
    if (!(s_nrm > 0.0) && *a.kdim > j + 1) *a.kdim = j + 1;
  }
  T* vn = a.V + (size_t)nv * a.N + beg;
  const T inv = (T)s_inv;
  for (int r = tid; r < n; r += ARN_THREADS) vn[r] = inv * ws[r];
  if (blockIdx.x == 0 && warp == 0) {
    const double p = red[0], q = s_nrm, r2 = p * p + q * q;
    double c = 1.0, s = 0.0;
    if (r2 > 0.0) {
      const double ir = rsqrt(r2);
      c = p * ir;
      s = q * ir;
    }
    // q_{j+1} = (-s q_j, c)
    for (int k = lane; k <= j; k += 32) a.Q[(size_t)nv * a.ni + k] = -s * a.Q[(size_t)j * a.ni + k];
    if (lane == 0) {
      a.Q[(size_t)nv * a.ni + nv] = c;
      a.cs[j] = c;
      a.sn[j] = s;
      a.H[j] = c * p + s * q;
      a.H[nv] = 0.0;
      const double gj = a.g[j];
      a.g[nv] = -s * gj;
      a.g[j] = c * gj;
      *a.res = fabs(s * gj);
      *(volatile unsigned*)a.epoch = base + 8u;
    }
  }
}

template <class T>
size_t arn_smem(long chunk, int ni) {
  return sizeof(double2) * ni + sizeof(double) * (4 * (size_t)ni + ARN_WARPS) + sizeof(T) * ((size_t)chunk + ARN_THREADS);
}

}  // namespace

template <class T>
cudaError_t plan_arnoldi(Krylov<T>& K, size_t* bytes) {
  K.ag = 0;
  *bytes = 0;
  const char* nco = getenv("DG_PMG_NO_COOP");   // 1: a kernel per operation
  if (nco && nco[0] == '1') return cudaSuccess;
  const int ni = K.nmax + 2;
  const long G = std::max<long>(1, std::min<long>(sm_count(), (K.N + 255) / 256)), chunk = (K.N + G - 1) / G;
  // (measured up to 11,321 entries a CTA, where a step takes 51 us against 58 of the kernels per operation)
  if (chunk > 12288) return cudaSuccess;
  const size_t smem = arn_smem<T>(chunk, ni);
  if (smem > 200 * 1024) return cudaSuccess;
  cudaError_t e = allow_max_smem(arnoldi_kernel<T>);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, arnoldi_kernel<T>, ARN_THREADS, smem);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaSuccess;
  K.ag = (int)((K.N + chunk - 1) / chunk);      // no CTA without entries
  K.achunk = chunk;
  const char* extra = getenv("DG_TEST_ARNOLDI_EXTRA");   // test hook: an exchange that is never complete
  K.aextra = extra && extra[0] == '1' ? 1 : 0;
  *bytes = sizeof(Pair64) * 2 * (size_t)ni * (K.ag + 1 + SUM_STRIDE) + sizeof(double) * (size_t)ni * ni;
  return cudaSuccess;
}

template <class T>
cudaError_t launch_arnoldi(const Krylov<T>& K, int j, cudaStream_t st) {
  ArnArgs<T> a;
  a.V = K.V;
  a.w = K.w;
  a.H = K.H + (size_t)j * (K.nmax + 1);
  a.cs = K.cs;
  a.sn = K.sn;
  a.g = K.g;
  a.res = K.res;
  a.kdim = K.kdim;
  a.ni = K.nmax + 2;
  a.px = (Pair64*)K.apx;
  a.sums = a.px + 2 * (size_t)a.ni * (K.ag + 1);
  a.Q = (double*)(a.sums + 2 * (size_t)a.ni * SUM_STRIDE);
  a.epoch = K.aepoch;
  a.status = K.astatus;
  a.N = K.N;
  a.chunk = K.achunk;
  a.j = j;
  a.extra = K.aextra;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(K.ag);
  cfg.blockDim = dim3(ARN_THREADS);
  cfg.dynamicSmemBytes = arn_smem<T>(K.achunk, a.ni);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  note_launch();
  return cudaLaunchKernelEx(&cfg, arnoldi_kernel<T>, a);
}

template cudaError_t plan_arnoldi<double>(Krylov<double>&, size_t*);
template cudaError_t plan_arnoldi<float>(Krylov<float>&, size_t*);
template cudaError_t launch_arnoldi<double>(const Krylov<double>&, int, cudaStream_t);
template cudaError_t launch_arnoldi<float>(const Krylov<float>&, int, cudaStream_t);

}  // namespace dgk
