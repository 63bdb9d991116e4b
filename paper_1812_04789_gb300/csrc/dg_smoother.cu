// Persistent GMRES(BJ) smoother of the inherited coarse levels: one
// cooperative launch runs a whole SMOOTH / SOLVE call of Algorithm 2 (nu
// iterations of GMRES right-preconditioned by element block Jacobi, Sec. 6.3,
// on the inherited block-sparse operator of Sec. 6.1), where the
// launch-per-operation path takes about eleven small kernels per iteration.
//
// One CTA per SM owns a contiguous range of elements for the whole call and
// keeps its rows of the Krylov basis V, of the preconditioned directions Z and
// of the work vector w in shared memory (the coarse levels are small: a level
// whose rows do not fit keeps the launch-per-operation smoother), and, where
// they fit as well (p = 0), its blocks.
//
// The coarse levels are bound by the exchanges between the CTAs, not by
// arithmetic: with three grid barriers per iteration (an arrival counter, the
// last CTA summing the partials, a release word) an iteration took 23 us at
// p = 0 on 16^3 elements, of which the barriers were 14.  Two things bring
// that down.
//  * One reduction per iteration instead of two: Gram-Schmidt twice with the
//    second pass delayed (the low-synchronisation CGS2 of Swirydowicz et al.
//    2021 and Bielich et al. 2022).  Exchange j carries, beside V^T w for the
//    new column, V^T v_j for the second pass over v_j itself, v_j.v_j and w.w:
//      s = V^T v_j, beta^2 = v_j.v_j - s.s, v_j <- (v_j - V s) / beta,
//      h_i = V_i.w (i < j), h_j = (v_j.w - s.V^T w) / beta,
//      v_{j+1} = rho^{-1} (w - V h),  rho^2 = w.w - h.h (an estimate; a scale only)
//    and column j - 1 of the Hessenberg matrix, whose last vector was still
//    v_j's first pass, is completed: H_{i,j-1} += rho s_i, H_{j,j-1} = rho beta.
//    The directions z_j = D^{-1} v_j are those of the first pass: the outer
//    form is flexible (A Z = V H holds for any Z), so they need no second pass.
//  * No barriers: every value that another CTA needs travels with its epoch in
//    the same 8-byte element (dg_exchange.cuh), and the reader polls the value
//    itself.  The partial sums take two such hops (to the CTA that
//    owns the sum and back), the directions one, in place of arrival, sum,
//    release and read.  Epochs only grow (a word in device memory holds the next one), so
//    nothing is cleared between calls.  z_j's buffer is reused every
//    iteration (exchange j ends only after every CTA has consumed z_j), the
//    partials' buffer every second one.
// Per iteration j:
//   w = A z_j (own rows; the neighbours' z_j polled), partials        | exchange
//   second pass for v_j, v_{j+1}, z_{j+1} = D^{-1} v_{j+1} published
// The sums over the CTAs, the squared norms, their differences and roots and a new
// Hessenberg column are FP64 and in a fixed order, the column rounded once when
// it is complete; all CTAs hold identical scalars and the final x += Z y needs no
// exchange.  The arithmetic inside a CTA is FP32.  A warp of its own
// keeps the Hessenberg matrix, the Givens rotations (behind the next
// exchange's wait) and the small least-squares solve off the critical path;
// one warp takes the scalars of an exchange.
// 16^3 elements, p_fine = 4 (us per call, means over ten allocations): p = 2, nu
// = 10: 880 -> 746; p = 1, nu = 10: 400 -> 180; p = 0, nu = 30: 690 -> 265.
// FP64 handles run the same kernel on FP64 vectors and blocks.  Bound by the FP64 pipe at p = 2 (the block-sparse product), by the
// exchanges below; the launch-per-operation smoother spent half of its time
// on kernels of 2 to 5 us.  9 x 10 x 12, p = 3: FP64 step 116 -> 85 ms.
//
// Every wait is bounded (2 s of the global timer): on expiry the CTA sets
// ST_TIMEOUT in the mesh status word and returns, and the other CTAs see the
// flag while they wait and return too; a launch that finds ST_TIMEOUT already
// set returns at once.  A handle whose status shows ST_TIMEOUT has an
// unfinished smoother result: the application is untrusted until the status
// is cleared (dg_status_sync) and the preconditioner refreshed.
#include <math.h>

#include <algorithm>

#include "dg_exchange.cuh"

namespace dgk {

// R consecutive rows of one column of a column-major block from 16 bytes, from
// device memory (streamed) or, RES, from shared memory.
template <class S>
struct Col16;
template <>
struct Col16<float> {
  static constexpr int R = 4;
  template <bool RES>
  __device__ __forceinline__ static void load(const float* p, float* v) {
    if constexpr (RES) {
      const float4 t = *reinterpret_cast<const float4*>(p);
      v[0] = t.x;
      v[1] = t.y;
      v[2] = t.z;
      v[3] = t.w;
    } else {
      asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                   : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                   : "l"(p));
    }
  }
};
template <>
struct Col16<double> {
  static constexpr int R = 2;
  template <bool RES>
  __device__ __forceinline__ static void load(const double* p, double* v) {
    if constexpr (RES) {
      const double2 t = *reinterpret_cast<const double2*>(p);
      v[0] = t.x;
      v[1] = t.y;
    } else {
      asm volatile("ld.global.nc.L1::no_allocate.v2.f64 {%0,%1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "l"(p));
    }
  }
};
template <>
struct Col16<unsigned short> {
  static constexpr int R = 8;
  template <bool RES>
  __device__ __forceinline__ static void load(const unsigned short* p, float* v) {
    if constexpr (RES) {
      const uint4 t = *reinterpret_cast<const uint4*>(p);
      const unsigned w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[2 * k] = __uint_as_float(w[k] << 16);
        v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
      }
    } else {
      ld_bf16x8(p, v);
    }
  }
};

// the vectors' type over blocks stored as S
template <class S>
struct CoopVal {
  using V = float;
};
template <>
struct CoopVal<double> {
  using V = double;
};

template <class S>
struct CoopArgs {
  using V = typename CoopVal<S>::V;
  const S* Dinv;        // inverse diagonal blocks, column-major, leading dimension ld, nb * ld apart
  const S* Dop;         // inherited diagonal blocks (same layout)
  const S* O;           // inherited neighbour blocks [E][nf] (same layout)
  const int* nbr;       // [E][nf]
  const V* b;
  V* x;
  typename Xch<V>::Z* zx;     // [N] the direction z_j
  typename Xch<V>::P* px;     // [2][ni][grid + 1] the CTAs' partial sums
  Pair64* sums;               // [2][ni][SUM_STRIDE] their sums over the CTAs
  unsigned* epoch;      // first free epoch - 1
  int* status;          // mesh status word (ST_TIMEOUT)
  int* kflag;           // Krylov status bits (ST_NONFINITE)
  int nu, nb, ld, E, chunk, epc, tpe, ns, ni, extra;
  int pre;              // ask for the blocks ahead of their use (a level that L2 holds)
};

constexpr int COOP_WORK = 512;                  // threads that compute
constexpr int COOP_THREADS = COOP_WORK + 32;    // and the scalar warp

// Start bringing `bytes` (a multiple of 16, 16-byte aligned) into L2.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// The CTA's partial sums of exchange j, a warp per item: (V_i.v_j, V_i.w) for
// i <= j and (w.w, 0), in the vectors' precision (a lane's rows, then the warp's butterfly),
// published as they are ready; w = null (the closing exchange): zeros for w.
template <class V>
__device__ void publish_dots(int j, const V* Vs, int ldv, const V* w, int rows, typename Xch<V>::P* out, int stride,
                             unsigned ep) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= COOP_WORK / 32) return;
  const V* vj = Vs + (size_t)j * ldv;
  for (int i = warp; i < j + 2; i += COOP_WORK / 32) {
    const V* v = i <= j ? Vs + (size_t)i * ldv : w;
    V fs = V(0), ft = V(0);
    if (v) {
      for (int r = lane; r < rows; r += 32) {
        const V x = v[r];
        if (i <= j) {
          fs = fma(x, vj[r], fs);
          if (w) ft = fma(x, w[r], ft);
        } else {
          fs = fma(x, x, fs);
        }
      }
    }
    warp_sum2(fs, ft);
    if (lane == 0) Xch<V>::stp(out + (size_t)i * stride, fs, ft, ep);
  }
}

// The scalars of exchange j (see the head of the file), by one warp from the
// sums in st: FP64 square roots and sums in all seventeen warps would cost more
// than the exchange (two FP64 lanes per SM; an instruction holds its warp for 64
// clocks, so what can be is one instruction on two lanes' values, and no lane
// leaves the others).  sv: the sums rounded to V (FP64 vectors take st).  rho is
// a scale only: a power of two, whose reciprocal is exact, near the norm as
// estimated in V.
template <class V>
struct Scal {
  V ib, hj, ir;
  double beta, hjd, rho;
  int fine, bad;
};
template <class V>
__device__ void exchange_scalars(const double2* st, typename Xch<V>::V2* sv, int j, Scal<V>* sc) {
  const int lane = threadIdx.x & 31;
  double be2 = 0.0, hb = 0.0;     // v_j.v_j - s.s, v_j.w - s.V^T w
  V tq = V(0), ww = V(0);
  for (int i0 = 0; i0 < j + 2; i0 += 32) {
    const int i = i0 + lane;
    const double2 q = st[min(i, j + 1)];
    typename Xch<V>::V2 r;
    r.x = (V)q.x;
    r.y = (V)q.y;
    if (sizeof(V) == 4 && i < j + 2) sv[i] = r;
    // below j minus the product, at j the sum itself
    const double a = i < j ? -q.x : 1.0;
    be2 = fma(a, i <= j ? q.x : 0.0, be2);
    hb = fma(a, i <= j ? q.y : 0.0, hb);
    const V t = i < j ? r.y : V(0);
    tq = fma(t, t, tq);
    ww = i == j + 1 ? r.x : ww;
  }
  warp_sum2(be2, hb);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tq += __shfl_xor_sync(0xffffffffu, tq, o);
  ww = __shfl_sync(0xffffffffu, ww, (j + 1) & 31);
  const bool fine = be2 > 0.0 && isfinite(be2);
  const double ib = rsqrt(fine ? be2 : 1.0);
  const double pr = (lane == 0 ? be2 : hb) * ib;       // beta, h_j
  const V cv = (V)(lane == 0 ? ib : pr);
  const V hj = __shfl_sync(0xffffffffu, cv, 1);
  const V est = fmax(ww - tq - hj * hj, V(1e-6) * ww);
  const bool use = est > V(0) && isfinite(est);
  int e;       // |e| <= 512, FP32 64
  if constexpr (std::is_same<V, double>::value)
    e = use ? ((__double2hiint(est) >> 20) - 1023) >> 1 : 0;
  else
    e = use ? ((__float_as_int(est) >> 23) - 127) >> 1 : 0;
  if (lane < 2) {
    double* o = lane == 0 ? &sc->beta : &sc->hjd;
    V* v = lane == 0 ? &sc->ib : &sc->hj;
    *o = pr;
    *v = cv;
    sc->rho = __hiloint2double((1023 + e) << 20, 0);
    if constexpr (std::is_same<V, double>::value)
      sc->ir = __hiloint2double((1023 - e) << 20, 0);
    else
      sc->ir = __int_as_float((127 - e) << 23);
    sc->fine = fine;
    sc->bad = !fine && !isfinite(be2);
  }
}

// Column k of the Hessenberg matrix, complete, through the rotations before it and one of its own (one lane)
template <class V>
__device__ void rotate_column(V* H, int ldh, int k, V* cs, V* sn, V* g) {
  V* h = H + (size_t)k * ldh;
  V p = h[0];
  for (int i = 0; i < k; ++i) {
    const V q = h[i + 1];
    h[i] = cs[i] * p + sn[i] * q;
    p = -sn[i] * p + cs[i] * q;
  }
  const V q = h[k + 1];
  V c = V(1), sv = V(0);
  if constexpr (std::is_same<V, double>::value) {
    const V r2 = p * p + q * q;
    if (r2 > V(0)) {
      const V ir = rsqrt(r2);
      c = p * ir;
      sv = q * ir;
    }
  } else {
    const V rr = hypotf(p, q);
    if (rr != 0.f) {
      c = p / rr;
      sv = q / rr;
    }
  }
  cs[k] = c;
  sn[k] = sv;
  h[k] = c * p + sv * q;
  g[k + 1] = -sv * g[k];
  g[k] = c * g[k];
}

// The inputs of the block-sparse product for the CTA's elements p0 .. p0 + nl:
// xs[el][who][nb], who = 0 the element itself, 1 + s its neighbour on face s.
// own = null: from the vector in (no epochs); else own rows from `own`
// (shared memory) and the others' from zx, polled for epoch ep.
template <class V>
__device__ bool stage_inputs(const int* src, int nsrc, int p0, int nl, int nb, float inv_nb, int e_beg, int ne,
                             const V* in, const V* own, const typename Xch<V>::Z* zx, unsigned ep, int* status, V* xs) {
  using X = Xch<V>;
  bool ok = true;
  if (threadIdx.x >= COOP_WORK) return ok;
  Wait wt;
  const int n = nl * nsrc * nb;
  for (int t0 = threadIdx.x; t0 < n; t0 += 4 * COOP_WORK) {
    typename X::Z v[4];
    const typename X::Z* ad[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = t0 + u * COOP_WORK;
      ad[u] = nullptr;
      if (t >= n) continue;
      const int pair = (int)(((float)t + 0.5f) * inv_nb), j = t - pair * nb;   // exact: t < 2^20
      const int e = src[p0 * nsrc + pair];
      if (!own) {
        xs[t] = __ldcg(in + (size_t)e * nb + j);
      } else if ((unsigned)(e - e_beg) < (unsigned)ne) {
        xs[t] = own[(e - e_beg) * nb + j];
      } else {
        ad[u] = zx + (size_t)e * nb + j;
        v[u] = X::ld(ad[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (!ad[u]) continue;
      while (ok && !X::has(v[u], ep)) {
        if (wt.expired(status)) ok = false;
        v[u] = X::ld(ad[u]);
      }
      xs[t0 + u * COOP_WORK] = X::val(v[u]);
    }
  }
  return ok;
}

// acc[R] += rows of one column-major block times x, a run of columns' loads in
// flight together.  The last, shorter run reads the last column again (times
// zero): with a test around each load, or a loop over the remaining columns,
// every load waits for the one before it.
template <class S, bool RES, class V>
__device__ __forceinline__ void col_run(const S* B, int nb, int ld, const V* x, V* acc) {
  constexpr int R = Col16<S>::R, U = sizeof(V) == 8 ? 12 : 48 / R;
  for (int c0 = 0; c0 < nb; c0 += U) {
    V v[U][R], xv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int c = min(c0 + u, nb - 1);
      Col16<S>::template load<RES>(B + (size_t)c * ld, v[u]);
      xv[u] = c0 + u < nb ? x[c] : V(0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (sizeof(V) == 4 || c0 + u < nb)     // (FP64: its pipe is the limit)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[j] = fma(v[u][j], xv[u], acc[j]);
  }
}

// acc[R] = rows R tt .. of (D_e x_e + sum_s O_{e,s} x_nbr) over the blocks
// [b0, b1) of one element: all blocks of a column in flight together where
// one thread takes them all, else block by block with a run of columns in
// flight.  rev: columns from the last to the first (the next product finds
// the last ones of this one in L2).
template <class S, int NF, bool RES, class V>
__device__ __forceinline__ void bsr_rows(const S* D, const S* O, int nb, int ld, size_t bs, int b0, int b1, bool rev,
                                         const V* xe, V* acc) {
  constexpr int R = Col16<S>::R, NSRC = 1 + NF;
#pragma unroll
  for (int j = 0; j < R; ++j) acc[j] = V(0);
  if (b0 == 0 && b1 == NSRC) {
    const S* base[NSRC];
    base[0] = D;
#pragma unroll
    for (int b = 1; b < NSRC; ++b) base[b] = O + (size_t)(b - 1) * bs;
#pragma unroll 2
    for (int c_ = 0; c_ < nb; ++c_) {
      const int c = rev ? nb - 1 - c_ : c_;
      V v[NSRC][R];
#pragma unroll
      for (int b = 0; b < NSRC; ++b) Col16<S>::template load<RES>(base[b] + (size_t)c * ld, v[b]);
#pragma unroll
      for (int b = 0; b < NSRC; ++b) {
        const V xv = xe[b * nb + c];
#pragma unroll
        for (int j = 0; j < R; ++j) acc[j] = fma(v[b][j], xv, acc[j]);
      }
    }
  } else {
    for (int b = b0; b < b1; ++b)
      col_run<S, RES>(b == 0 ? D : O + (size_t)(b - 1) * bs, nb, ld, xe + b * nb, acc);
  }
}

template <class S, int NF, bool RES>
__global__ void __launch_bounds__(COOP_THREADS, 1) coop_smooth_kernel(CoopArgs<S> a) {
  using V = typename CoopVal<S>::V;
  using X = Xch<V>;
  constexpr int R = Col16<S>::R, NSRC = 1 + NF;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nu = a.nu, ldh = nu + 1, nb = a.nb, ld = a.ld, tpe = a.tpe, ns = a.ns;
  const size_t bs = (size_t)nb * ld;
  const int rmax = a.chunk * nb;
  S* Rs = reinterpret_cast<S*>(smem_raw);             // RES: [chunk][Dop, O.., Dinv]
  V* Vs = reinterpret_cast<V*>(Rs + (RES ? (size_t)a.chunk * (NSRC + 1) * bs : 0));   // [nu + 1][rmax]
  V* Zs = Vs + (size_t)ldh * rmax;                // [nu][rmax]
  V* ws = Zs + (size_t)nu * rmax;                 // [rmax]
  V* ps = ws + rmax;                              // ns > 1: [ns][rmax] partial products
  V* xs = ps + (ns > 1 ? (size_t)ns * rmax : 0);  // [epc][NSRC][nb]
  V* H = xs + (size_t)a.epc * NSRC * nb;          // (nu + 1) x nu, column-major
  V* cs = H + (size_t)ldh * nu;
  V* sn = cs + nu;
  V* g = sn + nu;                                 // nu + 1, then y
  int* src = reinterpret_cast<int*>(g + ldh);         // [chunk][NSRC] element ids
  double2* st = reinterpret_cast<double2*>((reinterpret_cast<uintptr_t>(src + (size_t)a.chunk * NSRC) + 15) & ~(uintptr_t)15);   // [nu + 2]
  double* hd = reinterpret_cast<double*>(st + nu + 2);   // [nu + 1] the Hessenberg column begun
  typename X::V2* sv = sizeof(V) == 4 ? reinterpret_cast<typename X::V2*>(hd + ldh) : reinterpret_cast<typename X::V2*>(st);   // st in V
  __shared__ int timed_out;
  __shared__ Scal<V> scal;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, G = gridDim.x;
  const bool scalar_warp = warp == COOP_WORK / 32;
  const int e_beg = min(a.E, (int)blockIdx.x * a.chunk), ne = min(a.E, e_beg + a.chunk) - e_beg;
  const int rows = ne * nb;
  const float inv_nb = 1.0f / (float)nb;
  if (tid == 0) timed_out = (*(volatile int*)a.status & ST_TIMEOUT) ? 1 : 0;
  const unsigned base = *(volatile unsigned*)a.epoch;   // advanced at the end, after every CTA has read it
  for (int t = tid; t < ne * NSRC; t += COOP_THREADS) {
    const int el = t / NSRC, who = t - el * NSRC, e = e_beg + el;
    src[t] = who == 0 ? e : a.nbr[(size_t)e * NF + who - 1];
  }
  if constexpr (RES) {
    constexpr int V16 = 16 / sizeof(S);
    const int per = (int)(bs / V16);                  // 16-byte words per block
    uint4* dst = reinterpret_cast<uint4*>(Rs);
    for (int t = tid; t < ne * (NSRC + 1) * per; t += COOP_THREADS) {
      const int blk = t / per, q = t - blk * per, el = blk / (NSRC + 1), b = blk - el * (NSRC + 1);
      const size_t e = e_beg + el;
      const S* p = b == 0 ? a.Dop + e * bs : (b <= NF ? a.O + (e * NF + b - 1) * bs : a.Dinv + e * bs);
      dst[t] = __ldg(reinterpret_cast<const uint4*>(p) + q);
    }
  }
  __syncthreads();
  if (timed_out) return;   // an earlier wait ran out: leave x as it is
#define COOP_LEAVE_IF(fail)                                                       \
  if (__syncthreads_or((fail) ? 1 : 0)) {                                         \
    if (tid == 0) atomicMax(a.epoch, base + (unsigned)nu + 8u);                   \
    return;                                                                       \
  }

  // out = A in, or b - A in, on own rows
  const int span = a.epc * tpe, sp = tid / span, sub = (tid - sp * span) / tpe, tt = tid - sp * span - sub * tpe;
  const int bb0 = sp * NSRC / ns, bb1 = (sp + 1) * NSRC / ns;
#define COOP_PRODUCT(own, ep, bsub, out, rev)                                                             \
  for (int p0 = 0; p0 < ne; p0 += a.epc) {                                                                \
    const int nl = min(a.epc, ne - p0);                                                                   \
    const bool got = stage_inputs<V>(src, NSRC, p0, nl, nb, inv_nb, e_beg, ne, a.x, own, a.zx, ep, a.status, xs); \
    COOP_LEAVE_IF(!got)                                                                                   \
    if (sp < ns && sub < nl) {                                                                     \
      const int el = p0 + sub;                                                                            \
      const size_t e = e_beg + el;                                                                        \
      const S* D = (RES ? Rs + (size_t)el * (NSRC + 1) * bs : a.Dop + e * bs) + R * tt;                   \
      const S* O = (RES ? Rs + ((size_t)el * (NSRC + 1) + 1) * bs : a.O + e * NF * bs) + R * tt;          \
      V acc[R];                                                                                           \
      bsr_rows<S, NF, RES>(D, O, nb, ld, bs, bb0, bb1, rev, xs + (size_t)sub * NSRC * nb, acc);           \
      const int r0 = el * nb + R * tt;                                                                    \
      _Pragma("unroll") for (int k = 0; k < R; ++k) if (R * tt + k < nb) {                                \
        if (ns > 1)                                                                                       \
          ps[(size_t)sp * rmax + r0 + k] = acc[k];                                                        \
        else                                                                                              \
          out[r0 + k] = bsub ? __ldcg(bsub + (size_t)e_beg * nb + r0 + k) - acc[k] : acc[k];              \
      }                                                                                                   \
    }                                                                                                     \
    __syncthreads();                                                                                      \
  }                                                                                                       \
  if (ns > 1) {                                                                                           \
    for (int r = tid; r < rows; r += COOP_THREADS) {                                                      \
      V t = ps[r];                                                                                        \
      for (int k = 1; k < ns; ++k) t += ps[(size_t)k * rmax + r];                                         \
      out[r] = bsub ? __ldcg(bsub + (size_t)e_beg * nb + r) - t : t;                                      \
    }                                                                                                     \
    __syncthreads();                                                                                      \
  }

  // v_0 = r = b - A x, not normalised (exchange 0 brings its norm)
  {
    const V* none = nullptr;
    COOP_PRODUCT(none, 0u, a.b, Vs, false)
  }
  double rho = 1.0;         // |w - V h| as estimated: v_{j+1} = (w - V h) / rho
  int kdone = 0;
  for (int j = 0;; ++j) {
    const unsigned ep = base + 1u + (unsigned)j;
    V* vj = Vs + (size_t)j * rmax;
    if (j < nu) {
      // the blocks of the coming product, meanwhile (see CoopArgs::pre)
      const bool rev = (j & 1) == 0;
      if constexpr (!RES) {
        if (a.pre)
          for (int t = tid; t < ne * NSRC; t += COOP_THREADS) {
            const int el = t / NSRC, k = t - el * NSRC;
            const size_t e = e_beg + el;
            prefetch_l2(k == 0 ? a.Dop + e * bs : a.O + (e * NF + k - 1) * bs, (unsigned)(bs * sizeof(S)));
          }
      }
      // z_j = D^{-1} v_j: own rows to shared memory, published for the neighbours
      V* zs = Zs + (size_t)j * rmax;
      const int bsub_ = tid / tpe, btt = tid - bsub_ * tpe, bep = COOP_WORK / tpe;
      if (bsub_ < bep) {
        for (int el = bsub_; el < ne; el += bep) {
          const size_t e = e_beg + el;
          const S* M = (RES ? Rs + ((size_t)el * (NSRC + 1) + NSRC) * bs : a.Dinv + e * bs) + R * btt;
          const V* xe = vj + (size_t)el * nb;
          V acc[R];
#pragma unroll
          for (int k = 0; k < R; ++k) acc[k] = V(0);
          col_run<S, RES>(M, nb, ld, xe, acc);
          const int r0 = el * nb + R * btt;
#pragma unroll
          for (int k = 0; k < R; ++k)
            if (R * btt + k < nb) {
              zs[r0 + k] = acc[k];
              X::st(a.zx + (size_t)e_beg * nb + r0 + k, acc[k], ep);
            }
        }
      }
      __syncthreads();
      // w = A z_j
      const V* none = nullptr;
      COOP_PRODUCT(zs, ep, none, ws, rev)
    }
    // exchange j
    if constexpr (!RES) {
      if (j < nu && a.pre)
        for (int el = tid; el < ne; el += COOP_THREADS)
          prefetch_l2(a.Dinv + (size_t)(e_beg + el) * bs, (unsigned)(bs * sizeof(S)));
    }
    typename X::P* px = a.px + (size_t)(j & 1) * (G + 1) * a.ni;
    publish_dots<V>(j, Vs, rmax, j < nu ? ws : nullptr, rows, px + blockIdx.x, G + 1, ep);
    bool got = true;
    if (scalar_warp) {
      if (j >= 2 && lane == 0) rotate_column(H, ldh, j - 2, cs, sn, g);   // behind the exchange
    } else {
      got = gather_dots<V, COOP_WORK / 32>(px, G + 1, j + 2, G + a.extra, a.sums + (j & 1) * a.ni * SUM_STRIDE, ep, a.status, st);
      if (warp == 0) exchange_scalars<V>(st, sv, j, &scal);
    }
    COOP_LEAVE_IF(!got)
    const bool fine = scal.fine;
    const V ib = scal.ib, hj = scal.hj;
    if (scalar_warp) {
      // column j - 1 completed, column j begun (this warp alone)
      if (j == 0) {
        for (int i = lane; i < ldh; i += 32) g[i] = i == 0 && fine ? (V)scal.beta : V(0);
      } else {
        V* h = H + (size_t)(j - 1) * ldh;
        for (int i = lane; i < j; i += 32) h[i] = (V)fma(rho, st[i].x, hd[i]);
        if (lane == 0) h[j] = fine ? (V)(rho * scal.beta) : V(0);
      }
      if (j < nu && fine)
        for (int i = lane; i <= j; i += 32) hd[i] = i < j ? st[i].y : scal.hjd;
      __syncwarp();
    }
    kdone = j;
    if (!fine || j == nu) {   // the Krylov space is exhausted (or not finite), or complete
      if (scal.bad && tid == 0 && blockIdx.x == 0) atomicOr(a.kflag, ST_NONFINITE);
      break;
    }
    rho = scal.rho;
    const V ir = scal.ir;
    if (tid < COOP_WORK) {
      V* vn = vj + rmax;
      for (int r = tid; r < rows; r += COOP_WORK) {
        V v = vj[r], w = ws[r];
        const V* q = Vs + r;
#pragma unroll 8
        for (int i = 0; i < j; ++i) {
          const typename X::V2 c = sv[i];
          const V vi = q[(size_t)i * rmax];
          v = fma(-c.x, vi, v);
          w = fma(-c.y, vi, w);
        }
        v *= ib;
        vj[r] = v;
        vn[r] = fma(-hj, v, w) * ir;
      }
    }
    __syncthreads();
  }
  if (blockIdx.x == 0 && tid == 0) *(volatile unsigned*)a.epoch = base + (unsigned)nu + 8u;
  if (kdone == 0) return;   // b - A x = 0 (or not finite): nothing to smooth
  // y = H[:k,:k]^{-1} g[:k] (into g; the scalar warp, which rotated it), x += Z y on own rows
  if (scalar_warp) {
    if (lane == 0) rotate_column(H, ldh, kdone - 1, cs, sn, g);
    __syncwarp();
    for (int i = lane; i < kdone; i += 32) {    // the diagonal's reciprocals at once (into cs)
      const V d = H[(size_t)i * ldh + i];
      cs[i] = d != V(0) ? V(1) / d : V(0);
    }
    __syncwarp();
    for (int i = kdone - 1; i >= 0; --i) {
      const V y = g[i] * cs[i];
      __syncwarp();
      for (int c = lane; c < i; c += 32) g[c] = fma(-H[(size_t)i * ldh + c], y, g[c]);
      if (lane == 0) g[i] = y;
      __syncwarp();
    }
  }
  __syncthreads();
  V* xo = a.x + (size_t)e_beg * nb;
  for (int r = tid; r < rows; r += COOP_THREADS) {
    V acc = xo[r];
    for (int i = 0; i < kdone; ++i) acc = fma(g[i], Zs[(size_t)i * rmax + r], acc);
    xo[r] = acc;
  }
#undef COOP_PRODUCT
#undef COOP_LEAVE_IF
}

// dynamic shared memory in bytes; res: with the CTA's blocks
template <class S>
static size_t coop_smem(int nu, int nb, int ld, int nf, int chunk, int epc, int ns, bool res) {
  const size_t ldh = nu + 1, rmax = (size_t)chunk * nb;
  const size_t fl = ldh * rmax + nu * rmax + rmax + (ns > 1 ? ns * rmax : 0) + (size_t)epc * (1 + nf) * nb +
                    ldh * nu + 2 * (size_t)nu + ldh;
  using V = typename CoopVal<S>::V;
  const size_t sc = (2 * (nu + 2) + ldh) * sizeof(double) + (sizeof(V) == 4 ? 2 * (nu + 2) * sizeof(V) : 0);
  return fl * sizeof(V) + sizeof(int) * (size_t)chunk * (1 + nf) + 16 + sc +
         (res ? (size_t)chunk * (2 + nf) * nb * ld * sizeof(S) : 0);
}

template <class S, int NF>
static cudaError_t plan_coop(int nb, int ld, int E, int nu, CoopPlan* plan) {
  constexpr int R = Col16<S>::R;
  plan->ok = 0;
  if (ld % R || E < 1) return cudaSuccess;
  const int tpe = ld / R;
  if (tpe > COOP_WORK) return cudaSuccess;
  int dev = 0, nsm = 0, smax = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (nsm < 1) return cudaSuccess;
  int grid = std::min(E, nsm);
  const int chunk = (E + grid - 1) / grid;
  grid = (E + chunk - 1) / chunk;   // no CTA without elements
  const int epc = std::max(1, std::min(chunk, COOP_WORK / tpe));
  // where one thread per (element, rows) leaves most of the CTA idle, an
  // element's 1 + nf blocks are shared out over ns threads (p = 1, p = 0:
  // chains of dependent loads, not bandwidth)
  const int ns = epc < chunk ? 1 : std::max(1, std::min(1 + NF, COOP_WORK / (epc * tpe)));
  // a level whose blocks stay in L2 from one product to the next has them asked
  // for during the phases before (p = 1 on 16^3: 223 -> 190 us a call; 100 x 75
  // quads, p = 2: 290 -> 243); the blocks of a larger level come from DRAM
  // every time, and asking for them all at once only evicts what comes first
  // (p = 2 on 16^3, 328 MB: 745 -> 985 us)
  int l2 = 0;
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
  const int pre = (double)E * (2 + NF) * nb * ld * sizeof(S) <= 0.85 * l2 ? 1 : 0;
  if ((long)epc * (1 + NF) * nb >= (1 << 20)) return cudaSuccess;   // stage_inputs' exact index range
  for (int res = 1; res >= 0; --res) {
    const size_t smem = coop_smem<S>(nu, nb, ld, NF, chunk, epc, ns, res);
    auto kern = res ? coop_smooth_kernel<S, NF, true> : coop_smooth_kernel<S, NF, false>;
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    if (smem + fa.sharedSizeBytes > (size_t)smax) continue;   // rows only; then the per-operation smoother
    e = allow_max_smem(kern);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, COOP_THREADS, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) continue;
    plan->ok = 1;
    plan->nu_max = nu;
    plan->grid = grid;
    plan->chunk = chunk;
    plan->epc = epc;
    plan->tpe = tpe;
    plan->ns = ns;
    plan->pre = pre;
    plan->res = res;
    plan->smem = smem;
    using X = Xch<typename CoopVal<S>::V>;
    plan->part_bytes = sizeof(typename X::P) * 2 * (size_t)(grid + 1) * (nu + 2) + sizeof(Pair64) * 2 * (nu + 2) * SUM_STRIDE;
    plan->z_bytes = sizeof(typename X::Z) * (size_t)E * nb;
    return cudaSuccess;
  }
  return cudaSuccess;
}

cudaError_t plan_coop_smoother(int store, int nb, int nf, int E, int nu, CoopPlan* plan) {
  plan->ok = 0;
#define GO(NF)                                                                                     \
  return store == COOP_BF16   ? plan_coop<unsigned short, NF>(nb, ld_bf16(nb), E, nu, plan)       \
         : store == COOP_FP64 ? plan_coop<double, NF>(nb, inv_ld<double>(nb), E, nu, plan)        \
                              : plan_coop<float, NF>(nb, inv_ld<float>(nb), E, nu, plan)
  if (nf == 6) GO(6);
  if (nf == 4) GO(4);
  if (nf == 3) GO(3);
#undef GO
  return cudaSuccess;   // other face counts keep the launch-per-operation smoother
}

template <class S, int NF>
static cudaError_t launch_coop(const CoopPlan& pl, const S* Dinv, const S* Dop, const S* O, int ld, const int* nbr,
                               const typename CoopVal<S>::V* b, typename CoopVal<S>::V* x, int nu,
                               Krylov<typename CoopVal<S>::V>& K, const CoopBuffers& buf, int* status, int extra,
                               int nb, int E, cudaStream_t st) {
  using X = Xch<typename CoopVal<S>::V>;
  CoopArgs<S> a;
  a.Dinv = Dinv;
  a.Dop = Dop;
  a.O = O;
  a.nbr = nbr;
  a.b = b;
  a.x = x;
  a.zx = (typename X::Z*)buf.z;
  a.px = (typename X::P*)buf.part;
  a.sums = (Pair64*)(a.px + 2 * (size_t)(pl.grid + 1) * (pl.nu_max + 2));
  a.epoch = buf.epoch;
  a.status = status;
  a.kflag = K.kdim + 1;
  a.nu = nu;
  a.nb = nb;
  a.ld = ld;
  a.E = E;
  a.chunk = pl.chunk;
  a.epc = pl.epc;
  a.tpe = pl.tpe;
  a.ns = pl.ns;
  a.ni = pl.nu_max + 2;
  a.extra = extra > 0 ? 1 : 0;
  a.pre = pl.pre;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pl.grid);
  cfg.blockDim = dim3(COOP_THREADS);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  note_launch();
  if (pl.res) return cudaLaunchKernelEx(&cfg, coop_smooth_kernel<S, NF, true>, a);
  return cudaLaunchKernelEx(&cfg, coop_smooth_kernel<S, NF, false>, a);
}

cudaError_t launch_coop_smoother(const CoopPlan& pl, const float* Dinv, const float* Dop, const float* O,
                                 const unsigned short* Dinv16, const unsigned short* Dop16, const unsigned short* O16,
                                 const int* nbr, int nf, const float* b, float* x, int nu, Krylov<float>& K,
                                 const CoopBuffers& buf, int* status, int extra, int nb, int E, cudaStream_t st) {
  if (!pl.ok || nu < 1 || nu > pl.nu_max || nu > K.nmax) return cudaErrorInvalidValue;
#define GO(NF)                                                                                                     \
  return Dinv16 ? launch_coop<unsigned short, NF>(pl, Dinv16, Dop16, O16, ld_bf16(nb), nbr, b, x, nu, K, buf, status, \
                                                  extra, nb, E, st)                                                \
                : launch_coop<float, NF>(pl, Dinv, Dop, O, inv_ld<float>(nb), nbr, b, x, nu, K, buf, status, extra,   \
                                         nb, E, st)
  if (nf == 6) GO(6);
  if (nf == 4) GO(4);
  if (nf == 3) GO(3);
#undef GO
  return cudaErrorInvalidValue;
}

cudaError_t launch_coop_smoother(const CoopPlan& pl, const double* Dinv, const double* Dop, const double* O,
                                 const unsigned short*, const unsigned short*, const unsigned short*, const int* nbr,
                                 int nf, const double* b, double* x, int nu, Krylov<double>& K, const CoopBuffers& buf,
                                 int* status, int extra, int nb, int E, cudaStream_t st) {
  if (!pl.ok || nu < 1 || nu > pl.nu_max || nu > K.nmax) return cudaErrorInvalidValue;
#define GO(NF) \
  return launch_coop<double, NF>(pl, Dinv, Dop, O, inv_ld<double>(nb), nbr, b, x, nu, K, buf, status, extra, nb, E, st)
  if (nf == 6) GO(6);
  if (nf == 4) GO(4);
  if (nf == 3) GO(3);
#undef GO
  return cudaErrorInvalidValue;
}

}  // namespace dgk
