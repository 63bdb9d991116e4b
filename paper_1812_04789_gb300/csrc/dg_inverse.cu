// Batched inverse of the element blocks for block Jacobi (Sec. 6.3: the
// element-block smoother's factorisation, here an explicit inverse so that
// every application is one dense mat-vec per element).
//
// Gauss-Jordan elimination in place with partial pivoting: at step k the pivot
// is the largest |A[i][k]| over the rows i not yet used as pivots (the lowest
// row index on ties).  Rows are never swapped; after the n steps the matrix R
// holds the inverse with permuted rows and columns,
//   X[step(i)][prow(j)] = R[i][j],
// where prow(k) is the pivot row of step k and step(i) the step at which row i
// was the pivot.  A zero pivot marks the status word (the block is singular)
// and the step continues with pivot 1.
//
// Blocks come row-major, bstride elements apart.  The inverse leaves
// column-major with leading dimension ld = inv_ld(nb) (rows padded to a
// 16-byte multiple with zeros), the layout the block-Jacobi apply streams,
// except from the in-place global-memory path, which leaves it row-major.
//
// block_inverse_reg_kernel (nb < 40; nb <= 16 R): 256 threads as a 16 x 16 grid;
// thread (ty, tx) keeps the R x R entries of rows ty + 16 a and columns
// tx + 16 b in registers for the whole elimination, so a step costs R^2 FMAs
// per thread plus two shared-memory vectors (the pivot row and column) and
// three barriers.  The permuted, transposed result is staged in shared memory
// and written out coalesced.
// block_inverse_sm_kernel (blocks that fit shared memory with a panel): panels
// in registers, register-tiled updates in shared memory.
// block_inverse_blk_kernel (up to 512 rows): the same on the block in memory.
// block_inverse_kernel (the few sizes whose block fits shared memory without
// the panel): one warp per row in the update.  block_inverse_panel_kernel
// (blocks beyond 512 rows): panels of columns eliminated in shared memory, one
// rank-16 update of the block's other columns per panel.
#include <algorithm>
#include <climits>

#include "dg_internal.h"

namespace dgk {

namespace {

int num_sms_inv() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

// |x|, 0 for NaN, from the bits: a comparison with zero in floating point
// (fabs(x) >= 0 ? fabs(x) : 0) is folded to fabs(x) by the compiler, and a column
// of NaN (the blocks of an unphysical state) then had no pivot row at all
__device__ __forceinline__ float magnitude(float x) {
  const unsigned b = __float_as_uint(x) & 0x7fffffffu;
  return __uint_as_float(b > 0x7f800000u ? 0u : b);
}
__device__ __forceinline__ double magnitude(double x) {
  const long long b = __double_as_longlong(x) & 0x7fffffffffffffffll;
  return __longlong_as_double(b > 0x7ff0000000000000ll ? 0ll : b);
}
// whether candidate a is the better pivot of two (|value| larger, or equal with a
// lower row; INT_MAX: no candidate)
template <class T>
__device__ __forceinline__ bool better(T va, int ia, T vb, int ib) {
  return ib == INT_MAX ? ia != INT_MAX : va > vb || (va == vb && ia < ib);
}

template <class T, int R>
__global__ void __launch_bounds__(256, 1) block_inverse_reg_kernel(T* __restrict__ blocks, int nb,
                                                                   size_t bstride, long nblk, int* status) {
  constexpr int NP = 16 * R;
  __shared__ T colk[NP], prow[NP];
  __shared__ T cand_v[16], cand_s[16];
  __shared__ int cand_i[16];
  __shared__ int piv_row[NP], step_of[NP];
  __shared__ int s_p;
  __shared__ T s_piv;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* S = reinterpret_cast<T*>(smem_raw);   // nb * ld output staging (column-major)
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int ld = inv_ld<T>(nb), nl = nb * ld;
  for (long blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    T* Ag = blocks + (size_t)blk * bstride;
    T t[R][R];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) {
        const int i = ty + 16 * a, j = tx + 16 * b;
        t[a][b] = (i < nb && j < nb) ? Ag[(size_t)i * nb + j] : T(0);
      }
    unsigned used = 0;   // bit a: row ty + 16 a has been a pivot row
    bool bad = false;
    // k = 16 kb + kx: the register column kb is a compile-time index (the
    // unrolled kb loop), so reading and rewriting column k needs no selects
#pragma unroll
    for (int kb = 0; kb < R; ++kb)
    for (int kx = 0; kx < 16; ++kx) {
      const int k = 16 * kb + kx;
      if (k >= nb) break;
      T col[R];
#pragma unroll
      for (int a = 0; a < R; ++a) col[a] = t[a][kb];
      if (tx == kx) {   // the 16 owners of column k: best unused row of their R
        T best = T(-1), sv = T(0);
        int bi = INT_MAX;
#pragma unroll
        for (int a = 0; a < R; ++a) {
          const int i = ty + 16 * a;
          const T v = magnitude(col[a]);
          if (i < nb && !((used >> a) & 1u) && better(v, i, best, bi)) {
            best = v;
            bi = i;
            sv = col[a];
          }
        }
        cand_v[ty] = best;
        cand_i[ty] = bi;
        cand_s[ty] = sv;
      }
      __syncthreads();
      if (threadIdx.x < 32) {
        const int l = threadIdx.x;
        T v = l < 16 ? cand_v[l] : T(-1);
        int i = l < 16 ? cand_i[l] : INT_MAX;
        T sv = l < 16 ? cand_s[l] : T(0);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
          const T v2 = __shfl_down_sync(0xffffffffu, v, o);
          const int i2 = __shfl_down_sync(0xffffffffu, i, o);
          const T s2 = __shfl_down_sync(0xffffffffu, sv, o);
          if (better(v2, i2, v, i)) {
            v = v2;
            i = i2;
            sv = s2;
          }
        }
        if (l == 0) {
          s_p = i;
          s_piv = sv;
          piv_row[k] = i;
          step_of[i] = k;
        }
      }
      __syncthreads();
      const int p = s_p, pa = p >> 4;
      T piv = s_piv;
      if (!(fabs(piv) > T(0))) {
        bad = true;
        piv = T(1);
      }
      const T ipiv = T(1) / piv;
      if (ty == (p & 15)) {   // the pivot row, scaled; its column k entry becomes 1 / piv
#pragma unroll
        for (int a = 0; a < R; ++a)
          if (a == pa) {
#pragma unroll
            for (int b = 0; b < R; ++b) {
              const int j = tx + 16 * b;
              if (j < NP) prow[j] = (j == k) ? ipiv : t[a][b] * ipiv;
            }
          }
        used |= 1u << pa;
      }
      if (tx == kx) {
#pragma unroll
        for (int a = 0; a < R; ++a) {
          const int i = ty + 16 * a;
          colk[i] = (i == p) ? T(0) : col[a];
        }
      }
      __syncthreads();
      T pr[R], ck[R];
#pragma unroll
      for (int b = 0; b < R; ++b) pr[b] = prow[tx + 16 * b];
#pragma unroll
      for (int a = 0; a < R; ++a) ck[a] = colk[ty + 16 * a];
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) t[a][b] -= ck[a] * pr[b];
      if (ty == (p & 15)) {
#pragma unroll
        for (int a = 0; a < R; ++a)
          if (a == pa) {
#pragma unroll
            for (int b = 0; b < R; ++b) t[a][b] = pr[b];
          }
      }
      if (tx == kx) {
#pragma unroll
        for (int a = 0; a < R; ++a) {
          const int i = ty + 16 * a;
          t[a][kb] = (i == p) ? ipiv : -ck[a] * ipiv;
        }
      }
    }
    __syncthreads();   // piv_row / step_of complete
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) {
        const int i = ty + 16 * a, j = tx + 16 * b;
        if (i < nb && j < nb) S[(size_t)piv_row[j] * ld + step_of[i]] = t[a][b];
      }
    for (int e = threadIdx.x; e < nb * (ld - nb); e += blockDim.x) {
      const int c = e / (ld - nb);
      S[(size_t)c * ld + nb + (e - c * (ld - nb))] = T(0);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nl; e += blockDim.x) Ag[e] = S[e];
    if (bad && threadIdx.x == 0) atomicOr(status, ST_SINGULAR);
    __syncthreads();
  }
}

// Blocks too large for registers: the same elimination on a copy in shared
// memory (or in place in global memory).  One warp per row in the update.
template <class T>
__global__ void __launch_bounds__(256) block_inverse_kernel(T* __restrict__ blocks, int nb, size_t bstride,
                                                            long nblk, int use_smem, int* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // byte layout: colk[nb] | prow[nb] | piv_row[nb] | step_of[nb] | used[nb] | lead[nb] | A (16-aligned)
  T* colk = reinterpret_cast<T*>(smem_raw);
  T* prow = colk + nb;
  int* piv_row = reinterpret_cast<int*>(prow + nb);
  int* step_of = piv_row + nb;
  int* used = step_of + nb;
  int* lead = used + nb;
  __shared__ T wv[8], ws[8];
  __shared__ int wi[8];
  __shared__ int s_p;
  __shared__ T s_piv;
  T* As = reinterpret_cast<T*>((reinterpret_cast<uintptr_t>(lead + nb) + 15) & ~uintptr_t(15));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int nn = nb * nb;
  const int ld = inv_ld<T>(nb);
  for (long blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    T* Ag = blocks + (size_t)blk * bstride;
    T* A = use_smem ? As : Ag;
    if (use_smem)
      for (int e = threadIdx.x; e < nn; e += blockDim.x) A[e] = Ag[e];
    for (int i = threadIdx.x; i < nb; i += blockDim.x) used[i] = 0;
    __syncthreads();
    bool bad = false;
    for (int k = 0; k < nb; ++k) {
      T best = T(-1), sv = T(0);
      int bi = INT_MAX;
      for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        const T x = A[(size_t)i * nb + k], v = magnitude(x);
        if (!used[i] && better(v, i, best, bi)) {
          best = v;
          bi = i;
          sv = x;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const T v2 = __shfl_down_sync(0xffffffffu, best, o);
        const int i2 = __shfl_down_sync(0xffffffffu, bi, o);
        const T s2 = __shfl_down_sync(0xffffffffu, sv, o);
        if (better(v2, i2, best, bi)) {
          best = v2;
          bi = i2;
          sv = s2;
        }
      }
      if (lane == 0) {
        wv[warp] = best;
        wi[warp] = bi;
        ws[warp] = sv;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int w = 1; w < nw; ++w)
          if (better(wv[w], wi[w], best, bi)) {
            best = wv[w];
            bi = wi[w];
            sv = ws[w];
          }
        s_p = bi;
        s_piv = sv;
        piv_row[k] = bi;
        step_of[bi] = k;
        used[bi] = 1;
      }
      __syncthreads();
      const int p = s_p;
      T piv = s_piv;
      if (!(fabs(piv) > T(0))) {
        bad = true;
        piv = T(1);
      }
      const T ipiv = T(1) / piv;
      for (int j = threadIdx.x; j < nb; j += blockDim.x) prow[j] = (j == k) ? ipiv : A[(size_t)p * nb + j] * ipiv;
      for (int i = threadIdx.x; i < nb; i += blockDim.x) colk[i] = (i == p) ? T(0) : A[(size_t)i * nb + k];
      __syncthreads();
      for (int i = warp; i < nb; i += nw) {
        T* row = A + (size_t)i * nb;
        const T c = colk[i];
        if (i == p) {
          for (int j = lane; j < nb; j += 32) row[j] = prow[j];
        } else {
          for (int j = lane; j < nb; j += 32) row[j] = (j == k) ? -c * ipiv : row[j] - c * prow[j];
        }
      }
      __syncthreads();
    }
    // permute into the output: X[step_of[i]][piv_row[j]] = R[i][j], column-major
    if (use_smem) {
      for (int e = threadIdx.x; e < nn; e += blockDim.x) {
        const int i = e / nb, j = e - i * nb;
        Ag[(size_t)piv_row[j] * ld + step_of[i]] = A[e];
      }
      for (int e = threadIdx.x; e < nb * (ld - nb); e += blockDim.x) {
        const int c = e / (ld - nb);
        Ag[(size_t)c * ld + nb + (e - c * (ld - nb))] = T(0);
      }
    } else {
      // in place in global memory: the row permutation i -> step_of[i], then
      // the column permutation j -> piv_row[j], each applied cycle by cycle
      // (thread 0 marks every cycle's smallest index with the cycle length)
      for (int pass = 0; pass < 2; ++pass) {
        const int* to = pass == 0 ? step_of : piv_row;
        __syncthreads();
        if (threadIdx.x == 0) {
          for (int i = 0; i < nb; ++i) used[i] = 0;
          for (int i0 = 0; i0 < nb; ++i0) {
            lead[i0] = 0;
            if (used[i0]) continue;
            int c = i0, len = 0;
            do {
              used[c] = 1;
              c = to[c];
              ++len;
            } while (c != i0);
            lead[i0] = len > 1 ? len : 0;
          }
        }
        __syncthreads();
        for (int i0 = 0; i0 < nb; ++i0) {
          const int len = lead[i0];
          if (len == 0) continue;
          for (int x = threadIdx.x; x < nb; x += blockDim.x) {
            // pass 0 moves rows (x = column), pass 1 moves columns (x = row)
            const size_t str = pass == 0 ? (size_t)nb : 1, off = pass == 0 ? (size_t)x : (size_t)x * nb;
            T carry = A[off + (size_t)i0 * str];
            int src = i0;
            for (int s = 0; s < len; ++s) {
              const int dst = to[src];
              const T y = A[off + (size_t)dst * str];
              A[off + (size_t)dst * str] = carry;
              carry = y;
              src = dst;
            }
          }
        }
      }
    }
    if (bad && threadIdx.x == 0) atomicOr(status, ST_SINGULAR);
    __syncthreads();
  }
}

// Blocks too large for shared memory (nb = 420 at p = 6): Gauss-Jordan by
// panels of BP columns.  The BP elimination steps of a panel act on any other
// column x as x <- x + sum_c (X_c - e_{p_c}) x[p_c], where p_c is the pivot row
// of step c and X_c the panel's column c once the whole panel is eliminated
// (it is T e_{p_c}, T the product of the panel's steps: a GJ step changes a
// column only through its entry at the pivot row, and leaves e_i alone for a
// row i that is not the pivot).  So a panel is eliminated in shared memory
// (pivot search, the step on the panel's columns) and every other column of
// the block receives one rank-BP update, read and written once per panel
// instead of once per step.  Same pivot rule and in-place storage as above;
// the result is row-major, permuted in place at the end.
template <class T, int BP>
__global__ void __launch_bounds__(256) block_inverse_panel_kernel(T* __restrict__ blocks, int nb, size_t bstride,
                                                                  long nblk, int* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // byte layout: Pn[nb][BP] | piv_row[nb] | step_of[nb] | used[nb] | lead[nb]
  T* Pn = reinterpret_cast<T*>(smem_raw);
  int* piv_row = reinterpret_cast<int*>(Pn + (size_t)nb * BP);
  int* step_of = piv_row + nb;
  int* used = step_of + nb;
  int* lead = used + nb;
  __shared__ T wv[8], ws[8];
  __shared__ int wi[8];
  __shared__ int s_p;
  __shared__ T s_piv;
  __shared__ int pr[BP];          // pivot rows of the current panel
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (long blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    T* A = blocks + (size_t)blk * bstride;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) used[i] = 0;
    bool bad = false;
    for (int k0 = 0; k0 < nb; k0 += BP) {
      const int bw = min(BP, nb - k0);
      __syncthreads();
      for (int t = threadIdx.x; t < nb * BP; t += blockDim.x) {
        const int i = t / BP, c = t - i * BP;
        Pn[t] = c < bw ? A[(size_t)i * nb + k0 + c] : T(0);
      }
      __syncthreads();
      for (int c = 0; c < bw; ++c) {
        const int k = k0 + c;
        T best = T(-1), sv = T(0);
        int bi = INT_MAX;
        for (int i = threadIdx.x; i < nb; i += blockDim.x) {
          const T x = Pn[(size_t)i * BP + c], v = magnitude(x);
          if (!used[i] && better(v, i, best, bi)) {
            best = v;
            bi = i;
            sv = x;
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const T v2 = __shfl_down_sync(0xffffffffu, best, o);
          const int i2 = __shfl_down_sync(0xffffffffu, bi, o);
          const T s2 = __shfl_down_sync(0xffffffffu, sv, o);
          if (better(v2, i2, best, bi)) {
            best = v2;
            bi = i2;
            sv = s2;
          }
        }
        if (lane == 0) {
          wv[warp] = best;
          wi[warp] = bi;
          ws[warp] = sv;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
          for (int w = 1; w < nw; ++w)
            if (better(wv[w], wi[w], best, bi)) {
              best = wv[w];
              bi = wi[w];
              sv = ws[w];
            }
          s_p = bi;
          s_piv = sv;
          piv_row[k] = bi;
          step_of[bi] = k;
          used[bi] = 1;
          pr[c] = bi;
        }
        __syncthreads();
        const int p = s_p;
        T piv = s_piv;
        if (!(fabs(piv) > T(0))) {
          bad = true;
          piv = T(1);
        }
        const T ipiv = T(1) / piv;
        // the step on the panel's columns, a thread per row i != p (the pivot
        // row keeps its old values until every other row has used them)
        for (int i = threadIdx.x; i < nb; i += blockDim.x) {
          if (i == p) continue;
          T* pi = Pn + (size_t)i * BP;
          const T* pp = Pn + (size_t)p * BP;
          const T m = pi[c];
          for (int cc = 0; cc < bw; ++cc) pi[cc] = cc == c ? -m * ipiv : pi[cc] - m * pp[cc] * ipiv;
        }
        __syncthreads();
        for (int cc = threadIdx.x; cc < bw; cc += blockDim.x)
          Pn[(size_t)p * BP + cc] = cc == c ? ipiv : Pn[(size_t)p * BP + cc] * ipiv;
        __syncthreads();
      }
      // every other column: x <- x + sum_c (X_c - e_{p_c}) x[p_c], a thread per column:
      // the panel rows X[i][0..BP) in 16-byte loads, then the e_{p_c} terms on the
      // panel's pivot rows (distinct rows, one subtraction each)
      for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        if (j >= k0 && j < k0 + bw) continue;
        T xp[BP];
#pragma unroll
        for (int c = 0; c < BP; ++c) xp[c] = c < bw ? A[(size_t)pr[c] * nb + j] : T(0);
        // eight rows' loads in flight before their updates
        int i = 0;
        for (; i + 8 <= nb; i += 8) {
          T a[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) a[u] = A[(size_t)(i + u) * nb + j];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            T pi[BP];
            ld_vec<T, BP>(Pn + (size_t)(i + u) * BP, pi);
            T acc = a[u];
#pragma unroll
            for (int c = 0; c < BP; ++c) acc += pi[c] * xp[c];
            A[(size_t)(i + u) * nb + j] = acc;
          }
        }
        for (; i < nb; ++i) {
          T pi[BP];
          ld_vec<T, BP>(Pn + (size_t)i * BP, pi);
          T acc = A[(size_t)i * nb + j];
#pragma unroll
          for (int c = 0; c < BP; ++c) acc += pi[c] * xp[c];
          A[(size_t)i * nb + j] = acc;
        }
#pragma unroll
        for (int c = 0; c < BP; ++c)
          if (c < bw) A[(size_t)pr[c] * nb + j] -= xp[c];
      }
      for (int t = threadIdx.x; t < nb * bw; t += blockDim.x) {
        const int i = t / bw, c = t - i * bw;
        A[(size_t)i * nb + k0 + c] = Pn[(size_t)i * BP + c];
      }
    }
    // in place: the row permutation i -> step_of[i], then the column
    // permutation j -> piv_row[j], each applied cycle by cycle
    for (int pass = 0; pass < 2; ++pass) {
      const int* to = pass == 0 ? step_of : piv_row;
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int i = 0; i < nb; ++i) used[i] = 0;
        for (int i0 = 0; i0 < nb; ++i0) {
          lead[i0] = 0;
          if (used[i0]) continue;
          int c = i0, len = 0;
          do {
            used[c] = 1;
            c = to[c];
            ++len;
          } while (c != i0 && len <= nb);
          lead[i0] = len > 1 ? len : 0;
        }
      }
      __syncthreads();
      for (int i0 = 0; i0 < nb; ++i0) {
        const int len = lead[i0];
        if (len == 0) continue;
        for (int x = threadIdx.x; x < nb; x += blockDim.x) {
          const size_t str = pass == 0 ? (size_t)nb : 1, off = pass == 0 ? (size_t)x : (size_t)x * nb;
          T carry = A[off + (size_t)i0 * str];
          int src = i0;
          for (int s = 0; s < len; ++s) {
            const int dst = to[src];
            const T y = A[off + (size_t)dst * str];
            A[off + (size_t)dst * str] = carry;
            carry = y;
            src = dst;
          }
        }
      }
    }
    if (bad && threadIdx.x == 0) atomicOr(status, ST_SINGULAR);
    __syncthreads();
  }
}

// Blocks of up to 512 rows that do not fit registers or shared memory (FP32:
// nb = 280 and 420 at p = 5, 6; FP64: from 175), rows a multiple of 16 bytes:
// the panel elimination below with one CTA per SM, so that the blocks in
// flight (152 x 706 KB at nb = 420) stay in L2.
//  * The panel is held in registers, a thread per row, and eliminated with two
//    barriers per step: the pivot search is one warp reduction over the value's
//    bits and one over the warps' candidates, done by every warp for itself,
//    and the pivot row goes through shared memory.
//  * The update of the other columns, C += P Xp (Xp the panel's pivot rows as
//    they were), takes register tiles of RI rows x 16 bytes of columns: per
//    panel column RI + 16 bytes from shared memory for RI x 16 bytes of
//    results.  A panel of 128 bytes of columns makes it bound by the FP32 pipe;
//    panels of 16 FP32 columns are bound by the 2 nb^2 entries of L2 traffic.
//  * The two permutations of the result go through shared memory slab by slab
//    (coalesced), not cycle by cycle through memory.
// nb = 420, 4,096 blocks: 145 -> 28.6 ms; FP64 nb = 175, 1,728 blocks: 27.7 -> 23.5 ms
// (the FP64 pipe: 16 ms).
constexpr int BLK_THREADS = 512;
template <class T>
struct BlkTile {
  static constexpr int BW = 128 / sizeof(T);           // panel width
  static constexpr int RI = sizeof(T) == 4 ? 16 : 8;   // rows of a register tile
};
// |x| as an integer that orders like it, in two words; 0 = not a candidate
__device__ __forceinline__ void pivot_key(float x, bool cand, unsigned* hi, unsigned* lo) {
  *hi = cand ? __float_as_uint(magnitude(x)) + 1u : 0u;
  *lo = 0u;
}
__device__ __forceinline__ void pivot_key(double x, bool cand, unsigned* hi, unsigned* lo) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(magnitude(x));
  *hi = cand ? (unsigned)(b >> 32) + 1u : 0u;
  *lo = cand ? (unsigned)b : 0u;
}
// lowest lane with the largest key (hi, lo) of the warp; all lanes take part
template <class T>
__device__ __forceinline__ int warp_argmax(unsigned hi, unsigned lo) {
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  if (sizeof(T) == 4) return __ffs(__ballot_sync(0xffffffffu, hi == mh)) - 1;
  const unsigned l2 = hi == mh ? lo : 0u, ml = __reduce_max_sync(0xffffffffu, l2);
  return __ffs(__ballot_sync(0xffffffffu, hi == mh && l2 == ml)) - 1;
}

// VN consecutive entries of a matrix row (16 bytes, or one entry where rows are not aligned)
template <class T, int VN>
__device__ __forceinline__ void ld_row(const T* p, T* v) {
  if constexpr (VN == 1)
    v[0] = p[0];
  else
    ld_vec<T, VN>(p, v);
}
template <class T, int VN>
__device__ __forceinline__ void st_row(T* p, const T* v) {
  if constexpr (VN == 1)
    p[0] = v[0];
  else
    st_vec<T, VN>(p, v);
}

template <class T, int VN>
__global__ void __launch_bounds__(BLK_THREADS, 1) block_inverse_blk_kernel(T* __restrict__ blocks, int nb,
                                                                           size_t bstride, long nblk, int slab,
                                                                           int* status) {
  constexpr int BW = BlkTile<T>::BW, RI = BlkTile<T>::RI, V16 = 16 / sizeof(T);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nbp = (nb + RI - 1) / RI * RI, nv = nb / VN, nbx = (BW * nb + 1) / 2 * 2;
  T* Ps = reinterpret_cast<T*>(smem_raw);             // [BW][nbp] panel, transposed; later the permutations' slab
  T* Xp = Ps + (size_t)BW * nbp;                      // [BW][nb] pivot rows before the panel
  T* prow = Xp + nbx;                                 // [2][BW] pivot row of the step (alternating)
  int* piv_row = reinterpret_cast<int*>(prow + 2 * BW);
  int* step_of = piv_row + nb;
  __shared__ unsigned cand_hi[2][16], cand_lo[2][16];
  __shared__ int cand_row[2][16];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < nb; i += BLK_THREADS) step_of[i] = -1;   // no row has been a pivot (again at a block's end)
  for (long blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    T* A = blocks + (size_t)blk * bstride;
    bool bad = false, used = tid >= nb;
    for (int k0 = 0; k0 < nb; k0 += BW) {
      const int bw = min(BW, nb - k0);
      // the panel into registers, a row per thread (columns past the last: zero)
      T x[BW];
#pragma unroll
      for (int c = 0; c < BW; c += VN) {
        if (tid < nb && c < bw)
          ld_row<T, VN>(A + (size_t)tid * nb + k0 + c, x + c);
        else
#pragma unroll
          for (int u = 0; u < VN; ++u) x[c + u] = T(0);
      }
#pragma unroll
      for (int c = 0; c < BW; ++c) {
        if (c >= bw) break;
        const int par = c & 1;
        unsigned hi, lo;
        pivot_key(x[c], !used, &hi, &lo);
        const int wl = warp_argmax<T>(hi, lo);
        if (lane == wl) {
          cand_hi[par][warp] = hi;
          cand_lo[par][warp] = lo;
          cand_row[par][warp] = tid;
        }
        __syncthreads();
        const int b = lane & 15;
        const int wb = warp_argmax<T>(cand_hi[par][b], cand_lo[par][b]) & 15;
        const int p = cand_row[par][wb];
        T* pr = prow + par * BW;
        if (tid == p) {
#pragma unroll
          for (int u = 0; u < BW; ++u) pr[u] = x[u];
          used = true;
          piv_row[k0 + c] = p;
          step_of[p] = k0 + c;
        }
        __syncthreads();
        T piv = pr[c];
        if (!(fabs(piv) > T(0))) {
          bad = true;
          piv = T(1);
        }
        const T ipiv = T(1) / piv;
        if (tid == p) {
#pragma unroll
          for (int u = 0; u < BW; ++u) x[u] = u == c ? ipiv : x[u] * ipiv;
        } else {
          const T m = x[c] * ipiv;
#pragma unroll
          for (int u = 0; u < BW; u += V16) {
            T q[V16];
            ld_vec<T, V16>(pr + u, q);
#pragma unroll
            for (int w = 0; w < V16; ++w)
              if (u + w != c) x[u + w] -= m * q[w];
          }
          x[c] = -m;
        }
      }
      // pivot rows before the panel, the panel transposed and back in place
      for (int t = tid; t < bw * nv; t += BLK_THREADS) {
        const int c = t / nv, v = t - c * nv;
        T q[VN];
        ld_row<T, VN>(A + (size_t)piv_row[k0 + c] * nb + v * VN, q);
#pragma unroll
        for (int u = 0; u < VN; ++u) Xp[(size_t)c * nb + v * VN + u] = q[u];
      }
      if (tid < nbp) {
#pragma unroll
        for (int c = 0; c < BW; ++c) Ps[(size_t)c * nbp + tid] = tid < nb ? x[c] : T(0);
      }
      __syncthreads();
      if (tid < nb) {
#pragma unroll
        for (int c = 0; c < BW; c += VN)
          if (c < bw) st_row<T, VN>(A + (size_t)tid * nb + k0 + c, x + c);
      }
      // C += P Xp on the other columns (pivot rows: C = P Xp)
      const int vlo = k0 / VN, nvc = nv - bw / VN;      // columns' vectors outside the panel
      for (int t = tid; t < nbp / RI * nvc; t += BLK_THREADS) {
        const int rg = t / nvc, v_ = t - rg * nvc, v = v_ < vlo ? v_ : v_ + bw / VN, i0 = rg * RI;
        T acc[RI][VN];
        T* Ac = A + (size_t)i0 * nb + (size_t)v * VN;
#pragma unroll
        for (int i = 0; i < RI; ++i) ld_row<T, VN>(Ac + (size_t)min(i, nb - 1 - i0) * nb, acc[i]);
#pragma unroll
        for (int i = 0; i < RI; ++i) {
          const int so = i0 + i < nb ? step_of[i0 + i] : -1;
          if (so >= k0 && so < k0 + bw)
#pragma unroll
            for (int u = 0; u < VN; ++u) acc[i][u] = T(0);
        }
#pragma unroll 2
        for (int c = 0; c < bw; ++c) {
          T pi[RI], q[VN];
          ld_vec<T, RI>(Ps + (size_t)c * nbp + i0, pi);
          ld_row<T, VN>(Xp + (size_t)c * nb + (size_t)v * VN, q);
#pragma unroll
          for (int i = 0; i < RI; ++i)
#pragma unroll
            for (int u = 0; u < VN; ++u) acc[i][u] += pi[i] * q[u];
        }
#pragma unroll
        for (int i = 0; i < RI; ++i)
          if (i0 + i < nb) st_row<T, VN>(Ac + (size_t)i * nb, acc[i]);
      }
      __syncthreads();
    }
    // X[step_of[i]][piv_row[j]] = R[i][j]: rows by slabs of columns, then columns
    // by slabs of rows, each slab read whole before it is written back
    for (int j0 = 0; j0 < nb; j0 += slab) {
      const int w = min(slab, nb - j0);
      for (int t = tid; t < nb * w; t += BLK_THREADS) {
        const int i = t / w, j = t - i * w;
        Ps[(size_t)i * slab + j] = A[(size_t)i * nb + j0 + j];
      }
      __syncthreads();
      for (int t = tid; t < nb * w; t += BLK_THREADS) {
        const int i = t / w, j = t - i * w;             // row i of the result: R's row piv_row[i]
        A[(size_t)i * nb + j0 + j] = Ps[(size_t)piv_row[i] * slab + j];
      }
      __syncthreads();
    }
    for (int i0 = 0; i0 < nb; i0 += slab) {
      const int w = min(slab, nb - i0);
      for (int t = tid; t < nb * w; t += BLK_THREADS) Ps[t] = A[(size_t)i0 * nb + t];
      __syncthreads();
      for (int t = tid; t < nb * w; t += BLK_THREADS) {
        const int i = t / nb, j = t - i * nb;           // column j of the result: R's column step_of[j]
        A[(size_t)i0 * nb + t] = Ps[(size_t)i * nb + step_of[j]];
      }
      __syncthreads();
    }
    if (bad && tid == 0) atomicOr(status, ST_SINGULAR);
    __syncthreads();
    for (int i = tid; i < nb; i += BLK_THREADS) step_of[i] = -1;
  }
}

template <class T, int VN>
cudaError_t run_blk(T* A, int nb, size_t bstride, long nblk, int smax, int* status, cudaStream_t st, bool* done) {
  constexpr int BW = BlkTile<T>::BW, RI = BlkTile<T>::RI;
  *done = false;
  const size_t nbp = (nb + RI - 1) / RI * RI;
  if (nbp > (size_t)BLK_THREADS || nb % VN || bstride % VN || (reinterpret_cast<uintptr_t>(A) & (VN * sizeof(T) - 1)))
    return cudaSuccess;
  const size_t xp = ((size_t)BW * nb + 1) / 2 * 2;       // (16-byte multiple)
  const size_t tiles = ((size_t)BW * nbp + xp + 2 * BW) * sizeof(T), idx = 2 * (size_t)nb * sizeof(int);
  if (tiles + idx > (size_t)smax - 1024) return cudaSuccess;
  const int slab = (int)(((size_t)BW * nbp + (size_t)BW * nb) / nb);   // rows or columns that fit over Ps and Xp
  cudaError_t e = allow_max_smem(block_inverse_blk_kernel<T, VN>);
  if (e != cudaSuccess) return e;
  note_launch();
  block_inverse_blk_kernel<T, VN><<<(int)std::min<long>(nblk, num_sms_inv()), BLK_THREADS, tiles + idx, st>>>(
      A, nb, bstride, nblk, slab, status);
  *done = true;
  return cudaGetLastError();
}

// Blocks of 40 rows or more that fit shared memory (209 rows in FP32, 153 in FP64) with their panel: the elimination of
// block_inverse_blk_kernel on a copy in shared memory (rows padded to an odd
// number of 16-byte vectors, so that a thread per row reads its panel without
// bank conflicts), the inverse written column-major.  The panel's warps alone
// take part in its barriers.  A step of block_inverse_reg_kernel costs 2,600
// cycles at nb = 175 (three barriers, a serial pivot search, every thread's whole
// tile); here a step is 32 columns wide and the rest is one register-tiled
// update per panel.
// 4,096 FP32 blocks of 175 rows: 6.5 -> 3.8 ms, of 100: 2.76 -> 1.20; 3,600 of 180
// (block_inverse_kernel before): 39 -> 3.6; 1,080 FP64 blocks of 100 rows: 6.9 ->
// 2.8 ms, of 50: 1.24 -> 0.55.  Bound by the panel's steps (latency) and the FP32
// pipe in the update, FP64 by its pipe.
template <class T, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) block_inverse_sm_kernel(T* __restrict__ blocks, int nb, int lds,
                                                                        int ldo, size_t bstride, long nblk,
                                                                        int* status) {
  constexpr int BW = BlkTile<T>::BW, RI = BlkTile<T>::RI, V = 16 / sizeof(T);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nbp = (nb + RI - 1) / RI * RI, nv = (nb + V - 1) / V;
  T* S = reinterpret_cast<T*>(smem_raw);              // [nb][lds]
  T* Ps = S + (size_t)nb * lds;                       // [BW][nbp] panel, transposed
  T* Xp = Ps + (size_t)BW * nbp;                      // [BW][lds] pivot rows before the panel
  T* prow = Xp + (size_t)BW * lds;                    // [2][BW] pivot row of the step (alternating)
  int* piv_row = reinterpret_cast<int*>(prow + 2 * BW);
  int* step_of = piv_row + nb;
  __shared__ unsigned cand_hi[2][16], cand_lo[2][16];
  __shared__ int cand_row[2][16];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nrw = (nb + 31) / 32;   // warps with rows of the panel
  for (long blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    T* A = blocks + (size_t)blk * bstride;
    __syncthreads();
    for (int i = tid; i < nb; i += NT) step_of[i] = -1;
    for (int i = warp; i < nb; i += NT / 32)
      for (int j = lane; j < nv * V; j += 32) S[(size_t)i * lds + j] = j < nb ? A[(size_t)i * nb + j] : T(0);
    __syncthreads();
    bool bad = false, used = tid >= nb;
    for (int k0 = 0; k0 < nb; k0 += BW) {
      const int bw = min(BW, nb - k0);
      T x[BW];
      if (warp < nrw) {
#pragma unroll
        for (int c = 0; c < BW; c += V) {
          if (tid < nb && c < bw)
            ld_vec<T, V>(S + (size_t)tid * lds + k0 + c, x + c);
          else
#pragma unroll
            for (int u = 0; u < V; ++u) x[c + u] = T(0);
        }
#pragma unroll
        for (int c = 0; c < BW; ++c) {
          if (c >= bw) break;
          const int par = c & 1;
          unsigned hi, lo;
          pivot_key(x[c], !used, &hi, &lo);
          const int wl = warp_argmax<T>(hi, lo);
          if (lane == wl) {
            cand_hi[par][warp] = hi;
            cand_lo[par][warp] = lo;
            cand_row[par][warp] = tid;
          }
          asm volatile("bar.sync 1, %0;" ::"r"(nrw * 32) : "memory");
          const int b = lane < nrw ? lane : 0;
          const int wb = warp_argmax<T>(cand_hi[par][b], cand_lo[par][b]);
          const int p = cand_row[par][wb];
          T* pr = prow + par * BW;
          if (tid == p) {
#pragma unroll
            for (int u = 0; u < BW; ++u) pr[u] = x[u];
            used = true;
            piv_row[k0 + c] = p;
            step_of[p] = k0 + c;
          }
          asm volatile("bar.sync 1, %0;" ::"r"(nrw * 32) : "memory");
          T piv = pr[c];
          if (!(fabs(piv) > T(0))) {
            bad = true;
            piv = T(1);
          }
          const T ipiv = T(1) / piv;
          if (tid == p) {
#pragma unroll
            for (int u = 0; u < BW; ++u) x[u] = u == c ? ipiv : x[u] * ipiv;
          } else {
            const T m = x[c] * ipiv;
#pragma unroll
            for (int u = 0; u < BW; u += V) {
              T q[V];
              ld_vec<T, V>(pr + u, q);
#pragma unroll
              for (int w = 0; w < V; ++w)
                if (u + w != c) x[u + w] -= m * q[w];
            }
            x[c] = -m;
          }
        }
      }
      __syncthreads();
      // pivot rows before the panel; the panel transposed
      for (int t = tid; t < bw * nv; t += NT) {
        const int c = t / nv, v = t - c * nv;
        T q[V];
        ld_vec<T, V>(S + (size_t)piv_row[k0 + c] * lds + v * V, q);
        st_vec<T, V>(Xp + (size_t)c * lds + v * V, q);
      }
      if (tid < nbp) {
#pragma unroll
        for (int c = 0; c < BW; ++c) Ps[(size_t)c * nbp + tid] = tid < nb ? x[c] : T(0);
      }
      __syncthreads();
      if (tid < nb) {      // and back in place
#pragma unroll
        for (int c = 0; c < BW; ++c)
          if (c < bw) S[(size_t)tid * lds + k0 + c] = x[c];
      }
      // C += P Xp on the other columns (pivot rows: C = P Xp)
      const int vlo = k0 / V, pv = (bw + V - 1) / V, nvc = nv - pv;
      for (int t = tid; t < nbp / RI * nvc; t += NT) {
        const int rg = t / nvc, v_ = t - rg * nvc, v = v_ < vlo ? v_ : v_ + pv, i0 = rg * RI;
        T acc[RI][V];
        T* Sc = S + (size_t)i0 * lds + v * V;
#pragma unroll
        for (int i = 0; i < RI; ++i) {
          const int ic = min(i, nb - 1 - i0), so = step_of[i0 + ic];
          ld_vec<T, V>(Sc + (size_t)ic * lds, acc[i]);
          if (so >= k0 && so < k0 + bw)
#pragma unroll
            for (int u = 0; u < V; ++u) acc[i][u] = T(0);
        }
#pragma unroll 2
        for (int c = 0; c < bw; ++c) {
          T pi[RI], q[V];
          ld_vec<T, RI>(Ps + (size_t)c * nbp + i0, pi);
          ld_vec<T, V>(Xp + (size_t)c * lds + v * V, q);
#pragma unroll
          for (int i = 0; i < RI; ++i)
#pragma unroll
            for (int u = 0; u < V; ++u) acc[i][u] += pi[i] * q[u];
        }
#pragma unroll
        for (int i = 0; i < RI; ++i)
          if (i0 + i < nb) st_vec<T, V>(Sc + (size_t)i * lds, acc[i]);
      }
      __syncthreads();
    }
    // X[r][c] = R[piv_row[r]][step_of[c]], column-major, zeros in the padding rows
    for (int c = warp; c < nb; c += NT / 32) {
      const T* Sc = S + step_of[c];
      for (int r = lane; r < ldo; r += 32) A[(size_t)c * ldo + r] = r < nb ? Sc[(size_t)piv_row[r] * lds] : T(0);
    }
    if (bad && tid == 0) atomicOr(status, ST_SINGULAR);
  }
}

template <class T>
cudaError_t run_sm(T* A, int nb, size_t bstride, long nblk, int smax, int* status, cudaStream_t st, bool* done) {
  constexpr int BW = BlkTile<T>::BW, RI = BlkTile<T>::RI, V = 16 / sizeof(T);
  *done = false;
  const size_t nbp = (nb + RI - 1) / RI * RI, lds = (size_t)(((nb + V - 1) / V) | 1) * V;
  const size_t smem = ((size_t)nb * lds + BW * nbp + BW * lds + 2 * BW) * sizeof(T) + 2 * (size_t)nb * sizeof(int);
  if (smem > (size_t)smax - 1024 || nbp > 256) return cudaSuccess;
  // up to 128 rows two CTAs of 256 threads share an SM's registers
  const bool small = nb <= 128;
  cudaError_t e = small ? allow_max_smem(block_inverse_sm_kernel<T, 256>) : allow_max_smem(block_inverse_sm_kernel<T, 512>);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = small ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, block_inverse_sm_kernel<T, 256>, 256, smem)
            : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, block_inverse_sm_kernel<T, 512>, 512, smem);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaSuccess;
  const int grid = (int)std::min<long>(nblk, (long)occ * num_sms_inv());
  note_launch();
  if (small)
    block_inverse_sm_kernel<T, 256><<<grid, 256, smem, st>>>(A, nb, (int)lds, inv_ld<T>(nb), bstride, nblk, status);
  else
    block_inverse_sm_kernel<T, 512><<<grid, 512, smem, st>>>(A, nb, (int)lds, inv_ld<T>(nb), bstride, nblk, status);
  *done = true;
  return cudaGetLastError();
}

template <class T, int R>
cudaError_t run_reg(T* A, int nb, size_t bstride, long nblk, int* status, cudaStream_t st) {
  const size_t smem = (size_t)nb * inv_ld<T>(nb) * sizeof(T);
  if (smem > 48 * 1024)
    allow_max_smem(block_inverse_reg_kernel<T, R>);
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, block_inverse_reg_kernel<T, R>, 256, smem);
  const long grid = std::min<long>(nblk, (long)std::max(1, occ) * num_sms_inv());
  note_launch();
  block_inverse_reg_kernel<T, R><<<(int)grid, 256, smem, st>>>(A, nb, bstride, nblk, status);
  return cudaGetLastError();
}

}  // namespace

template <class T>
cudaError_t launch_block_inverse(T* A, int nb, size_t bstride, long nblk, int* status, int* transposed,
                                 cudaStream_t st) {
  *transposed = 1;
  if (nblk <= 0) return cudaSuccess;
  int smax = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  // the line: 7,500 FP32 blocks of 40 rows 805 us in registers, 693 in shared
  // memory; 4,096 of 50 560 and 488; the register tile of fewer rows is small
  if (nb < 40) {
    const int R = (nb + 15) / 16;
    if (R <= 1) return run_reg<T, 1>(A, nb, bstride, nblk, status, st);
    if (R <= 2) return run_reg<T, 2>(A, nb, bstride, nblk, status, st);
    return run_reg<T, 3>(A, nb, bstride, nblk, status, st);
  }
  bool done = false;
  const cudaError_t es = run_sm<T>(A, nb, bstride, nblk, smax, status, st, &done);
  if (es != cudaSuccess || done) return es;
  const int threads = 256;
  const size_t base = 2 * nb * sizeof(T) + 4 * nb * sizeof(int) + 32;
  const size_t full = base + (size_t)nb * nb * sizeof(T);
  const int use_smem = full <= (size_t)smax - 1024;
  if (!use_smem) {
    cudaError_t e = run_blk<T, 16 / (int)sizeof(T)>(A, nb, bstride, nblk, smax, status, st, &done);
    if (e != cudaSuccess) return e;
    if (sizeof(T) == 8 && !done)   // FP64 rows of an odd number of entries (nb = 175)
      if ((e = run_blk<T, sizeof(T) == 8 ? 1 : 4>(A, nb, bstride, nblk, smax, status, st, &done)) != cudaSuccess)
        return e;
    if (done) {
      *transposed = 0;
      return cudaSuccess;
    }
  }
  if (!use_smem) {   // panels of 16 columns in shared memory, rank-16 updates of the rest in global memory
    constexpr int BP = 16;
    const size_t psm = (size_t)nb * BP * sizeof(T) + 4 * (size_t)nb * sizeof(int);
    if (psm <= (size_t)smax - 1024) {
      if (psm > 48 * 1024) allow_max_smem(block_inverse_panel_kernel<T, BP>);
      int occ = 0;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, block_inverse_panel_kernel<T, BP>, 256, psm);
      const long grid = std::min<long>(nblk, (long)std::max(1, occ) * num_sms_inv());
      *transposed = 0;
      note_launch();
      block_inverse_panel_kernel<T, BP><<<(int)grid, 256, psm, st>>>(A, nb, bstride, nblk, status);
      return cudaGetLastError();
    }
  }
  const size_t smem = use_smem ? full : base;
  if (smem > 48 * 1024)
    allow_max_smem(block_inverse_kernel<T>);
  const long grid = std::min<long>(nblk, (use_smem ? 1L : 8L) * num_sms_inv());
  *transposed = use_smem;
  note_launch();
  block_inverse_kernel<T><<<(int)grid, threads, smem, st>>>(A, nb, bstride, nblk, use_smem, status);
  return cudaGetLastError();
}
template cudaError_t launch_block_inverse<double>(double*, int, size_t, long, int*, int*, cudaStream_t);
template cudaError_t launch_block_inverse<float>(float*, int, size_t, long, int*, int*, cudaStream_t);

}  // namespace dgk
