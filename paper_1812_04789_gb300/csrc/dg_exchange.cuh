// What the CTAs of a persistent cooperative kernel exchange: values that travel
// with their epoch (the reader polls the value itself), sums over the CTAs in
// two hops, and waits that end.
#pragma once
#include "dg_internal.h"

namespace dgk {

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// A word and its epoch in one 64-bit element, and two such elements in one
// 16-byte access.  PTX makes each element of a vector access single-copy atomic,
// no more: the two words of an element always arrive together, the two elements
// may not, so every element carries its own epoch.  (With elements of 32 bits a
// reader could see the new epoch beside the old word.)
using Word = unsigned long long;
struct __align__(16) Pair {
  Word a, b;
};
__device__ __forceinline__ Word with_epoch(unsigned x, unsigned ep) { return ((Word)ep << 32) | x; }
__device__ __forceinline__ bool has_epoch(Word v, unsigned ep) { return (unsigned)(v >> 32) == ep; }
__device__ __forceinline__ Word ld_word(const Word* p) {
  Word v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_word(Word* p, Word v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ Pair ld_pair(const Pair* p) {
  Pair v;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0,%1}, [%2];" : "=l"(v.a), "=l"(v.b) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_pair(Pair* p, unsigned x, unsigned y, unsigned ep) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1,%2};" ::"l"(p), "l"(with_epoch(x, ep)), "l"(with_epoch(y, ep))
               : "memory");
}

// What travels between the CTAs, every 32-bit word of a value in an element
// with its epoch: Z a direction's entry, P a pair of sums (s, t).
template <class V>
struct Xch;
template <>
struct Xch<float> {
  using Z = Word;
  using P = Pair;
  using V2 = float2;
  __device__ __forceinline__ static Z ld(const Z* p) { return ld_word(p); }
  __device__ __forceinline__ static bool has(Z v, unsigned ep) { return has_epoch(v, ep); }
  __device__ __forceinline__ static float val(Z v) { return __uint_as_float((unsigned)v); }
  __device__ __forceinline__ static void st(Z* p, float f, unsigned ep) {
    st_word(p, with_epoch(__float_as_uint(f), ep));
  }
  __device__ __forceinline__ static P ldp(const P* p) { return ld_pair(p); }
  __device__ __forceinline__ static bool hasp(const P& q, unsigned ep) {
    return has_epoch(q.a, ep) && has_epoch(q.b, ep);
  }
  __device__ __forceinline__ static V2 valp(const P& q) {
    return make_float2(__uint_as_float((unsigned)q.a), __uint_as_float((unsigned)q.b));
  }
  __device__ __forceinline__ static void stp(P* p, float s, float t, unsigned ep) {
    st_pair(p, __float_as_uint(s), __float_as_uint(t), ep);
  }
};
struct Pair64 {
  Pair s, t;
};
template <>
struct Xch<double> {
  using Z = Pair;
  using P = Pair64;
  using V2 = double2;
  __device__ __forceinline__ static Z ld(const Z* p) { return ld_pair(p); }
  __device__ __forceinline__ static bool has(const Z& v, unsigned ep) {
    return has_epoch(v.a, ep) && has_epoch(v.b, ep);
  }
  __device__ __forceinline__ static double val(const Z& v) {
    return __hiloint2double((int)(unsigned)v.b, (int)(unsigned)v.a);
  }
  __device__ __forceinline__ static void st(Z* p, double f, unsigned ep) {
    st_pair(p, (unsigned)__double2loint(f), (unsigned)__double2hiint(f), ep);
  }
  __device__ __forceinline__ static P ldp(const P* p) { return {ld_pair(&p->s), ld_pair(&p->t)}; }
  __device__ __forceinline__ static bool hasp(const P& q, unsigned ep) { return has(q.s, ep) && has(q.t, ep); }
  __device__ __forceinline__ static V2 valp(const P& q) { return make_double2(val(q.s), val(q.t)); }
  __device__ __forceinline__ static void stp(P* p, double s, double t, unsigned ep) {
    st(&p->s, s, ep);
    st(&p->t, t, ep);
  }
};
// A bounded wait: expired() is called once per failed poll and looks at the
// clock and the status word every 64th time.
struct Wait {
  unsigned n = 0;
  unsigned long long t0 = 0;
  __device__ __forceinline__ bool expired(int* status) {
    if ((++n & 63u) != 0) return false;
    if (*(volatile int*)status & ST_TIMEOUT) return true;
    const unsigned long long t = global_ns();
    if (t0 == 0) t0 = t;
    if (t - t0 > 2000000000ull) {
      atomicOr(status, ST_TIMEOUT);
      return true;
    }
    return false;
  }
};

// (h, l) += x, FP32 with the rounding error of the addition kept in l
__device__ __forceinline__ void two_add(double& h, double&, double x) { h += x; }
__device__ __forceinline__ void two_add(float& h, float& l, float x) {
  const float s = h + x, b = s - h;
  l += (h - (s - b)) + (x - b);
  h = s;
}

// Sums of fs and ft over a warp: the first exchange leaves fs to the lower and
// ft to the upper half, so five additions do for both.
template <class V>
__device__ __forceinline__ void warp_sum2(V& fs, V& ft) {
  const bool up = threadIdx.x & 16;
  V a = (up ? ft : fs) + __shfl_xor_sync(0xffffffffu, up ? fs : ft, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  fs = __shfl_sync(0xffffffffu, a, 0);
  ft = __shfl_sync(0xffffffffu, a, 16);
}

// st[i] = the sums over all CTAs of the items i < ni of an exchange: CTA i mod G
// owns item i, a warp of it polls the G partials in[i stride + c] (5 loads of a
// lane at once), adds them (FP32: in two-float arithmetic), a lane's CTAs and then the
// lanes by a butterfly, and publishes the sum, and one warp of every CTA
// polls the ni sums.  Two hops of little traffic: one hop, with every CTA
// reading all G x ni partials, saturated the L2 with polls and took 8 us.
// False where a wait ran out.
template <class V, int WARPS>
__device__ bool gather_dots(const typename Xch<V>::P* in, int stride, int ni, int G, typename Xch<V>::P* sums,
                            unsigned ep, int* status, typename Xch<V>::V2* st) {
  using X = Xch<V>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, C = gridDim.x;
  bool ok = true;
  if (warp >= WARPS) return ok;
  Wait wt;
  // (the owned items i = blockIdx.x + k C, shared out over the warps; warp 0 collects)
  for (int i = blockIdx.x + (warp - 1) * C; warp > 0 && i < ni; i += (WARPS - 1) * C) {
    V hs = V(0), ls = V(0), ht = V(0), lt = V(0);
    for (int c0 = lane; c0 < G; c0 += 160) {
      typename X::P q[5];
#pragma unroll
      for (int u = 0; u < 5; ++u) q[u] = X::ldp(in + (size_t)i * stride + min(c0 + 32 * u, G - 1));
#pragma unroll
      for (int u = 0; u < 5; ++u) {
        if (c0 + 32 * u >= G) continue;
        while (ok && !X::hasp(q[u], ep)) {
          if (wt.expired(status)) ok = false;
          q[u] = X::ldp(in + (size_t)i * stride + c0 + 32 * u);
        }
        const typename X::V2 v = X::valp(q[u]);
        two_add(hs, ls, v.x);
        two_add(ht, lt, v.y);
      }
    }
    if constexpr (std::is_same<V, double>::value) {
      warp_sum2(hs, ht);
    } else {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const V a = __shfl_xor_sync(0xffffffffu, hs, o), b = __shfl_xor_sync(0xffffffffu, ls, o);
        const V c = __shfl_xor_sync(0xffffffffu, ht, o), d = __shfl_xor_sync(0xffffffffu, lt, o);
        two_add(hs, ls, a);
        ls += b;
        two_add(ht, lt, c);
        lt += d;
      }
    }
    if (__all_sync(0xffffffffu, ok) && lane == 0) X::stp(sums + i, hs + ls, ht + lt, ep);
  }
  if (warp == 0) {
    for (int i = lane; i < ni; i += 32) {
      typename X::P q = X::ldp(sums + i);
      while (ok && !X::hasp(q, ep)) {
        if (wt.expired(status)) ok = false;
        q = X::ldp(sums + i);
      }
      st[i] = X::valp(q);
    }
  }
  return ok;
}

}  // namespace dgk
