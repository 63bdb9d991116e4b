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
// A published sum has a 128-byte line to itself: all CTAs poll all sums, and four
// to a line it hung on where the lines lay (100 x 75, p = 0, nu = 30: 273 to 330 us a
// smoother call over ten allocations, 281 to 283 with lines apart).
constexpr int SUM_STRIDE = 128 / sizeof(Pair64);
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

// A warp polls *p, a value a lane (lanes that are not active: nothing), until all
// have arrived (each lane until its own has); false where the wait ran out.  All lanes go on together: lanes
// that leave such a loop one after the other execute what follows one after the
// other too, and an FP64 instruction holds its warp for 64 clocks however few of
// its lanes take part.
template <class X, class P>
__device__ __forceinline__ bool poll_warp(const P* p, bool active, P& q, unsigned ep, Wait& wt, int* status) {
  bool have = !active;
  for (;;) {
    if (!have) {
      q = X::ldp(p);
      have = X::hasp(q, ep);
    }
    if (__all_sync(0xffffffffu, have)) return true;
    if (__any_sync(0xffffffffu, wt.expired(status))) return false;
  }
}

// st[i] = sums[i SUM_STRIDE] = the sums over all CTAs of the items i < ni of an exchange, in FP64
// whatever the partials' precision: CTA i mod G owns item i, a group of five warps
// of it polls the G partials in[i stride + c], one a lane (152 CTAs), adds them
// by butterflies and publishes the sum, and one warp of every CTA polls the ni
// sums.  Two hops of little traffic: one hop, with every CTA reading all G x ni
// partials, saturated the L2 with polls and took 8 us.  (One warp adding five
// partials a lane would take 25 FP64 instructions in a row, five warps 10.)  False
// where a wait ran out.
template <class V, int WARPS>
__device__ bool gather_dots(const typename Xch<V>::P* in, int stride, int ni, int G, Pair64* sums, unsigned ep,
                            int* status, double2* st) {
  using X = Xch<V>;
  using X64 = Xch<double>;
  constexpr int GW = 5, NG = (WARPS - 1) / GW;
  __shared__ double2 gpart[2][NG][GW];     // (alternating: one barrier an item)
  __shared__ int gok[2][NG][GW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, C = gridDim.x;
  bool ok = true;
  if (warp >= WARPS) return ok;
  Wait wt;
  const int g = (warp - 1) / GW, gw = warp - 1 - g * GW;
  // (the owned items i = blockIdx.x + k C, shared out over the groups; warp 0 collects)
  if (warp > 0 && g < NG) {
    int par = 0;
    for (int i = blockIdx.x + g * C; i < ni; i += NG * C, par ^= 1) {
      double hs = 0.0, ht = 0.0;
      for (int c0 = gw * 32; ok && c0 < G; c0 += GW * 32) {
        const bool active = c0 + lane < G;
        typename X::P q = {};
        ok = poll_warp<X>(in + (size_t)i * stride + c0 + lane, active, q, ep, wt, status);
        const typename X::V2 v = X::valp(q);
        const double x = (double)v.x, y = (double)v.y;     // (0 where there is no CTA)
        if (c0 == gw * 32) {
          hs = x;
          ht = y;
        } else {
          hs += x;
          ht += y;
        }
      }
      warp_sum2(hs, ht);
      if (lane == 0) {
        gpart[par][g][gw] = make_double2(hs, ht);
        gok[par][g][gw] = ok;
      }
      __syncwarp();
      asm volatile("bar.sync %0, %1;" ::"r"(2 + g), "n"(GW * 32) : "memory");
      if (gw == 0) {
        const int k = min(lane & 15, GW - 1);
        const double2 pr = gpart[par][g][k];
        const bool in_k = (lane & 15) < GW, every = __all_sync(0xffffffffu, gok[par][g][k] != 0);
        double a = lane & 16 ? pr.y : pr.x;
        if (!in_k) a = 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        const double t = __shfl_sync(0xffffffffu, a, 16);
        if (every && lane == 0) X64::stp(sums + (size_t)i * SUM_STRIDE, a, t, ep);
      }
    }
  }
  if (warp == 0) {
    for (int i0 = 0; ok && i0 < ni; i0 += 32) {
      const bool active = i0 + lane < ni;
      Pair64 q = {};
      ok = poll_warp<X64>(sums + (size_t)(i0 + lane) * SUM_STRIDE, active, q, ep, wt, status);
      if (active) st[i0 + lane] = X64::valp(q);
    }
    __syncwarp();
  }
  return ok;
}

}  // namespace dgk
