// The sums over the CTAs of a persistent kernel (gather_dots, dg_exchange.cuh)
// against sums in long double on the host: FP32 and FP64 partials, one CTA to
// all SMs, fewer and more sums than CTAs and lanes, three exchanges in a row on
// the alternating buffers.  The partials alternate in sign and span seven
// decades, so that the sum is far below its terms.  Exit status 0 iff every
// CTA holds the same bits and every error is at most 160 2^-53 of the terms'
// sum of magnitudes (FP64 additions of up to 152 terms; FP32 ones miss it by 2^20).
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "dg_exchange.cuh"
using namespace dgk;

constexpr int THREADS = 512, ROUNDS = 3;

template <class V>
__global__ void __launch_bounds__(THREADS, 1) sums_kernel(typename Xch<V>::P* px, Pair64* sums, const V* s, const V* t,
                                                          int ni, int* status, double2* out) {
  __shared__ double2 st[80];
  const int G = gridDim.x, b = blockIdx.x;
  for (int r = 0; r < ROUNDS; ++r) {
    typename Xch<V>::P* p = px + (size_t)(r & 1) * ni * (G + 1);
    for (int i = threadIdx.x; i < ni; i += THREADS) {
      const size_t k = ((size_t)r * ni + i) * G + b;
      Xch<V>::stp(p + (size_t)i * (G + 1) + b, s[k], t[k], 1u + r);
    }
    const bool ok = gather_dots<V, THREADS / 32>(p, G + 1, ni, G, sums + (r & 1) * ni * SUM_STRIDE, 1u + r, status, st);
    if (__syncthreads_or(ok ? 0 : 1)) return;
    for (int i = threadIdx.x; i < ni; i += THREADS) out[((size_t)r * G + b) * ni + i] = st[i];
    __syncthreads();
  }
}

template <class V>
int run(int G, int ni) {
  std::vector<V> s((size_t)ROUNDS * ni * G), t(s.size());
  unsigned x = 12345u + G * 131u + ni;
  auto rnd = [&] { return (x = x * 1664525u + 1013904223u) >> 8; };
  for (size_t k = 0; k < s.size(); ++k) {
    s[k] = (V)((k & 1 ? -1.0 : 1.0) * std::pow(10.0, rnd() % 7) * (1.0 + rnd() / 16777216.0));
    t[k] = (V)(rnd() / 16777216.0 - 0.5);
  }
  typename Xch<V>::P* px;
  Pair64* sums;
  V *ds, *dt;
  int* status;
  double2* out;
  const size_t npx = (size_t)2 * ni * (G + 1), no = (size_t)ROUNDS * G * ni, nsum = (size_t)2 * ni * SUM_STRIDE;
  if (cudaMalloc(&px, npx * sizeof(*px)) || cudaMalloc(&sums, nsum * sizeof(Pair64)) ||
      cudaMalloc(&ds, s.size() * sizeof(V)) || cudaMalloc(&dt, s.size() * sizeof(V)) || cudaMalloc(&status, 4) ||
      cudaMalloc(&out, no * sizeof(double2)))
    return 2;
  cudaMemset(px, 0, npx * sizeof(*px));
  cudaMemset(sums, 0, nsum * sizeof(Pair64));
  cudaMemset(status, 0, 4);
  cudaMemset(out, 0, no * sizeof(double2));
  cudaMemcpy(ds, s.data(), s.size() * sizeof(V), cudaMemcpyHostToDevice);
  cudaMemcpy(dt, t.data(), s.size() * sizeof(V), cudaMemcpyHostToDevice);
  const V *cs = ds, *ct = dt;
  void* args[] = {&px, &sums, &cs, &ct, &ni, &status, &out};
  if (cudaLaunchCooperativeKernel((void*)sums_kernel<V>, dim3(G), dim3(THREADS), args, 0, 0)) return 2;
  std::vector<double2> h(no);
  if (cudaMemcpy(h.data(), out, no * sizeof(double2), cudaMemcpyDeviceToHost)) return 2;
  double worst = 0.0;
  bool same = true;
  for (int r = 0; r < ROUNDS; ++r)
    for (int i = 0; i < ni; ++i) {
      long double es = 0, et = 0, as = 0, at = 0;
      for (int c = 0; c < G; ++c) {
        const size_t k = ((size_t)r * ni + i) * G + c;
        es += s[k], et += t[k], as += std::fabs((double)s[k]), at += std::fabs((double)t[k]);
      }
      for (int b = 0; b < G; ++b) {
        const double2 v = h[((size_t)r * G + b) * ni + i];
        same = same && std::memcmp(&v, &h[(size_t)r * G * ni + i], sizeof(v)) == 0;
        worst = std::fmax(worst, (double)(std::fabs((double)((long double)v.x - es)) / as));
        worst = std::fmax(worst, (double)(std::fabs((double)((long double)v.y - et)) / at));
      }
    }
  printf("FP%d G=%d ni=%d: %.2e of the terms, same bits %d\n", (int)sizeof(V) * 8, G, ni, worst, (int)same);
  cudaFree(px), cudaFree(sums), cudaFree(ds), cudaFree(dt), cudaFree(status), cudaFree(out);
  return worst <= 160.0 * std::ldexp(1.0, -53) && same ? 0 : 1;
}

int main() {
  int rc = 0;
  const int sms = sm_count();
  for (int G : {1, 2, 15, 33, sms})
    for (int ni : {1, 2, 31, 33, 66}) rc |= run<float>(G, ni) | run<double>(G, ni);
  return rc;
}
