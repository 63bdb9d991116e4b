// FP64 instances of the sum-factorised block probe (dg_probe_sf.cuh).
#include "dg_probe_sf.cuh"

namespace dgk {

// (above p = 4 the stages do not fit shared memory in FP64: probe64_kernel)
bool probe_sf64_ok(const Mesh& M) { return probe_sf_ok(M) && M.p <= 4; }

cudaError_t launch_probe_sf(const Mesh& M, const double* W, double sigma, double* D, size_t dstride,
                            cudaStream_t st) {
  if (!probe_sf64_ok(M)) return cudaErrorNotSupported;
  switch (M.p + 1) {
    case 2: return run_probe_sf<double, 2, 5, 5, 3, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
    case 3: return run_probe_sf<double, 3, 5, 5, 4, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
    case 4: return run_probe_sf<double, 4, 5, 1, 5, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
    case 5: return run_probe_sf<double, 5, 3, 1, 3, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
  }
  return cudaErrorNotSupported;
}

}  // namespace dgk
