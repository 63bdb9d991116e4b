// FP32 instances of the sum-factorised block probe (dg_probe_sf.cuh) that
// interpolate the state's traces (handles without the trace cache).
#include "dg_probe_sf.cuh"

namespace dgk {

cudaError_t launch_probe_sf_interp(const Mesh& M, const float* W, float sigma, float* D, size_t dstride,
                                   cudaStream_t st) {
  switch (M.p + 1) {
    case 2: return run_probe_sf<float, 2, 5, 5, 3, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
    case 3: return run_probe_sf<float, 3, 5, 5, 4, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
    case 4: return run_probe_sf<float, 4, 5, 5, 2, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
    case 5: return run_probe_sf<float, 5, 5, 1, 3, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
    case 6: return run_probe_sf<float, 6, 5, 1, 4, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
    case 7: return run_probe_sf<float, 7, 2, 1, 2, false>(M, W, sigma, D, dstride, nullptr, nullptr, st);
  }
  return cudaErrorNotSupported;
}

}  // namespace dgk
