// FP32 instances of the sum-factorised block probe (dg_probe_sf.cuh).
#include "dg_probe_sf.cuh"

namespace dgk {

// Whether the FP32 diagonal blocks of this mesh come from the sum-factorised
// probe: the meshes of the FP32 product's kernels, no direction of one element
// (its faces feed the diagonal block twice).
bool probe_sf_ok(const Mesh& M) {
  if (!sf32_ok(M)) return false;
  for (int k = 0; k < 3; ++k)
    if (M.desc.n[k] == 1) return false;
  return true;
}

cudaError_t launch_probe_sf_interp(const Mesh& M, const float* W, float sigma, float* D, size_t dstride,
                                   cudaStream_t st);   // dg_probe_sf32i.cu: the state's traces interpolated

cudaError_t launch_probe_sf(const Mesh& M, const float* W, float sigma, float* D, size_t dstride, const float* Pv,
                            const float* Pf, cudaStream_t st) {
  if (!probe_sf_ok(M)) return cudaErrorNotSupported;
  if (!Pv || !Pf) return launch_probe_sf_interp(M, W, sigma, D, dstride, st);
  const float4 *v = reinterpret_cast<const float4*>(Pv), *f = reinterpret_cast<const float4*>(Pf);
  switch (M.p + 1) {
    case 2: return run_probe_sf<float, 2, 5, 5, 3, true>(M, W, sigma, D, dstride, v, f, st);
    case 3: return run_probe_sf<float, 3, 5, 5, 4, true>(M, W, sigma, D, dstride, v, f, st);
    case 4: return run_probe_sf<float, 4, 5, 5, 2, true>(M, W, sigma, D, dstride, v, f, st);
    case 5: return run_probe_sf<float, 5, 5, 1, 3, true>(M, W, sigma, D, dstride, v, f, st);
    case 6: return run_probe_sf<float, 6, 5, 1, 4, true>(M, W, sigma, D, dstride, v, f, st);
    case 7: return run_probe_sf<float, 7, 5, 1, 2, true>(M, W, sigma, D, dstride, v, f, st);
  }
  return cudaErrorNotSupported;
}

}  // namespace dgk
