// FP32 instances of the sum-factorised neighbour blocks (dg_nbr_sf.cuh).
#include "dg_nbr_sf.cuh"

namespace dgk {

cudaError_t launch_nbr_sf(const Mesh& M, const float* W, float* O, int nmc, int colmajor, const float* Pf,
                          cudaStream_t st) {
  if (!probe_sf_ok(M) || !Pf) return cudaErrorNotSupported;
  const float4* f = reinterpret_cast<const float4*>(Pf);
  switch (M.p + 1) {
    case 2: return run_nbr_sf<float, 2>(M, W, O, nmc, colmajor, f, st);
    case 3: return run_nbr_sf<float, 3>(M, W, O, nmc, colmajor, f, st);
    case 4: return run_nbr_sf<float, 4>(M, W, O, nmc, colmajor, f, st);
    case 5: return run_nbr_sf<float, 5>(M, W, O, nmc, colmajor, f, st);
    case 6: return run_nbr_sf<float, 6>(M, W, O, nmc, colmajor, f, st);
    case 7: return run_nbr_sf<float, 7>(M, W, O, nmc, colmajor, f, st);
  }
  return cudaErrorNotSupported;
}

}  // namespace dgk
