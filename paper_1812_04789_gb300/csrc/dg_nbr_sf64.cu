// FP64 instances of the sum-factorised neighbour blocks (dg_nbr_sf.cuh).
#include "dg_nbr_sf.cuh"

namespace dgk {

// (above p = 4 the face Jacobians and traces do not fit shared memory in FP64,
// and probe_sf64_ok has no diagonal blocks)
cudaError_t launch_nbr_sf(const Mesh& M, const double* W, double* O, int nmc, int colmajor, cudaStream_t st) {
  if (!probe_sf64_ok(M)) return cudaErrorNotSupported;
  switch (M.p + 1) {
    case 2: return run_nbr_sf<double, 2>(M, W, O, nmc, colmajor, nullptr, st);
    case 3: return run_nbr_sf<double, 3>(M, W, O, nmc, colmajor, nullptr, st);
    case 4: return run_nbr_sf<double, 4>(M, W, O, nmc, colmajor, nullptr, st);
    case 5: return run_nbr_sf<double, 5>(M, W, O, nmc, colmajor, nullptr, st);
  }
  return cudaErrorNotSupported;
}

}  // namespace dgk
