// The tensor-core kernel's base-3 forms (see qtea_mma.h): M = 1, and M >= 2 in one to four n8 tiles.
#include "qtea_mma.h"

namespace qtea {

cudaError_t b3mma_configure(size_t smem_optin) {
  cudaError_t e = x_configure<1, kXDiag, true>(smem_optin);
  if (e == cudaSuccess) e = x_configure<1, kXRows, true>(smem_optin);
  if (e == cudaSuccess) e = x_configure<2, kXRows, true>(smem_optin);
  if (e == cudaSuccess) e = x_configure<3, kXRows, true>(smem_optin);
  if (e == cudaSuccess) e = x_configure<4, kXRows, true>(smem_optin);
  return e;
}

cudaError_t launch_b3mma(const TensorMaps& maps, const XParams& p, int grid, size_t smem, cudaStream_t st) {
  if (p.M == 1) return x_launch<1, kXDiag, true>(maps, p, grid, smem, st);
  switch (x_mt(x_mode(true, p.M, true), p.M)) {
    case 1: return x_launch<1, kXRows, true>(maps, p, grid, smem, st);
    case 2: return x_launch<2, kXRows, true>(maps, p, grid, smem, st);
    case 3: return x_launch<3, kXRows, true>(maps, p, grid, smem, st);
    default: return x_launch<4, kXRows, true>(maps, p, grid, smem, st);
  }
}

}  // namespace qtea
