// The tensor-core kernel's 2-bit forms (see qtea_mma.h): v*x split (M <= 4, or up to four tiles), and v in A (M <= 8, M <= 16).
#include "qtea_mma.h"

namespace qtea {

cudaError_t mma2_configure(size_t smem_optin) {
  cudaError_t e = x_configure<1, kXSplit2, false>(smem_optin);
  if (e == cudaSuccess) e = x_configure<1, kXSplit2, true>(smem_optin);
  if (e == cudaSuccess) e = x_configure<2, kXSplit2, true>(smem_optin);
  if (e == cudaSuccess) e = x_configure<3, kXSplit2, true>(smem_optin);
  if (e == cudaSuccess) e = x_configure<4, kXSplit2, true>(smem_optin);
  if (e == cudaSuccess) e = x_configure<1, kXV2, false>(smem_optin);
  if (e == cudaSuccess) e = x_configure<1, kXV2, true>(smem_optin);
  if (e == cudaSuccess) e = x_configure<2, kXV2, false>(smem_optin);
  if (e == cudaSuccess) e = x_configure<2, kXV2, true>(smem_optin);
  return e;
}

cudaError_t launch_mma2(const TensorMaps& maps, const XParams& p, bool grp, bool split, int grid, size_t smem,
                        cudaStream_t st) {
  const int mode = x_mode(false, p.M, split), mt = x_mt(mode, p.M);
  if (mode == kXV2) {
    if (mt == 1)
      return grp ? x_launch<1, kXV2, true>(maps, p, grid, smem, st) : x_launch<1, kXV2, false>(maps, p, grid, smem, st);
    return grp ? x_launch<2, kXV2, true>(maps, p, grid, smem, st) : x_launch<2, kXV2, false>(maps, p, grid, smem, st);
  }
  switch (mt) {
    case 1:
      return grp ? x_launch<1, kXSplit2, true>(maps, p, grid, smem, st) : x_launch<1, kXSplit2, false>(maps, p, grid, smem, st);
    case 2: return x_launch<2, kXSplit2, true>(maps, p, grid, smem, st);
    case 3: return x_launch<3, kXSplit2, true>(maps, p, grid, smem, st);
    default: return x_launch<4, kXSplit2, true>(maps, p, grid, smem, st);
  }
}

}  // namespace qtea
