// Debug-check instantiations of the polynomial separable-PSF render kernel, a translation unit
// of its own so that the two sets of instantiations compile in parallel.
#include "render_poly.cuh"

namespace e2e {

cudaError_t launch_render_poly_checked(int K, int DX, int DY, const MixedArgs& a, int n_items, size_t smem,
                                       cudaStream_t st) {
#define E2E_V(KK, X, Y) \
  if (K == KK && DX == X && DY == Y) return launch_poly_one<KK, X, Y, true>(a, n_items, smem, st);
  E2E_POLY_VARIANTS(E2E_V)
#undef E2E_V
  return cudaErrorInvalidValue;
}

}  // namespace e2e
