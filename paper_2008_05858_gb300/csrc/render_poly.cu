// Production instantiations of the polynomial separable-PSF render kernel (render_poly.cuh).
#include "render_poly.cuh"

namespace e2e {

bool poly_variant_supported(int K) { return K >= 3; }

size_t poly_smem_bytes(int area, int JB, int nk_max, int nd) { return PolyLayout(32 * JB, nk_max, nd, area).total; }

int poly_row_f4(int K) { return 4 * poly_role_f4(K); }

cudaError_t launch_render_poly(int K, int DX, int DY, const DevSlice* slices, const double* const* flux_tab,
                               const double* u_all, const Item* items, int n_items, float2* store, int B, int JB,
                               int nk_max, int max_deg, size_t smem, cudaStream_t st, int* err) {
  if (n_items == 0) return cudaSuccess;
  MixedArgs a{slices, flux_tab, u_all, items, store, B, JB, nk_max, max_deg, err, 0};
  if (err) return launch_render_poly_checked(K, DX, DY, a, n_items, smem, st);
#define E2E_V(KK, X, Y) \
  if (K == KK && DX == X && DY == Y) return launch_poly_one<KK, X, Y, false>(a, n_items, smem, st);
  E2E_POLY_VARIANTS(E2E_V)
#undef E2E_V
  return cudaErrorInvalidValue;
}

}  // namespace e2e
