// Instantiations of the forward time-step kernel with the convolutional PML
// (modes FWD, FWD_STORE).
#include "stencil_impl.cuh"

namespace mamute {

cudaError_t dispatch_pml_forward(const StepArgs& a, int n_items, int max_planes, int tx, int ty,
                                 bool dens, int mode, cudaStream_t s, int* occ) {
#define MAMUTE_T(TX, TY)                                                                        \
  if (tx == TX && ty == TY && mode == MODE_FWD)                                                  \
    return launch_mode<TX, TY, MODE_FWD, true>(a, n_items, max_planes, dens, s, occ);             \
  if (tx == TX && ty == TY && mode == MODE_FWD_STORE)                                            \
    return launch_mode<TX, TY, MODE_FWD_STORE, true>(a, n_items, max_planes, dens, s, occ);
  MAMUTE_TILES(MAMUTE_T)
#undef MAMUTE_T
  return cudaErrorInvalidValue;
}

}  // namespace mamute
