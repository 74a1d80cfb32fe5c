// Instantiations of the adjoint time-step kernel with the convolutional PML
// (modes ADJ_STORED, ADJ_STEP).
#include "stencil_impl.cuh"

namespace mamute {

cudaError_t dispatch_pml_adjoint(const StepArgs& a, int n_items, int max_planes, int tx, int ty,
                                 bool dens, int mode, cudaStream_t s, int* occ) {
#define MAMUTE_T(TX, TY)                                                                        \
  if (tx == TX && ty == TY && mode == MODE_ADJ_STORED)                                                  \
    return launch_mode<TX, TY, MODE_ADJ_STORED, true>(a, n_items, max_planes, dens, s, occ);             \
  if (tx == TX && ty == TY && mode == MODE_ADJ_STEP)                                            \
    return launch_mode<TX, TY, MODE_ADJ_STEP, true>(a, n_items, max_planes, dens, s, occ);
  MAMUTE_TILES(MAMUTE_T)
#undef MAMUTE_T
  return cudaErrorInvalidValue;
}

}  // namespace mamute
