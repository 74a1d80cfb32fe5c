// Time-step kernel front end: supported tile shapes, occupancy and launch
// (the kernel itself is in stencil_impl.cuh, instantiated in stencil_fwd.cu,
// stencil_adj.cu, stencil_pml_fwd.cu and stencil_pml_adj.cu).
#include "stencil_impl.cuh"

namespace mamute {

bool tile_supported(int tx, int ty) {
#define MAMUTE_T(TX, TY) if (tx == TX && ty == TY) return true;
  MAMUTE_TILES(MAMUTE_T)
#undef MAMUTE_T
  return false;
}

static cudaError_t dispatch(const StepArgs& a, int n_items, int max_planes, int tx, int ty,
                            bool dens, bool pml, int mode, cudaStream_t s, int* occ) {
  if (pml)
    return mode == MODE_FWD || mode == MODE_FWD_STORE
               ? dispatch_pml_forward(a, n_items, max_planes, tx, ty, dens, mode, s, occ)
               : dispatch_pml_adjoint(a, n_items, max_planes, tx, ty, dens, mode, s, occ);
  if (mode == MODE_FWD || mode == MODE_FWD_PH || mode == MODE_FWD_STORE ||
      mode == MODE_FWD_STORE_PH)
    return dispatch_forward(a, n_items, max_planes, tx, ty, dens, mode, s, occ);
  return dispatch_adjoint(a, n_items, max_planes, tx, ty, dens, mode, s, occ);
}

int step_blocks_per_sm(int tx, int ty, bool dens, bool pml, int mode, int max_planes) {
  int occ = 0;
  StepArgs a{};
  const cudaError_t e = dispatch(a, 0, max_planes, tx, ty, dens, pml, mode, nullptr, &occ);
  if (e == cudaSuccess) return occ;
  cudaGetLastError();  // the caller takes another shape
  return e == cudaErrorInvalidValue ? 0 : -1;
}

cudaError_t launch_step(const StepArgs& a, int n_items, int max_planes, int tx, int ty, bool dens,
                        bool pml, int mode, cudaStream_t s) {
  if (n_items <= 0) return cudaSuccess;
  return dispatch(a, n_items, max_planes, tx, ty, dens, pml, mode, s, nullptr);
}

}  // namespace mamute
