// Launch interface of the convolutional-PML kernels (internal to libmamute).
//
// A CPML step is one launch per axis over that axis's layer slabs, which
// updates the memory variables and leaves their contribution to the second
// derivative in the array E, followed by the main step kernel, which adds E
// to its 25-point sum (StepArgs, step_kernel<..., PML>).
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace mamute {

// The slabs of one shot window: along axis a (0: x, 1: y, 2: z) the cells
// [0, lo) and [hi, N) within border + 4 of a face that has a layer (the layer
// and the 4 cells that the eighth-order derivatives of the memory variables
// reach); hi == lo is one range [0, N).  Along x both ends are widened to
// multiples of 4.  Memory variables are stored on the slabs only, n cells
// along the axis (slot s, or s - hi + lo in the upper slab):
//   z: [slot][Ny][pitch]   y: [Nz][slot][pitch]   x: [Nz][Ny][slot]
// at element off of each array.
struct CpmlVol {
  int lo[3], hi[3], n[3];
  long long off[3];
  int prof[3];  // the axis's b and c of cell s at CpmlArgs::b / c [prof + kCpmlPad + s]
};
// Cells before and after each profile (c = 0, b = 1), so that a thread may
// read the profile of the cells around its own without a bounds test.
constexpr int kCpmlPad = 12;

struct CpmlArgs {
  const VolDesc* vols;
  const CpmlVol* cv;
  const float* b;    // b = exp(-(d + alpha) dt), see CpmlVol::prof
  const float* c;    // c = d (b - 1) / (d + alpha)
  const float* u;    // forward: u^n; reverse: the adjoint level being propagated (pool layout)
  // Memory variables before and after the step; forward: Psi and Zeta (updated
  // in place: m2 == m2n); reverse: their multipliers.  m1 and m1n differ (a
  // thread reads its neighbours' old values), in the reverse m2 and m2n too.
  const float* m1;
  float* m1n;
  const float* m2;
  float* m2n;
  float* E;          // sum over the axes (pool layout); zero outside the slabs
};

// Grid extents of the slab launches over all shot windows.
struct CpmlExtent {
  int nvol;
  long long cols[3];  // threads across the axis, at most: x: rows x groups of 4 slots
  int len[3];         // longest slab along the axis (y, z)
  long long threads[3];  // threads of a launch with unsplit slabs, over all windows (y, z)
  bool apart;            // modelling on small windows: an axis's pieces over several launches
};

// Psi_a <- b_a Psi_a + c_a D1_a u, Zeta_a <- b_a Zeta_a + c_a (D2_a u + D1_a Psi_a),
// E = sum_a (D1_a Psi_a + Zeta_a); cpml_launches() launches.
cudaError_t launch_cpml_forward(const CpmlArgs& c, const CpmlExtent& e, cudaStream_t s);
// y_a = c_a (Zb_a + psi), Zb_a <- b_a (Zb_a + psi), p_a = Pb_a - D1_a (psi + y_a),
// Pb_a <- b_a p_a, E = sum_a (D2_a y_a - D1_a (c_a p_a)); one launch per axis.
cudaError_t launch_cpml_reverse(const CpmlArgs& c, const CpmlExtent& e, cudaStream_t s);
// Launches of one launch_cpml_forward call.
int cpml_launches(const CpmlExtent& e);

}  // namespace mamute
