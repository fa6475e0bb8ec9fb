// Kinematic-mode kernels (dg_kin.cuh) of orders 1..5.
#include "dg_kin.cuh"

namespace dgpf {

bool kin_kernels(int p, KinKernels *out) {
  switch (p) {
    case 1: *out = {&launch_kin_volume<1>, &launch_kin_stage<1>, &launch_kin_velocity_table<1>}; return true;
    case 2: *out = {&launch_kin_volume<2>, &launch_kin_stage<2>, &launch_kin_velocity_table<2>}; return true;
    case 3: *out = {&launch_kin_volume<3>, &launch_kin_stage<3>, &launch_kin_velocity_table<3>}; return true;
    case 4: *out = {&launch_kin_volume<4>, &launch_kin_stage<4>, &launch_kin_velocity_table<4>}; return true;
    case 5: *out = {&launch_kin_volume<5>, &launch_kin_stage<5>, &launch_kin_velocity_table<5>}; return true;
    default: return false;
  }
}

// Sets what the kernels of a captured sequence read (KinTime) for a start at time t and steps of size
// dt: one thread per stage.  Stage times t + k dt + frac dt, frac = 0, 1/2, 1/2, 1.
__global__ void k_kin_set_time(KinParams kp, double *kt, double t, double dt) {
  const int st = threadIdx.x;
  if (st == 0) {
    kt[KT_HALF] = 0.5 * dt;
    kt[KT_DT] = dt;
    kt[KT_SIXTH] = dt / 6.0;
  }
  const double frac = (st & 3) == 0 ? 0.0 : (st & 3) == 3 ? 1.0 : 0.5;
  kt[KT_C + st] = kin_time_factor(kp, (t + (st >> 2) * dt) + frac * dt);
}

}  // namespace dgpf
