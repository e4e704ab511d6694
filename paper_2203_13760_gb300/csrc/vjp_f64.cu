// Instantiations of the stage VJP kernels in FP64: 3D marches along z over
// 16 x 8 columns, 16 x 4 with viscous fluxes, whose cotangent rings of the
// tangential derivatives need the room; the FP64 plane rings fill the shared
// memory of one CTA per SM.  Threads per CTA by the tasks of a pass, as in FP32:
// 320 and 224 in 3D (64^3 step 9.86 -> 9.57 ms inviscid against 256 threads,
// 12.96 -> 11.94 ms viscous against 128), 384 in 2D (256^2 viscous step 1934 ->
// 1886 us against 256).
#include "vjp_inst.cuh"

namespace jf {

template <>
VjpLaunch<double> vjp_launcher<double>(int dim, bool visc) {
  if (dim == 3) return visc ? &launch_vjp3<double, true, 16, 4, 224, 1> : &launch_vjp3<double, false, 16, 8, 320, 1>;
  if (dim == 2)
    return visc ? &launch_vjp<double, 2, true, 16, 16, 1, 384> : &launch_vjp<double, 2, false, 16, 16, 1, 384>;
  if (dim == 1)
    return visc ? &launch_vjp<double, 1, true, 128, 1, 2, 160> : &launch_vjp<double, 1, false, 128, 1, 2, 160>;
  return nullptr;
}

}  // namespace jf
