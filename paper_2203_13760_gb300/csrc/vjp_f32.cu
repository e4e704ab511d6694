// Instantiations of the stage VJP kernels in FP32 (approximate division and
// square root, like the forward FP32 kernels).  Threads per CTA: the passes over
// a box or plane have nearly the same number of tasks, and the last round of a
// pass should be full.
//   3D   marches along z over 32 x 8 columns (one CTA per SM by shared memory):
//        808 tasks over the cells, 1536 over the faces, 532 over the cells with
//        halo of a plane.  576 threads hold the last in one round; 128^3 viscous
//        step 3214 us with 512 threads, 3004 with 576, 3171 with 544, 3.3-3.5 ms
//        from 608 on (spills).
//   2D   16 x 16 boxes (two CTAs per SM): 640 to 760 tasks a pass, two rounds of
//        384 threads; 256^2 viscous step 70.2 -> 67.2 us, 100 x 61 (one box per
//        SM) 51.3 -> 45.6 us against 256 threads.
//   1D   128-cell boxes: up to 134 tasks a pass, one round of 160 threads.
#include "vjp_inst.cuh"

namespace jf {

template <>
VjpLaunch<float> vjp_launcher<float>(int dim, bool visc) {
  if (dim == 3) return visc ? &launch_vjp3<float, true, 32, 8, 576, 1> : &launch_vjp3<float, false, 32, 8, 576, 1>;
  if (dim == 2)
    return visc ? &launch_vjp<float, 2, true, 16, 16, 2, 384> : &launch_vjp<float, 2, false, 16, 16, 2, 384>;
  if (dim == 1) return visc ? &launch_vjp<float, 1, true, 128, 1, 2, 160> : &launch_vjp<float, 1, false, 128, 1, 2, 160>;
  return nullptr;
}

}  // namespace jf
