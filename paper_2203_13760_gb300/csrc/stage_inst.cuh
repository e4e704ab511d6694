// Launch wrappers that instantiate the stage kernel for one tile shape.
#pragma once
#include "variants.h"

namespace jf {

// MINB: CTAs per SM the register allocation must allow (__launch_bounds__).
template <typename T, int DIM, bool VISC, int BX, int BY, int MINB, int SCH>
cudaError_t prepare_stage() {
  constexpr size_t smem = launch_smem<T, DIM, VISC, BX, BY, SCH>();
  return cudaFuncSetAttribute(stage_kernel<T, DIM, VISC, BX, BY, MINB, SCH>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// NEXT: with programmatic dependence (launch_next), if the kernel allows it.
template <bool NEXT, typename... P, typename... A>
cudaError_t launch_stage_kernel(void (*k)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, A... args) {
  if constexpr (NEXT) return launch_next(k, grid, threads, smem, s, args...);
  k<<<grid, threads, smem, s>>>(static_cast<P>(args)...);
  return cudaGetLastError();
}

// CTAs that arrive while the predecessor's still run take the slots these leave,
// so that a launch that fills some slots of every SM but not all may come to rest
// on a few SMs.  An FP64 stage, which the SM's FP64 pipe bounds, then takes as long
// as its fullest SM: 160^2 (270 CTAs, three slots per SM) 86 us against 61 by plain
// launches, 20000 cells (667, eight) 29.6 against 20.1.  Such launches are plain;
// fewer CTAs than SMs spread out either way, and full SMs leave no choice.
inline bool spreads_evenly(long long ctas, int slots) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return false;
  return ctas <= sms || (ctas + sms - 1) / sms >= slots;
}

// A.zchunk: planes per CTA of a z-march (DIM_Y2: rows of the 2D grid).
template <typename T, int DIM, bool VISC, int BX, int BY, int MINB, int SCH>
cudaError_t launch_stage(const StageArgs<T>& A0, const Gas<T>& g, cudaStream_t s) {
  const size_t smem = launch_smem<T, DIM, VISC, BX, BY, SCH>();
  StageArgs<T> A = A0;
  if constexpr (DIM == DIM_Y2) rows_as_planes(A);
  const dim3 grid((A.nx + BX - 1) / BX, plane_dims(DIM) == 2 ? (A.ny + BY - 1) / BY : 1,
                  marches(DIM) ? (A.nz + A.zchunk - 1) / A.zchunk : 1);
  constexpr bool next = overlapped_launch(SCH, DIM);
  auto k = stage_kernel<T, DIM, VISC, BX, BY, MINB, SCH>;
  constexpr unsigned nt = Geo<BX, BY, DIM, VISC>::NT;
  if (next && sizeof(T) == 8 && MINB > 1 && !spreads_evenly((long long)grid.x * grid.y * grid.z, MINB))
    return launch_stage_kernel<false>(k, grid, nt, smem, s, A, nullptr, nullptr, 0, 0, g);
  return launch_stage_kernel<next>(k, grid, nt, smem, s, A, nullptr, nullptr, 0, 0, g);
}

template <typename T, int DIM, bool VISC, int BX, int BY, int MINB, int SCH>
cudaError_t prepare_batch(int* blocks_per_sm) {
  auto k = stage_kernel<T, DIM, VISC, BX, BY, MINB, SCH>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)launch_smem<T, DIM, VISC, BX, BY, SCH>());
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, Geo<BX, BY, DIM, VISC>::NT,
                                                       launch_smem<T, DIM, VISC, BX, BY, SCH>());
}

// rows: z-march kernels (3D, DIM_Y2), the planes (rows) of a work item's
// chunk (other kernels ignore it).
template <typename T, int DIM, bool VISC, int BX, int BY, int MINB, int SCH>
cudaError_t launch_batch(const SimDesc<T>* sims, const WorkItem* work, int nwork, int stage, const Gas<T>& g,
                         int* flag, int grid, int rows, cudaStream_t s) {
  const size_t smem = launch_smem<T, DIM, VISC, BX, BY, SCH>();
  StageArgs<T> A{};
  A.flag = flag;
  A.zchunk = rows;
#ifdef JF_DEBUG_BOUNDS
  A.trace = debug_trace_dev();
#endif
  // Plain where the CTAs fill the SMs for several items: programmatic dependence
  // costs a step of 64 walled 64^2 grids 7 %, viscous 10 %.  With an item per CTA (but for
  // marches) it gives time: trajectories of eight 64^2 grids 319 us, 340 the plain
  // way; so it does the network's stages of a training step (2312 us, 2427).
  auto k = stage_kernel<T, DIM, VISC, BX, BY, MINB, SCH>;
  constexpr unsigned nt = Geo<BX, BY, DIM, VISC>::NT;
  if constexpr (overlapped_launch(SCH, DIM) && !marches(DIM))
    if (SCH == SCH_NN || nwork <= grid)
      return launch_stage_kernel<true>(k, dim3(grid), nt, smem, s, A, sims, work, nwork, stage, g);
  return launch_stage_kernel<false>(k, dim3(grid), nt, smem, s, A, sims, work, nwork, stage, g);
}

template <typename T, int DIM, bool VISC, int BX, int BY, int MINB, int SCH>
StageVariant<T> make_variant() {
  StageVariant<T> v{DIM == DIM_Y2 ? 2 : DIM, VISC, BX, BY, launch_smem<T, DIM, VISC, BX, BY, SCH>(),
                    &prepare_stage<T, DIM, VISC, BX, BY, MINB, SCH>, &launch_stage<T, DIM, VISC, BX, BY, MINB, SCH>,
                    nullptr, nullptr, Geo<BX, BY, DIM, VISC>::NT, SCH, MINB, DIM == DIM_Y2};
  v.prepare_batch = &prepare_batch<T, DIM, VISC, BX, BY, MINB, SCH>;
  v.launch_batch = &launch_batch<T, DIM, VISC, BX, BY, MINB, SCH>;
  return v;
}

}  // namespace jf
