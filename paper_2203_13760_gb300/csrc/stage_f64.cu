// Instantiations of the stage kernel in FP64 (divisions and square roots:
// approximation and refinement steps, trcp / tsqrt).
#include <vector>

#include "stage_inst.cuh"

namespace jf {

// The default-scheme kernels (WENO5-JS, HLLC, Einfeldt) of every tile shape,
// then the run-time-scheme kernels of stage_f64_gen.cu (one tile shape each)
// and the flux-splitting kernels of stage_f64_roe.cu.
template <>
const StageVariant<double>* stage_variants<double>(int* count) {
  static const std::vector<StageVariant<double>> table = [] {
    std::vector<StageVariant<double>> v = {
      // 3D (the first entry per configuration is the default): 32 x 7, one
      // CTA of 8 warps per SM, the z state of a column in registers (with
      // it, the carried viscous stencils and the tile 32 x 6 -> 32 x 7 the
      // 128^3 step went from 22.7 to 20.3 ms)
      make_variant<double, 3, true, 32, 7, 1, SCH_DEFAULT>(),
      make_variant<double, 3, true, 32, 4, 1, SCH_DEFAULT>(),
      make_variant<double, 3, true, 32, 2, 2, SCH_DEFAULT>(),
      make_variant<double, 3, false, 32, 7, 1, SCH_DEFAULT>(),
      make_variant<double, 3, false, 32, 4, 1, SCH_DEFAULT>(),
      make_variant<double, 3, false, 32, 2, 2, SCH_DEFAULT>(),
      // 2D
      make_variant<double, 2, true, 32, 8, 1, SCH_DEFAULT>(),
      make_variant<double, 2, true, 32, 4, 2, SCH_DEFAULT>(),
      make_variant<double, 2, true, 32, 3, 3, SCH_DEFAULT>(),
      make_variant<double, 2, false, 32, 8, 1, SCH_DEFAULT>(),
      make_variant<double, 2, false, 32, 4, 2, SCH_DEFAULT>(),
      make_variant<double, 2, false, 32, 3, 3, SCH_DEFAULT>(),
      // 1D: 30 cells, whatever the length (stage of 200, 20000 and 10^6 cells in
      // 128-cell tiles 26.0, 46.7 and 1100 us, now 8.3, 20.1 and 753)
      make_variant<double, 1, true, 30, 1, 8, SCH_DEFAULT>(),
      make_variant<double, 1, false, 30, 1, 8, SCH_DEFAULT>(),
    };
    int ng = 0;
    const StageVariant<double>* gen = general_variants_f64(&ng);
    v.insert(v.end(), gen, gen + ng);
    const StageVariant<double>* roe = roe_variants_f64(&ng);
    v.insert(v.end(), roe, roe + ng);
    const StageVariant<double>* nn = nn_variants_f64(&ng);
    v.insert(v.end(), nn, nn + ng);
    const StageVariant<double>* ext = ext_variants_f64(&ng);
    v.insert(v.end(), ext, ext + ng);
    const StageVariant<double>* rows = rows_variants_f64(&ng);
    v.insert(v.end(), rows, rows + ng);
    return v;
  }();
  *count = (int)table.size();
  return table.data();
}

}  // namespace jf
