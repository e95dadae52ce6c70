// Instantiation unit: heat with a Kahan-compensated binary32 update, binary32 storage (single grid).
#include "launch.cuh"

namespace swept {
const OpTable *optable_heat_kahan_f32() { return Launch<HeatKahanOp<float>>::marching_table(); }
}  // namespace swept
