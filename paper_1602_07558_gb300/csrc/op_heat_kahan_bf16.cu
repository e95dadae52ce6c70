// Instantiation unit: heat with a Kahan-compensated binary32 update, bfloat16 storage (single grid).
#include "launch.cuh"

namespace swept {
const OpTable *optable_heat_kahan_bf16() { return Launch<HeatKahanOp<__nv_bfloat16>>::marching_table(); }
}  // namespace swept
