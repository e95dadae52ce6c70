// Instantiation unit: marching form, the same with bfloat16 storage.
#include "march.cuh"

namespace swept {
const MarchTable *marchtable_heat_kahan_bf16() { return March<HeatKahanOp<__nv_bfloat16>>::table(); }
}  // namespace swept
