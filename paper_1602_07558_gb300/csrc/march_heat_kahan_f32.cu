// Instantiation unit: marching form, heat in binary32 with a Kahan-compensated update.
#include "march.cuh"

namespace swept {
const MarchTable *marchtable_heat_kahan_f32() { return March<HeatKahanOp<float>>::table(); }
}  // namespace swept
