// Instantiation unit: marching form, Euler in binary32 with a Kahan-compensated update.
#include "march.cuh"

namespace swept {
const MarchTable *marchtable_euler_kahan_f32() { return March<EulerKahanOp<float>>::table(); }
}  // namespace swept
