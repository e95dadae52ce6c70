// Instantiation unit: marching form, the same with bfloat16 storage.
#include "march.cuh"

namespace swept {
const MarchTable *marchtable_euler_kahan_bf16() { return March<EulerKahanOp<__nv_bfloat16>>::table(); }
}  // namespace swept
