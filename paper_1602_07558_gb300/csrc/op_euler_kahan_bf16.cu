// Instantiation unit: the Euler system in binary32 with a Kahan-compensated update, bfloat16
// storage (single grid).
#include "launch.cuh"

namespace swept {
const OpTable *optable_euler_kahan_bf16() { return Launch<EulerKahanOp<__nv_bfloat16>>::marching_table(); }
}  // namespace swept
