// Instantiation unit: the Euler system in binary32 with a Kahan-compensated update, binary32
// storage (single grid).
#include "launch.cuh"

namespace swept {
const OpTable *optable_euler_kahan_f32() { return Launch<EulerKahanOp<float>>::marching_table(); }
}  // namespace swept
