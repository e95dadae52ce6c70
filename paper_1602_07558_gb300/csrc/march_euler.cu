// Instantiation unit: marching form, Euler, midpoint RK2.
#include "march.cuh"

namespace swept {
const MarchTable *marchtable_euler() { return March<EulerOp>::table(); }
}  // namespace swept
