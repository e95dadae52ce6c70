// Instantiation unit: marching form, forward-Euler 5-point heat update.
#include "march.cuh"

namespace swept {
const MarchTable *marchtable_heat() { return March<HeatOp>::table(); }
}  // namespace swept
