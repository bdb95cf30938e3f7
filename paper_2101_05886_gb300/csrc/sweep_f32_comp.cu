// sweep_f32_comp.cu - the component-wise sweep (float).
#include "sweep.cuh"

namespace fpk {
FPK_SWEEP_UNIT(f32_comp, float, false, 3)
}  // namespace fpk
