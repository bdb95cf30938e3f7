// sweep_f32_wide.cu - the sweep for states far from unit scale (float).
#include "sweep.cuh"

namespace fpk {
FPK_SWEEP_UNIT(f32_wide, float, false, 4)
}  // namespace fpk
