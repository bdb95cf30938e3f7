// sweep_f32_bnd_wide.cu - the sweep for states far from unit scale (float, boundary rules compiled in).
#include "sweep.cuh"

namespace fpk {
FPK_SWEEP_UNIT(f32_bnd_wide, float, true, 4)
}  // namespace fpk
