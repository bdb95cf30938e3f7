// sweep_f32_bnd_comp.cu - the component-wise sweep (float, boundary rules compiled in).
#include "sweep.cuh"

namespace fpk {
FPK_SWEEP_UNIT(f32_bnd_comp, float, true, 3)
}  // namespace fpk
