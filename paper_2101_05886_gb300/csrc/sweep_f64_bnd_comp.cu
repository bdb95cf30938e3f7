// sweep_f64_bnd_comp.cu - the component-wise sweep (double, boundary rules compiled in).
#include "sweep.cuh"

namespace fpk {
FPK_SWEEP_UNIT(f64_bnd_comp, double, true, 3)
}  // namespace fpk
