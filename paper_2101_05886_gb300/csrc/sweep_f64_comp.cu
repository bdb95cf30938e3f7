// sweep_f64_comp.cu - the component-wise sweep (double).
#include "sweep.cuh"

namespace fpk {
FPK_SWEEP_UNIT(f64_comp, double, false, 3)
}  // namespace fpk
