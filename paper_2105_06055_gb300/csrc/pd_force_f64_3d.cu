// The 3D force pipelines in double precision (a unit of their own for build parallelism).
#define PD_FORCE_UNIT 643
#include "pd_force_impl.cuh"

namespace pd {
PD_FORCE_PIPELINES(, double, 3)
PD_FORCE_DISPATCH(, double)
}  // namespace pd
