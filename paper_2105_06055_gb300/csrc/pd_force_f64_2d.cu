// The 2D force pipelines in double precision (a unit of their own for build parallelism).
#define PD_FORCE_UNIT 642
#include "pd_force_impl.cuh"

namespace pd {
PD_FORCE_PIPELINES(, double, 2)
}  // namespace pd
