// The 2D force pipelines in single precision (a unit of their own for build parallelism).
#define PD_FORCE_UNIT 322
#include "pd_force_impl.cuh"

namespace pd {
PD_FORCE_PIPELINES(, float, 2)
}  // namespace pd
