// The 3D force pipelines in single precision (a unit of their own for build parallelism).
#define PD_FORCE_UNIT 323
#include "pd_force_impl.cuh"

namespace pd {
PD_FORCE_PIPELINES(, float, 3)
PD_FORCE_DISPATCH(, float)
}  // namespace pd
