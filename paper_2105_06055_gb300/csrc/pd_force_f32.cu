// Instantiation of the force pipelines for float (separate unit for build parallelism).
#define PD_FORCE_UNIT_F32
#include "pd_force_impl.cuh"

namespace pd {
PD_FORCE_INSTANCES(, float)
}  // namespace pd
