// Instantiation of the force pipelines for double (separate unit for build parallelism).
#define PD_FORCE_UNIT_F64
#include "pd_force_impl.cuh"

namespace pd {
PD_FORCE_INSTANCES(, double)
}  // namespace pd
