// Instantiation of the boundary-field sums (one unit).
#define PD_HORIZON_UNIT
#include "pd_horizon.cuh"

namespace pd {
PD_GFIELD_INSTANCES()
}  // namespace pd
