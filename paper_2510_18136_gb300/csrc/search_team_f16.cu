// Team search kernels for F16 rows read in place.
#include "search_team.cuh"

namespace nsfrb {
NSFRB_INSTANTIATE_TEAM(2)
}  // namespace nsfrb
