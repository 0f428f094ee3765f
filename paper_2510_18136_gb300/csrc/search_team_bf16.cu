// Team search kernels for BF16 rows read in place.
#include "search_team.cuh"

namespace nsfrb {
NSFRB_INSTANTIATE_TEAM(1)
}  // namespace nsfrb
