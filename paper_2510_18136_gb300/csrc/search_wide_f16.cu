// Wide-window search kernels for F16 rows read in place.
#include "search_wide.cuh"

namespace nsfrb {
NSFRB_INSTANTIATE_WIDE(2)
}  // namespace nsfrb
