// Wide-window search kernels for BF16 rows read in place.
#include "search_wide.cuh"

namespace nsfrb {
NSFRB_INSTANTIATE_WIDE(1)
}  // namespace nsfrb
