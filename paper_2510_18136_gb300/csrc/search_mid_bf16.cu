// Mid-window search kernels for BF16 rows read in place.
#include "search_mid.cuh"

namespace nsfrb {
NSFRB_INSTANTIATE_MID(1)
}  // namespace nsfrb
