// Mid-window search kernels for F16 rows read in place.
#include "search_mid.cuh"

namespace nsfrb {
NSFRB_INSTANTIATE_MID(2)
}  // namespace nsfrb
