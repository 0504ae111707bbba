// TE images: a share of the line lengths (compiled apart, so that the unrolled kernels build in parallel).
#include "k_post_il.cuh"

namespace t2sh {
T2SH_POST_PART(launch_post_il_a, T2SH_POST_LENGTHS_A)
}  // namespace t2sh
