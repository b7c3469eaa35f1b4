// Second-order (TSC) particle kernel, mobile species, runtime-sized region (see push_mobile.cuh).
#include "push_mobile.cuh"

namespace gbpic {

cudaError_t launch_push2_dyn(pic_ctx *c, int si, const ExtDev &ext) { return push::launch_push_dyn<2, 0>(c, si, ext); }

}  // namespace gbpic
