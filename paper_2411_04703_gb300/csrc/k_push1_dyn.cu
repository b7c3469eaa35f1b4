// First-order (CIC) particle kernel, mobile species, runtime-sized region (see push_mobile.cuh).
#include "push_mobile.cuh"

namespace gbpic {

cudaError_t launch_push1_dyn(pic_ctx *c, int si, const ExtDev &ext) { return push::launch_push_dyn<1, 0>(c, si, ext); }
cudaError_t launch_push1_dyn_ec(pic_ctx *c, int si, const ExtDev &ext) { return push::launch_push_dyn<1, 1>(c, si, ext); }

}  // namespace gbpic
