// Second-order (TSC) particle kernel, mobile species on the default tile (see push_mobile.cuh).
#include "push_mobile.cuh"

namespace gbpic {

cudaError_t launch_push2_fixed(pic_ctx *c, int si, const ExtDev &ext) { return push::launch_push_fixed<2, 0>(c, si, ext); }

}  // namespace gbpic
