// Second-order (TSC) particle kernel, mobile species on the default tile, energy-conserving gather (see push_mobile.cuh).
#include "push_mobile.cuh"

namespace gbpic {

cudaError_t launch_push2_fixed_ec(pic_ctx *c, int si, const ExtDev &ext) { return push::launch_push_fixed<2, 1>(c, si, ext); }

}  // namespace gbpic
