// Second-order (TSC) particle kernel, frozen species (see push_impl.cuh).
#include "push_mobile.cuh"

namespace gbpic {

cudaError_t launch_push2_frozen(pic_ctx *c, int si, const ExtDev &ext) { return push::launch_frozen<2>(c, si, ext); }

}  // namespace gbpic
