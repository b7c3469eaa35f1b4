// Second-order (TSC) kernel of frozen species (see push_impl.cuh).
#include "push_impl.cuh"

namespace gbpic {

cudaError_t launch_push2_frozen(pic_ctx *c, int si) { return push::launch_frozen<2>(c, si); }

}  // namespace gbpic
