// First-order (CIC) instantiations of the particle kernels: frozen species, and mobile species on
// the default tile (see push_impl.cuh, push_mobile.cuh).
#include "push_mobile.cuh"

namespace gbpic {

cudaError_t launch_push1_frozen(pic_ctx *c, int si) { return push::launch_frozen<1>(c, si); }
cudaError_t launch_push1_fixed(pic_ctx *c, int si, const ExtDev &ext) { return push::launch_push_fixed<1, 0>(c, si, ext); }
cudaError_t launch_push1_fixed_ec(pic_ctx *c, int si, const ExtDev &ext) { return push::launch_push_fixed<1, 1>(c, si, ext); }

}  // namespace gbpic
