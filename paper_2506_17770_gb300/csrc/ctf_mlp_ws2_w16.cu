// ctf_mlp_ws2_w16.cu -- the packed-group learned kernels (ctf_mlp_ws2.cuh)
// for warp tiles 16 pixels wide.
#include "ctf_mlp_ws2.cuh"

namespace ctf {
PfKernels pf_kernels_w16() { return pf_kernels<16>(); }
}  // namespace ctf
