// ctf_mlp_ws2_w8.cu -- the packed-group learned kernels (ctf_mlp_ws2.cuh)
// for warp tiles 8 pixels wide.
#include "ctf_mlp_ws2.cuh"

namespace ctf {
PfKernels pf_kernels_w8() { return pf_kernels<8>(); }
}  // namespace ctf
