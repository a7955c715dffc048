// ctf_mlp_ws2_w4.cu -- the packed-group learned kernels (ctf_mlp_ws2.cu)
// for warp tiles 4 pixels wide.
#define CTF_MLP_WS2_PART
#include "ctf_mlp_ws2.cu"

namespace ctf {
PfKernels pf_kernels_w4() { return pf_kernels<4>(); }
}  // namespace ctf
