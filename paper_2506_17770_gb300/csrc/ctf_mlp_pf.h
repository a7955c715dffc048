// ctf_mlp_pf.h -- the host's view of the packed-group kernels of
// ctf_mlp_ws2.cu, which are compiled in one unit per tile width
// (ctf_mlp_ws2.cu itself, _w4.cu, _w16.cu) and launched from ctf_mlp_pf.cu.
#pragma once
#include <cuda_runtime.h>

#include "ctf_internal.h"
#include "ctf_mlp.cuh"

namespace ctf {

// Arguments of the persistent batch kernel.
struct PfBatch {
    const BatchViewDev *views;
    const int *index;
    const long long *item_begin;
    int nkind, nviews;
    long long total_items;
    unsigned long long *stats;
    int *err;
};

using PfFn = void (*)(const ExactParams, const MlpDevice, const MlpEpilogue, int *);
using BatchPfFn = void (*)(const PfBatch, const MlpDevice, const MlpEpilogue);

// Variants: plain, fallbacks C / C+ (Box and Mask), two texels per lane
// (List Merge, Box and Mask).
enum { kPfPlain = 0, kPfFallback = 1, kPfTwoTexels = 2, kPfNumVars = 3 };

// The kernels of one tile width (nullptr where a variant does not exist) and
// their launch shape.
struct PfKernels {
    PfFn (*filter)(int alg, int mask_dim, bool stats, int var, bool fp8);
    BatchPfFn (*batch)(int alg, int mask_dim, bool stats);
    int threads, launch_regs, ctas_per_sm;
    int tiles[kPfNumVars];  // tiles of a group
    int smem[kPfNumVars];   // dynamic shared memory
    int batch_smem;
};
PfKernels pf_kernels_w8();
PfKernels pf_kernels_w4();
PfKernels pf_kernels_w16();

}  // namespace ctf
