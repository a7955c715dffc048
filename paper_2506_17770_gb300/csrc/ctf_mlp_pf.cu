// ctf_mlp_pf.cu -- launches of the packed-group learned kernels
// (ctf_mlp_ws2.cu): single views and the learned views of a batch.
#include <cstdint>
#include <mutex>
#include <set>
#include <utility>
#include <cuda_runtime.h>

#include "ctf_internal.h"
#include "ctf_mlp_pf.h"
#include "ctf_select.cuh"

namespace ctf {
namespace {

// The kernels for a tile width (8, 4 or 16).
const PfKernels *kernels_of(int tile_w) {
    static const PfKernels w8 = pf_kernels_w8(), w4 = pf_kernels_w4(), w16 = pf_kernels_w16();
    return tile_w == 8 ? &w8 : tile_w == 4 ? &w4 : tile_w == 16 ? &w16 : nullptr;
}

cudaError_t pf_prepare(const void *fn, int smem_bytes, int launch_regs) {
    static std::mutex mu;
    static std::set<std::pair<int, const void *>> done;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair(dev, fn);
    if (done.count(key)) return cudaSuccess;
    // more CTAs on an SM than the layout expects would find no free TMEM;
    // fewer (a build with more registers) would be slower than measured
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e != cudaSuccess) return e;
    if (fa.numRegs > launch_regs) return cudaErrorInvalidDeviceFunction;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
    if (e == cudaSuccess) done.insert(key);
    return e;
}

}  // namespace

bool mlp_filter_pf_fallback_applies(const ExactParams &p, int alg) {
    return (alg == ALG_BOX || alg == ALG_MASK) && p.fallback != 0 && p.tpl == 1 && !p.group_dedup;
}

bool mlp_filter_pf_two_applies(const ExactParams &p, int alg) {
    return (alg == ALG_LIST || alg == ALG_BOX || alg == ALG_MASK) && p.fallback == 0 && p.tpl == 2 && !p.group_dedup;
}

cudaError_t prepare_mlp_filter_pf(int alg, int tile_w, int mask_dim) {
    const PfKernels *k = kernels_of(tile_w);
    if (!k) return cudaErrorInvalidValue;
    for (int var = 0; var < kPfNumVars; ++var)
        for (int v = 0; v < 4; ++v) {
            PfFn fn = k->filter(alg, mask_dim, (v & 1) != 0, var, (v & 2) != 0);
            if (!fn) continue;  // no such variant for this algorithm
            const cudaError_t e = pf_prepare(reinterpret_cast<const void *>(fn), k->smem[var], k->launch_regs);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

cudaError_t launch_mlp_filter_pf(const ExactParams &p, const MlpDevice &m, const MlpEpilogue &ep, int alg, int tile_w,
                                 int mask_dim, int *err, cudaStream_t stream) {
    const int var = p.fallback != 0 ? kPfFallback : (p.tpl == 2 ? kPfTwoTexels : kPfPlain);
    if (var == kPfFallback && !mlp_filter_pf_fallback_applies(p, alg)) return cudaErrorInvalidValue;
    if (var == kPfTwoTexels && !mlp_filter_pf_two_applies(p, alg)) return cudaErrorInvalidValue;
    const PfKernels *k = kernels_of(tile_w);
    PfFn fn = k ? k->filter(alg, mask_dim, p.stats != nullptr, var, m.fp8 != 0) : nullptr;
    if (!fn) return cudaErrorInvalidValue;
    if (p.n_tiles == 0) return cudaSuccess;
    if (p.n_tiles > 0x7fffffffLL) return cudaErrorInvalidValue;  // tile positions use 32-bit arithmetic
    cudaError_t e = pf_prepare(reinterpret_cast<const void *>(fn), k->smem[var], k->launch_regs);
    if (e != cudaSuccess) return e;
    const long long groups = (p.n_tiles + k->tiles[var] - 1) / k->tiles[var];
    const long long cap = (long long)device_sm_count() * k->ctas_per_sm;
    const int grid = (int)(groups < cap ? groups : cap);
    return launch_dependent(fn, grid, k->threads, k->smem[var], stream, p, m, ep, err);
}

int mlp_batch_pf_tiles() { return kernels_of(8)->tiles[kPfPlain]; }

bool mlp_batch_pf_applies(int alg, int group_dedup) {
    return (alg == ALG_STF || alg == ALG_LIST || alg == ALG_BOX || alg == ALG_MASK) && !group_dedup;
}

cudaError_t prepare_mlp_batch_pf(int alg, int tile_w, int mask_dim) {
    const PfKernels *k = kernels_of(tile_w);
    if (!k) return cudaErrorInvalidValue;
    for (int st = 0; st < 2; ++st) {
        BatchPfFn fn = k->batch(alg, mask_dim, st != 0);
        if (!fn) return cudaErrorInvalidValue;
        const cudaError_t e = pf_prepare(reinterpret_cast<const void *>(fn), k->batch_smem, k->launch_regs);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_mlp_batch_pf(const BatchViewDev *views, int nviews, const int *index, const long long *item_begin,
                                int nkind, long long total_items, unsigned long long *stats, int *err,
                                const MlpDevice &m0, const MlpEpilogue &ep0, int alg, int tile_w, int mask_dim,
                                cudaStream_t s) {
    const PfKernels *k = kernels_of(tile_w);
    BatchPfFn fn = k ? k->batch(alg, mask_dim, stats != nullptr) : nullptr;
    if (!fn) return cudaErrorInvalidValue;
    if (total_items <= 0) return cudaSuccess;
    cudaError_t e = pf_prepare(reinterpret_cast<const void *>(fn), k->batch_smem, k->launch_regs);
    if (e != cudaSuccess) return e;
    PfBatch b;
    b.views = views;
    b.index = index;
    b.item_begin = item_begin;
    b.nkind = nkind;
    b.nviews = nviews;
    b.total_items = total_items;
    b.stats = stats;
    b.err = err;
    const long long cap = (long long)device_sm_count() * k->ctas_per_sm;
    const int grid = (int)(total_items < cap ? total_items : cap);
    return launch_dependent(fn, grid, k->threads, k->batch_smem, s, b, m0, ep0);
}

}  // namespace ctf
