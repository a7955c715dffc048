// ctf_mlp_dense.cu -- learned texel evaluations that need no selection: the
// per-pixel 4-tap filter (every pixel evaluates its four texels) and the
// decode of an explicit list of texels.
//
// The roles and the chain are those of the packed-group kernel
// (ctf_mlp_ws2.cu): per CTA (four per SM) one consumer warpgroup runs the
// tcgen05 MLP chains over 128-row tiles, and four producer warps compute the
// features straight into the layer-1 operand of a stage of 256 rows, four
// stages in rotation.  Every row is used, so a stage is exactly two chains.
//   - 4-tap: a stage holds two pixel tiles; producer warps 0 and 1 take one
//     tile each of the even stages, warps 2 and 3 of the odd ones, so the
//     producers need no barrier among themselves.  A lane computes the
//     features of its pixel's four texels: the coordinates along each axis
//     are computed once for two texels each and shared by the taps.  Row
//     128 t + 32 k + lane is tap k of pixel `lane` of tile t; the consumer
//     gathers the four rows of a pixel in tap order.
//   - decode: each producer thread computes two of the stage's rows, and the
//     consumer stores the row values to the output itself.
// What bounds it: instruction issue, of the features (about 600 warp
// instructions a pixel tile) and of the epilogues.  The kernel with one role
// per warp that this replaces ran 4-tap at 24% occupancy with the four taps
// of a pixel one after the other.
#include <cstdint>
#include <mutex>
#include <set>
#include <utility>

#define CTF_MLP_WS2_PART
#include "ctf_mlp_ws2.cu"

namespace ctf {
namespace {

constexpr int kDStages = 4;
constexpr int kDRows = 2 * kRows;  // rows of a stage
// shared memory: operand image, MMA barrier and TMEM slot, hand-over barriers, stages
constexpr int kDBar = kImgBytes, kDTmem = kDBar + 8, kDHand = kDBar + 16;
constexpr int kDStage0 = kDHand + 16 * kDStages;
constexpr int kDX = 0;                        // layer-1 operand, 32 B a row; the row values (16 B) overlay it
constexpr int kDWord = kDX + kDRows * 32;     // 4-tap: float2 (s, t) per pixel of the two tiles
constexpr int kDInfo = kDWord + 64 * 8;       // 4-tap: uint32 per pixel: pixel index, or kDOutside; bit 31 active
constexpr int kDEmpty = kDInfo + 64 * 4;      // 4-tap: int per tile: no active pixel
constexpr int kDStageBytes = kDEmpty + 16;
constexpr int kDBytes = kDStage0 + kDStages * kDStageBytes;
constexpr uint32_t kDOutside = 0x7fffffffu, kDActive = 0x80000000u;
static_assert(kDStage0 % 16 == 0 && kDStageBytes % 16 == 0, "16-byte operand buffers");
static_assert(4 * (kDBytes + 1024 + 128) <= 228 * 1024, "four CTAs fit on an SM");
static_assert(32768ull * 32768ull <= kDOutside, "a pixel index fits beside the flag");

struct DenseArgs {
    ExactParams p;   // 4-tap: the view
    const int2 *xy;  // decode: n texels
    int n, Wt, Ht;
    float4 *out;
    int *err;
};

__device__ __forceinline__ uint64_t *d_full(unsigned char *sm, int s) {
    return reinterpret_cast<uint64_t *>(sm + kDHand) + s;
}
__device__ __forceinline__ uint64_t *d_done(unsigned char *sm, int s) {
    return reinterpret_cast<uint64_t *>(sm + kDHand) + kDStages + s;
}

// One axis of a latent grid at texel coordinates c and c + 1 of the
// footprint (clamped to the texture): the cells on both sides and the
// fraction, as in texel_features.
struct GridAxis {
    int lo[2], hi[2];
    float f[2];
    __device__ __forceinline__ GridAxis(int c, int size, float scale, int cells) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int t = min(max(c + i, 0), size - 1);
            const float g = __fsub_rn(__fmul_rn(__fadd_rn((float)t, 0.5f), scale), 0.5f);
            const float g0 = floorf(g);
            f[i] = __fsub_rn(g, g0);
            const int x0 = (int)g0;
            lo[i] = min(max(x0, 0), cells - 1);
            hi[i] = min(max(x0 + 1, 0), cells - 1);
        }
    }
};

// Features of the four texels of a footprint into rows row0 + 32 k of the
// operand at X: the arithmetic of texel_features, one tap after the other.
template <bool kFp8>
__device__ __forceinline__ void quad_features(const MlpDevice &m, int ulx, int uly, int Wt, int Ht, unsigned char *X,
                                              int row0, const float *inv_a1) {
    const GridAxis x0(ulx, Wt, m.sx[0], m.gw[0]), x1(ulx, Wt, m.sx[1], m.gw[1]);
    const GridAxis y0(uly, Ht, m.sy[0], m.gh[0]), y1(uly, Ht, m.sy[1], m.gh[1]);
#pragma unroll 1
    for (int j = 0; j < 2; ++j) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float f[kMlpIn];
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const GridAxis &ax = g ? x1 : x0, &ay = g ? y1 : y0;
                const uint4 *L = reinterpret_cast<const uint4 *>(m.lat[g]);
                const long long cells = (long long)m.gw[g] * m.gh[g];
                const int ylo = j ? ay.lo[1] : ay.lo[0], yhi = j ? ay.hi[1] : ay.hi[0];
                const float fx = ax.f[i], fy = j ? ay.f[1] : ay.f[0];
                const uint4 q00 = __ldg(L + ck(ylo * m.gw[g] + ax.lo[i], cells, m.err, kBndLatent));
                const uint4 q10 = __ldg(L + ck(ylo * m.gw[g] + ax.hi[i], cells, m.err, kBndLatent));
                const uint4 q01 = __ldg(L + ck(yhi * m.gw[g] + ax.lo[i], cells, m.err, kBndLatent));
                const uint4 q11 = __ldg(L + ck(yhi * m.gw[g] + ax.hi[i], cells, m.err, kBndLatent));
                blend_latents(q00, q10, q01, q11, fx, fy, f + 8 * g);
            }
            store_x_row_at(X, row0 + 32 * (2 * j + i), f, kFp8, inv_a1);
        }
    }
}

// TW: width of the warp tile for 4-tap, 0 for the decode of a list.
template <int TW, bool kStats, bool kFp8>
__global__ void __launch_bounds__(kPThreads, kPCtasPerSm)
    mlp_dense_kernel(const DenseArgs a, const MlpDevice m, const __grid_constant__ MlpEpilogue ep) {
    constexpr bool kTap = TW != 0;
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ unsigned long long block_stats[kNumStats];
    const int lane = threadIdx.x & 31;
    const int warp = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0);
    uint64_t *mma_bar = reinterpret_cast<uint64_t *>(sm + kDBar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + kDTmem);
    if (kStats && threadIdx.x < kNumStats) block_stats[threadIdx.x] = 0;
    for (int i = threadIdx.x; i < kImgBytes / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(sm)[i] = __ldg(m.img + i);
    tc::fence_proxy_async();  // the image before the MMAs that read it
    if (threadIdx.x == 0) {
        tc::mbar_init(mma_bar, 1);
        for (int s = 0; s < kDStages; ++s) {
            tc::mbar_init(d_full(sm, s), kTap ? 2 : kPProducerWarps);
            tc::mbar_init(d_done(sm, s), 1);
        }
        tc::fence_mbar_init();
    }
    if (warp == 0) {
        __syncwarp();  // tcgen05.alloc needs the whole warp
        tc::tmem_alloc(tslot, kTmemCols);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    // (as in the packed-group kernel)
    grid_wait();
    grid_trigger();
    const uint32_t tmem = *tslot;
    Counters cnt;
#pragma unroll
    for (int i = 0; i < kNumStats; ++i) cnt.v[i] = 0;
    const long long n_groups = kTap ? (a.p.n_tiles + 1) / 2 : ((long long)a.n + kDRows - 1) / kDRows;

    if (warp < 4) {
        // ---------------- consumer ----------------
        const int tid = threadIdx.x;
        uint32_t phase = 0;
        for (long long j = 0;; ++j) {
            const long long grp = blockIdx.x + j * gridDim.x;
            if (grp >= n_groups) break;
            const int s = (int)(j % kDStages);
            unsigned char *st = sm + kDStage0 + s * kDStageBytes;
            bool ok = tc::mbar_wait(d_full(sm, s), (uint32_t)((j / kDStages) & 1), kMaxTries);
            __syncwarp();
            if (bar_or<1, kRows>(!ok)) {
                if (tid == 0) atomicExch(a.err, CTF_ERR_TIMEOUT);
                break;
            }
            float4 *outrow = reinterpret_cast<float4 *>(st + kDX);
            const uint32_t sX = tc::smem_addr(st + kDX);
            for (int c = 0; c < 2 && ok; ++c) {
                // a chain without a row to evaluate is skipped
                const bool skip = kTap ? __shfl_sync(FULL, reinterpret_cast<const int *>(st + kDEmpty)[c], 0) != 0
                                       : kRows * c >= a.n - grp * kDRows;
                if (skip) continue;
                float4 v;
                bool bad = false;
                ok = p_chain<true, kFp8>(sm, tmem, mma_bar, phase, sX + 4096u * (uint32_t)c, warp, true, ep, v, bad,
                                         a.err);
                if (!ok) break;
                if (kTap) {
                    // (chain c's values overlay operand rows of chain 0, which has been read)
                    outrow[ck(kRows * c + tid, kDRows, a.err, kBndRow)] = v;
                } else {
                    const long long row = grp * kDRows + kRows * c + tid;
                    if (row < a.n) a.out[ck(row, a.n, a.err, kBndDecodeList)] = v;
                }
                ok = !bar_or<1, kRows>(bad);
                if (!ok && tid == 0) atomicExch(a.err, CTF_ERR_TIMEOUT);
            }
            if (!ok) break;
            if (kTap && warp < 2) {
                const uint32_t info = reinterpret_cast<const uint32_t *>(st + kDInfo)[32 * warp + lane];
                const uint32_t pixel = info & kDOutside;
                if (pixel != kDOutside) {
                    const uint32_t idx = ck(pixel, view_pixels(a.p), a.err, kBndPixel);
                    float4 res = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (info & kDActive) {
                        const float2 f = reinterpret_cast<const float2 *>(st + kDWord)[32 * warp + lane];
                        float w[4];
                        bilinear_weights(f.x, f.y, w);
                        float2 rg = make_float2(0.f, 0.f), ba = make_float2(0.f, 0.f);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const float4 t = outrow[ck(kRows * warp + 32 * k + lane, kDRows, a.err, kBndRow)];
                            const float2 wk = make_float2(w[k], w[k]);
                            rg = __ffma2_rn(wk, make_float2(t.x, t.y), rg);
                            ba = __ffma2_rn(wk, make_float2(t.z, t.w), ba);
                        }
                        res = make_float4(rg.x, rg.y, ba.x, ba.y);
                    }
                    __stcs(a.p.out + idx, res);
                    if (a.p.evals) a.p.evals[idx] = (info & kDActive) ? 4 : 0;
                }
            }
            __syncwarp();
            cons_bar();  // every consumer warp has read the stage
            if (tid == 0) p_arrive(d_done(sm, s));
        }
    } else {
        // ---------------- producers ----------------
        const int pw = warp - 4;
        const float *inv_a1 = reinterpret_cast<const float *>(sm + kImgA1);
        for (long long j = kTap ? pw >> 1 : 0;; j += kTap ? 2 : 1) {
            const long long grp = blockIdx.x + j * gridDim.x;
            if (grp >= n_groups) break;
            const int s = (int)(j % kDStages);
            unsigned char *st = sm + kDStage0 + s * kDStageBytes;
            if (j >= kDStages) {  // the consumer has read group j - kDStages from this stage
                const bool ok = __all_sync(FULL, tc::mbar_wait(d_done(sm, s), (uint32_t)(((j - kDStages) / kDStages) & 1),
                                                               kMaxTries));
                if (!ok) {
                    if (lane == 0) atomicExch(a.err, CTF_ERR_TIMEOUT);
                    break;
                }
            }
            if constexpr (kTap) {
                constexpr uint32_t TH = 32 / TW;
                const ExactParams &p = a.p;
                const int t = pw & 1;
                const uint32_t tile = (uint32_t)(2 * grp) + (uint32_t)t, tiles_x = (uint32_t)p.tiles_x;
                const uint32_t by = tile / tiles_x, bx = tile - by * tiles_x;
                const uint32_t px = bx * TW + (uint32_t)lane % TW, py = by * TH + (uint32_t)lane / TW;
                const bool inside = px < (uint32_t)p.W && py < (uint32_t)p.H;
                const uint32_t idx = py * (uint32_t)p.W + px;
                const Inputs in = load_inputs_any<false>(p, inside, idx);
                PixelSetup ps;
                ps.active = inside && in.cov != 0;
                setup_coords(in.uv, (float)p.Wt, (float)p.Ht, ps);
                const uint32_t A = __ballot_sync(FULL, ps.active);
                if (kStats && tile < (uint32_t)p.n_tiles) {
                    cnt.v[kStatTilesTotal] += 1;
                    cnt.v[kStatTilesEmpty] += A == 0 ? 1 : 0;
                    cnt.v[kStatTilesDirect] += A != 0 ? 1 : 0;
                    cnt.v[kStatPixelsActive] += __popc(A);
                    cnt.v[kStatTexelEvals] += 4 * __popc(A);
                    cnt.v[kStatTexelEvalsUnique] += 4 * __popc(A);
                }
                reinterpret_cast<float2 *>(st + kDWord)[32 * t + lane] = make_float2(ps.s, ps.t);
                reinterpret_cast<uint32_t *>(st + kDInfo)[32 * t + lane] =
                    (inside ? idx : kDOutside) | (ps.active ? kDActive : 0u);
                if (lane == 0) reinterpret_cast<int *>(st + kDEmpty)[t] = A == 0;
                // (inactive lanes evaluate a texel of their own, which nobody reads)
                if (A != 0) quad_features<kFp8>(m, ps.ulx, ps.uly, p.Wt, p.Ht, st + kDX, kRows * t + lane, inv_a1);
            } else {
#pragma unroll 1
                for (int c = 0; c < 2; ++c) {
                    const int r = kRows * c + 32 * pw + lane;
                    const long long i = grp * kDRows + r;
                    if (i >= a.n) break;
                    const int2 t = a.xy[ck(i, a.n, a.err, kBndDecodeList)];
                    float f[kMlpIn];
                    texel_features(m, min(max(t.x, 0), a.Wt - 1), min(max(t.y, 0), a.Ht - 1), f);
                    store_x_row_at(st + kDX, r, f, kFp8, inv_a1);
                }
            }
            tc::fence_proxy_async();  // generic-proxy writes -> the MMAs' async proxy
            __syncwarp();
            if (lane == 0) p_arrive(d_full(sm, s));
        }
    }

    if (kStats && a.p.stats && lane == 0) {
#pragma unroll
        for (int i = 0; i < kNumStats; ++i)
            if (cnt.v[i]) atomicAdd(&block_stats[i], (unsigned long long)cnt.v[i]);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();  // tcgen05.dealloc needs the whole warp
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, kTmemCols);
    }
    if (kStats && a.p.stats && threadIdx.x < kNumStats && block_stats[threadIdx.x])
        atomicAdd(a.p.stats + threadIdx.x, block_stats[threadIdx.x]);
}

using DenseFn = void (*)(const DenseArgs, const MlpDevice, const MlpEpilogue);

template <int TW>
DenseFn dense_pick(bool stats, bool fp8) {
    if constexpr (TW != 0) {
        if (stats) return fp8 ? mlp_dense_kernel<TW, true, true> : mlp_dense_kernel<TW, true, false>;
    }
    return fp8 ? mlp_dense_kernel<TW, false, true> : mlp_dense_kernel<TW, false, false>;
}

DenseFn dense_kernel(int tile_w, bool stats, bool fp8) {
    switch (tile_w) {
    case 0: return dense_pick<0>(false, fp8);
    case 8: return dense_pick<8>(stats, fp8);
    case 4: return dense_pick<4>(stats, fp8);
    case 16: return dense_pick<16>(stats, fp8);
    default: return nullptr;
    }
}

cudaError_t dense_prepare(DenseFn fn) {
    static std::mutex mu;
    static std::set<std::pair<int, const void *>> done;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair(dev, reinterpret_cast<const void *>(fn));
    if (done.count(key)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kDBytes);
    if (e == cudaSuccess) done.insert(key);
    return e;
}

cudaError_t dense_launch(const DenseArgs &a, const MlpDevice &m, const MlpEpilogue &ep, DenseFn fn, long long groups,
                         cudaStream_t stream) {
    cudaError_t e = dense_prepare(fn);
    if (e != cudaSuccess) return e;
    const long long cap = (long long)device_sm_count() * kPCtasPerSm;
    return launch_dependent(fn, (int)(groups < cap ? groups : cap), kPThreads, kDBytes, stream, a, m, ep);
}

}  // namespace

cudaError_t launch_mlp_decode(const MlpDevice &m, const MlpEpilogue &ep, int Wt, int Ht, const int2 *xy, int n,
                              float4 *out, int *err, cudaStream_t stream) {
    if (n <= 0) return cudaSuccess;
    DenseArgs a{};
    a.xy = xy;
    a.n = n;
    a.Wt = Wt;
    a.Ht = Ht;
    a.out = out;
    a.err = err;
    return dense_launch(a, m, ep, dense_kernel(0, false, m.fp8 != 0), ((long long)n + kDRows - 1) / kDRows, stream);
}

cudaError_t prepare_mlp_4tap(int tile_w) {
    for (int v = 0; v < 4; ++v) {
        DenseFn fn = dense_kernel(tile_w, (v & 1) != 0, (v & 2) != 0);
        if (!fn || tile_w == 0) return cudaErrorInvalidValue;
        const cudaError_t e = dense_prepare(fn);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_mlp_4tap(const ExactParams &p, const MlpDevice &m, const MlpEpilogue &ep, int tile_w, int *err,
                            cudaStream_t stream) {
    DenseFn fn = tile_w == 0 ? nullptr : dense_kernel(tile_w, p.stats != nullptr, m.fp8 != 0);
    if (!fn) return cudaErrorInvalidValue;
    if (p.n_tiles == 0) return cudaSuccess;
    if (p.n_tiles > 0x7fffffffLL) return cudaErrorInvalidValue;  // tile positions use 32-bit arithmetic
    DenseArgs a{};
    a.p = p;
    a.err = err;
    return dense_launch(a, m, ep, fn, (p.n_tiles + 1) / 2, stream);
}

}  // namespace ctf
