// ctf_bicubic.cu -- the exact-decode filter with the bicubic filters of
// Sec. 4.2 (cubic B-spline and Catmull-Rom over a 4x4 footprint): per-pixel
// 16-tap, one-tap STF, List Merge, Box Sampling and Mask Sampling.
//
// The paper notes that the algorithms serve any discrete filter, with only
// the footprint corners, the weights, the bits each pixel sets and the final
// loop changed (Sec. 4.2, Appendix).  So this kernel is the bilinear one of
// ctf_filter.cu with a 4x4 footprint: the texels from one left of and above
// the upper-left texel of the bilinear footprint, separable weights
// w_x(s) w_y(t), a 4x4 block of bits per pixel in the mask, 16 taps gathered
// by shuffles and summed as acc = fma(w_k, p_k, acc) in tap order
// k = 4 j + i.  Minified and over-budget warps take one-tap STF, which draws
// a tap per axis with probability |w| / sum |w|; Catmull-Rom's negative
// lobes scale the texel by the signed sums.  One texel per lane, block
// textures only.
#include <climits>
#include <cstdint>
#include <cuda_runtime.h>

#include "ctf_device.cuh"
#include "ctf_internal.h"
#include "ctf_select.cuh"
#include "ctf_exact_tile.cuh"

namespace ctf {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;

// 1-D cubic weights of the taps at -1, 0, 1, 2 from the upper-left texel,
// f in [0, 1); every term one round-to-nearest operation in the order
// written.  B-spline: ((1-f)^3, 3f^3 - 6f^2 + 4, -3f^3 + 3f^2 + 3f + 1,
// f^3) / 6; Catmull-Rom: (2f^2 - f^3 - f, 3f^3 - 5f^2 + 2,
// -3f^3 + 4f^2 + f, f^3 - f^2) / 2.
template <int FILT>
__device__ __forceinline__ void cubic_weights(float f, float w[4]) {
    const float f2 = __fmul_rn(f, f), f3 = __fmul_rn(f2, f);
    if (FILT == 1) {
        const float u = __fsub_rn(1.0f, f);
        w[0] = __fdiv_rn(__fmul_rn(__fmul_rn(u, u), u), 6.0f);
        w[1] = __fdiv_rn(__fadd_rn(__fsub_rn(__fmul_rn(3.0f, f3), __fmul_rn(6.0f, f2)), 4.0f), 6.0f);
        w[2] = __fdiv_rn(
            __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(-3.0f, f3), __fmul_rn(3.0f, f2)), __fmul_rn(3.0f, f)), 1.0f),
            6.0f);
        w[3] = __fdiv_rn(f3, 6.0f);
    } else {
        w[0] = __fmul_rn(0.5f, __fsub_rn(__fsub_rn(__fmul_rn(2.0f, f2), f3), f));
        w[1] = __fmul_rn(0.5f, __fadd_rn(__fsub_rn(__fmul_rn(3.0f, f3), __fmul_rn(5.0f, f2)), 2.0f));
        w[2] = __fmul_rn(0.5f, __fadd_rn(__fadd_rn(__fmul_rn(-3.0f, f3), __fmul_rn(4.0f, f2)), f));
        w[3] = __fmul_rn(0.5f, __fsub_rn(f3, f2));
    }
}

// One of 4 taps drawn with probability |w_i| / sum |w|: cumulative sums in
// tap order, the first i with xi S < c_i; g = S with the sign of w_i.
__device__ __forceinline__ int pick_tap(const float w[4], float xi, float &g) {
    const float a0 = fabsf(w[0]), a1 = fabsf(w[1]), a2 = fabsf(w[2]), a3 = fabsf(w[3]);
    const float c0 = a0, c1 = __fadd_rn(c0, a1), c2 = __fadd_rn(c1, a2), S = __fadd_rn(c2, a3);
    const float t = __fmul_rn(xi, S);
    const int i = t < c0 ? 0 : (t < c1 ? 1 : (t < c2 ? 2 : 3));
    // (selects: an indexed array would go through local memory)
    g = (i == 0 ? w[0] : i == 1 ? w[1] : i == 2 ? w[2] : w[3]) < 0.f ? -S : S;
    return i;
}

// What bounds it: instructions issued.  A 1920x1080 Mask view with Catmull-Rom,
// magnified 1 to 32 times: 46.4 us with a 64-bit division a tile, the inputs
// loaded when they are needed, a rank per tap and a mask word per footprint
// row, 28.3 us now.  Five or six CTAs per SM take 28.8 and 31.1 us; the taps by
// 16-byte reads from shared memory instead of three shuffles 28.0.
template <int ALG, int TW, int MD, int FILT, bool kStats>
__global__ void __launch_bounds__(kThreads, 4) bicubic_filter_kernel(const ExactParams p) {
    constexpr int TH = 32 / TW;
    constexpr bool kJac = ALG >= ALG_LIST;
    constexpr int NW = (MD * MD + 31) / 32;
    __shared__ DecodeTables tabs;
    __shared__ int rank_slots[kWarps][32];
    __shared__ unsigned long long block_stats[kNumStats];

    if (threadIdx.x < kNumStats) block_stats[threadIdx.x] = 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int *ranks = rank_slots[warp];
    const int tx = lane % TW, ty = lane / TW;
    const uint32_t lt = lanemask_lt();
    Counters cnt;
#pragma unroll
    for (int i = 0; i < kNumStats; ++i) cnt.v[i] = 0;
    const float fW = (float)p.Wt, fH = (float)p.Ht;

    // the tile walk and the prefetch of the bilinear kernel (ctf_filter.cu)
    const uint32_t W = (uint32_t)p.W, H = (uint32_t)p.H;
    const uint32_t ntiles = (uint32_t)p.n_tiles, tiles_x = (uint32_t)p.tiles_x;
    const uint32_t lim_x = (W - (uint32_t)tx + TW - 1) / TW, lim_y = (H - (uint32_t)ty + TH - 1) / TH;
    const uint32_t lane_off = (uint32_t)ty * W + (uint32_t)tx;
    const uint32_t stride = gridDim.x * kWarps;
    const uint32_t sbx = stride % tiles_x, sby = stride / tiles_x;
    const uint32_t tile0 = blockIdx.x * kWarps + warp;
    const uint32_t n_mine = tile0 < ntiles ? (ntiles - 1u - tile0) / stride + 1u : 0u;
    uint32_t nbx = tile0 % tiles_x, nby = tile0 / tiles_x;
    bool ninside = n_mine > 0 && nbx < lim_x && nby < lim_y;
    uint32_t nidx = nby * (TH * W) + nbx * TW + lane_off;
    DecodeTableLoad<kThreads> tl;
    tl.load(p.tables);
    grid_wait();
    grid_trigger();
    Inputs nxt = load_inputs_any<kJac>(p, ninside, nidx);
    tl.store(&tabs);
    __syncthreads();

    for (uint32_t it = 0; it < n_mine; ++it) {
        const int px = (int)(nbx * TW) + tx, py = (int)(nby * TH) + ty;
        const bool inside = ninside;
        const uint32_t idx = nidx;
        const Inputs in = nxt;
        nbx += sbx;
        nby += sby;
        if (nbx >= tiles_x) {
            nbx -= tiles_x;
            ++nby;
        }
        ninside = it + 1u < n_mine && nbx < lim_x && nby < lim_y;
        nidx = nby * (TH * W) + nbx * TW + lane_off;
        nxt = load_inputs_any<kJac>(p, ninside, nidx);
        PixelSetup ps;
        ps.active = inside && in.cov != 0;
        setup_coords(in.uv, fW, fH, ps);
        const int ox = ps.ulx - 1, oy = ps.uly - 1;  // the 4x4 footprint's corner
        float wx[4], wy[4];
        cubic_weights<FILT>(ps.s, wx);
        cubic_weights<FILT>(ps.t, wy);

        const uint32_t A = __ballot_sync(FULL, ps.active);
        const int nactive = __popc(A);
        if (kStats) {
            cnt.v[kStatTilesTotal] += 1;
            cnt.v[kStatPixelsActive] += nactive;
            if (A == 0) cnt.v[kStatTilesEmpty] += 1;
        }
        float4 res = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t count = 0;
        if (A == 0) {
            if (inside) store_pixel(p, idx, res, 0);
            continue;
        }

        if (ALG == ALG_4TAP) {  // per pixel: all 16 taps
            if (kStats) {
                cnt.v[kStatTilesDirect] += 1;
                cnt.v[kStatTexelEvals] += 16 * nactive;
                cnt.v[kStatTexelEvalsUnique] += 16 * nactive;
            }
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
            for (int k = 0; k < 16; ++k) {
                const float w = __fmul_rn(wx[k & 3], wy[k >> 2]);
                const float3 v = fetch_decode(p, ox + (k & 3), oy + (k >> 2), &tabs);
                acc.x = __fmaf_rn(w, v.x, acc.x);
                acc.y = __fmaf_rn(w, v.y, acc.y);
                acc.z = __fmaf_rn(w, v.z, acc.z);
                acc.w = __fmaf_rn(w, 1.0f, acc.w);
            }
            if (ps.active) {
                res = acc;
                count = 16;
            }
            if (inside) store_pixel(p, idx, res, (uint8_t)count);
            continue;
        }

        // ---- step 1: minification vote, the texel set, the success test
        bool fits = false, mini = false;
        int n = 0, minx = 0, miny = 0, bw = 0, bh = 0, mcls = 0;
        uint32_t word = 0;            // a mask of one word (mcls 1); else lane w holds word w
        int before = 0;               // and the number of bits in the words before it
        ListUnion<4> lu;              // List Merge with a larger box (mcls 4)
        uint32_t lsrc[4];             // List Merge: list indices of the taps, four a word
        if (ALG >= ALG_LIST) {
            mini = __any_sync(FULL, ps.active && is_minified(in.jac, fW, fH));
            if (!mini) {
                minx = __reduce_min_sync(FULL, ps.active ? ox : INT_MAX);
                miny = __reduce_min_sync(FULL, ps.active ? oy : INT_MAX);
                const int maxx = __reduce_max_sync(FULL, ps.active ? ox : INT_MIN) + 3;
                const int maxy = __reduce_max_sync(FULL, ps.active ? oy : INT_MIN) + 3;
                bw = maxx - minx + 1;
                bh = maxy - miny + 1;
                const int t00 = (oy - miny) * bw + (ox - minx);
                if (ALG == ALG_BOX) {
                    if (bw <= p.budget && bh <= p.budget && bw * bh <= p.budget) {
                        n = bw * bh;
                        fits = true;
                    }
                } else {
                    // Mask Sampling, and List Merge with a box of at most 16 x 16
                    // (the same set; larger boxes: one distinct texel at a time)
                    if (bw <= MD && bh <= MD) {
                        const int area = bw * bh;
                        mcls = area <= 32 ? 1 : 3;
                        // a pixel's bits: the 4 rows of a footprint at the
                        // box's corner (the same for every lane), moved by t00
                        if (mcls == 1) {
                            const uint32_t rows = 0xFu | (0xFu << bw) | (0xFu << (2 * bw)) | (0xFu << (3 * bw));
                            word = __reduce_or_sync(FULL, ps.active ? rows << t00 : 0u);
                            n = __popc(word);
                        } else {
                            const unsigned long long rows =
                                0xFull | (0xFull << bw) | (0xFull << (2 * bw)) | (0xFull << (3 * bw));
                            const uint32_t r0 = ps.active ? (uint32_t)rows : 0u, r1 = ps.active ? (uint32_t)(rows >> 32) : 0u;
                            const int sh = t00 & 31, w0 = t00 >> 5;
                            const uint32_t m0 = r0 << sh, m1 = __funnelshift_l(r0, r1, sh), m2 = __funnelshift_l(r1, 0u, sh);
#pragma unroll
                            for (int w = 0; w < NW; ++w) {
                                if (32 * w >= area || n > p.budget) break;
                                const uint32_t m = w == w0 ? m0 : (w == w0 + 1 ? m1 : (w == w0 + 2 ? m2 : 0u));
                                const uint32_t all = __reduce_or_sync(FULL, m);
                                if (lane == w) {
                                    word = all;
                                    before = n;
                                }
                                n += __popc(all);
                            }
                        }
                        fits = n <= p.budget;
                    } else if (ALG == ALG_LIST) {
                        mcls = 4;
                        lu = list_union<4, false>(ps.active, ox, oy, p.budget, lane, lt, ranks, p.err);
                        n = lu.n;
#pragma unroll
                        for (int r = 0; r < 4; ++r) lsrc[r] = lu.idx[r];
                        fits = n <= p.budget;
                    }
                }
                if (fits) {
                    if (p.edge_remap) {
                        fits = n <= nactive;
                    } else {
                        const uint32_t need = n >= 32 ? FULL : ((1u << n) - 1u);
                        fits = (A & need) == need;
                    }
                }
            }
        }

        if (!fits) {
            // ---- one-tap STF (minified, over budget, or the STF algorithm)
            if (kStats) {
                if (ALG >= ALG_LIST) {
                    cnt.v[kStatTilesFallbackMinified] += mini ? 1 : 0;
                    cnt.v[kStatTilesFallbackBudget] += mini ? 0 : 1;
                } else {
                    cnt.v[kStatTilesDirect] += 1;
                }
                cnt.v[kStatTexelEvals] += nactive;
                cnt.v[kStatTexelEvalsUnique] += nactive;
            }
            uint4 r = philox4x32_10(make_uint4((uint32_t)px, (uint32_t)(py + p.y0), (uint32_t)p.view, 0u), p.k0, p.k1);
            float gx, gy;
            const int i = pick_tap(wx, __fmul_rn((float)(r.x >> 8), 5.9604644775390625e-08f), gx);
            const int j = pick_tap(wy, __fmul_rn((float)(r.y >> 8), 5.9604644775390625e-08f), gy);
            const float3 v = fetch_decode(p, ox + i, oy + j, &tabs);
            if (ps.active) {
                res = FILT == 2 ? make_float4(__fmul_rn(__fmul_rn(v.x, gx), gy), __fmul_rn(__fmul_rn(v.y, gx), gy),
                                              __fmul_rn(__fmul_rn(v.z, gx), gy), __fmul_rn(__fmul_rn(1.0f, gx), gy))
                                : make_float4(v.x, v.y, v.z, 1.0f);
                count = 1;
            }
            if (inside) store_pixel(p, idx, res, (uint8_t)count);
            continue;
        }

        // ---- success: texel i by lane h(i, A) (or lane i); the counts follow that
        if (kStats) {
            cnt.v[kStatTilesSuccess] += 1;
            cnt.v[kStatTexelEvals] += n;
            cnt.v[kStatTexelEvalsUnique] += n;
        }
        const bool full = A == FULL;
        const int my_i = (full || !p.edge_remap) ? lane : (((A >> lane) & 1u) ? __popc(A & lt) : 32);
        count = my_i < n ? 1u : 0u;
        const int t00 = (oy - miny) * bw + (ox - minx);
        int qx = ps.ulx, qy = ps.uly;  // the texel this lane decodes
        int row[4];                    // lane holding tap 4 r; the next three lanes hold the next three taps
        if (ALG == ALG_BOX || mcls == 1) {
            // a box of at most 32 texels: lane L decodes box position L
            const bool in_set = ALG == ALG_BOX ? lane < n : ((word >> lane) & 1u) != 0;
            if (in_set) {
                const int q = div_small(lane, bw);
                qx = minx + (lane - q * bw);
                qy = miny + q;
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) row[r] = t00 + r * bw;
        } else if (ALG == ALG_MASK || mcls == 3) {
            // lane i decodes the texel of rank i (every lane of the warp does
            // the arithmetic, whichever pixels are active); the four taps of a
            // row are neighbours in the mask, so their ranks follow one another
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int t = t00 + r * bw;
                const uint32_t wd = __shfl_sync(FULL, word, t >> 5);
                row[r] = __shfl_sync(FULL, before, t >> 5) + __popc(wd & ((1u << (t & 31)) - 1u));
            }
            // bit `lane` of each word files its position at its rank
            const int words = (bw * bh + 31) >> 5;
            for (int w = 0; w < words; ++w) {
                const uint32_t wd = __shfl_sync(FULL, word, w);
                const int b = __shfl_sync(FULL, before, w) + __popc(wd & lt);
                if ((wd >> lane) & 1u) ranks[ck(b, 32, p.err, kBndRanks)] = 32 * w + lane;
            }
            __syncwarp();
            if (lane < n) {
                const int t = ranks[lane];
                const int q = div_small(t, bw);
                qx = minx + (t - q * bw);
                qy = miny + q;
            }
            __syncwarp();
        } else if (lane < n) {  // the list's order
            qx = lu.tx;
            qy = lu.ty;
        }
        if (ALG == ALG_LIST && mcls != 4) {
#pragma unroll
            for (int r = 0; r < 4; ++r) lsrc[r] = (uint32_t)row[r] * 0x01010101u + 0x03020100u;
        }
        // ---- decode, gather the 16 taps, filter in tap order.  Alpha is 1, and
        // fma(w, 1, a) is a + w; red and green run as a pair
        const float3 val = fetch_decode(p, qx, qy, &tabs);
        float2 rg = make_float2(0.f, 0.f);
        float ab = 0.f, aw = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int sl = ALG == ALG_LIST ? (int)(lsrc[k >> 2] >> (8 * (k & 3))) : row[k >> 2] + (k & 3);
            const float2 w = __fmul2_rn(make_float2(wx[k & 3], wx[k & 3]), make_float2(wy[k >> 2], wy[k >> 2]));
            const float vx = __shfl_sync(FULL, val.x, sl);
            const float vy = __shfl_sync(FULL, val.y, sl);
            const float vz = __shfl_sync(FULL, val.z, sl);
            rg = __ffma2_rn(w, make_float2(vx, vy), rg);
            ab = __fmaf_rn(w.x, vz, ab);
            aw = __fadd_rn(aw, w.x);
        }
        const float4 acc = make_float4(rg.x, rg.y, ab, aw);
        if (ps.active) res = acc;
        else count = 0;
        if (inside) store_pixel(p, idx, res, (uint8_t)count);
    }

    if (kStats) {
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < kNumStats; ++i)
                if (cnt.v[i]) atomicAdd(&block_stats[i], (unsigned long long)cnt.v[i]);
        }
        __syncthreads();
        if (threadIdx.x < kNumStats && block_stats[threadIdx.x]) atomicAdd(p.stats + threadIdx.x, block_stats[threadIdx.x]);
    }
}

using KernelFn = void (*)(const ExactParams);

template <int ALG, int TW, int FILT, bool kStats>
KernelFn pick_mask(int md) {
    if constexpr (ALG == ALG_MASK) {
        return md == 11 ? bicubic_filter_kernel<ALG, TW, 11, FILT, kStats>
                        : bicubic_filter_kernel<ALG, TW, 16, FILT, kStats>;
    } else {
        return bicubic_filter_kernel<ALG, TW, 16, FILT, kStats>;
    }
}

template <int TW, int FILT, bool kStats>
KernelFn pick_alg(int alg, int md) {
    switch (alg) {
    case ALG_4TAP: return pick_mask<ALG_4TAP, TW, FILT, kStats>(md);
    case ALG_STF: return pick_mask<ALG_STF, TW, FILT, kStats>(md);
    case ALG_LIST: return pick_mask<ALG_LIST, TW, FILT, kStats>(md);
    case ALG_BOX: return pick_mask<ALG_BOX, TW, FILT, kStats>(md);
    case ALG_MASK: return pick_mask<ALG_MASK, TW, FILT, kStats>(md);
    default: return nullptr;
    }
}

template <int FILT, bool kStats>
KernelFn pick_tile(int alg, int tile_w, int md) {
    switch (tile_w) {
    case 8: return pick_alg<8, FILT, kStats>(alg, md);
    case 4: return pick_alg<4, FILT, kStats>(alg, md);
    case 16: return pick_alg<16, FILT, kStats>(alg, md);
    default: return nullptr;
    }
}

}  // namespace

cudaError_t launch_bicubic_filter(const ExactParams &p, int alg, int tile_w, int mask_dim, int filter,
                                  cudaStream_t stream) {
    const bool st = p.stats != nullptr;
    KernelFn fn = nullptr;
    if (filter == 1) fn = st ? pick_tile<1, true>(alg, tile_w, mask_dim) : pick_tile<1, false>(alg, tile_w, mask_dim);
    else if (filter == 2) fn = st ? pick_tile<2, true>(alg, tile_w, mask_dim) : pick_tile<2, false>(alg, tile_w, mask_dim);
    if (!fn) return cudaErrorInvalidValue;
    if (p.n_tiles == 0) return cudaSuccess;
    if (p.n_tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    const long long want = (p.n_tiles + kWarps - 1) / kWarps;
    const long long cap = (long long)device_sm_count() * resident_ctas(reinterpret_cast<const void *>(fn), kThreads);
    const int grid = (int)(want < cap ? want : cap);
    return launch_dependent(fn, grid, kThreads, 0, stream, p);
}

}  // namespace ctf
