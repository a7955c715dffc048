// ctf_mlp_ws2.cu -- learned-decode filter for STF, Box and Mask Sampling on
// single views and batches: warps specialised by role.
//
// A CTA of 256 threads (four per SM) takes the groups of 8 pixel tiles g0,
// g0 + G, ... (G = gridDim.x) in turn:
//   - warpgroup 1 (warps 4-7, the producers, two tiles of the group each)
//     runs step 1 of the collaborative flow (Sec. 3) on its tiles and lists
//     their texels in consecutive rows (a shared-memory counter gives each
//     tile its rows);
//   - warpgroup 0 (warps 0-3, the consumer) writes the features of the rows
//     straight into the group's layer-1 operand buffer in the tensor cores'
//     layout, owns the 128 TMEM lanes and runs the tcgen05 MLP chain(s) over
//     the group's rows: three MMA layers, the
//     two hidden epilogues (bias, ReLU, conversion to the next operand) and
//     the output epilogue into the row values; then it gathers, filters and
//     stores the group's pixels from the row values (warp w the tiles w and
//     4 + w).
// One elected consumer thread issues the MMAs; every consumer thread polls
// their barrier.  Warps whose 32 rows all lie past the group's last row skip
// their epilogues.  The hidden activations stay in tensor memory: each
// epilogue writes them next to the accumulator, and the next layer's MMAs
// read their A operand from there.
// Three stages of group buffers (operand rows, half of which the row values
// overwrite once the rows have been consumed, per-pixel words, first rows)
// rotate over consecutive groups, so the producers may run two groups ahead
// of the consumer.  The producers hand a stage over with a full barrier (four
// arrivals) and get it back with a done barrier (one arrival, after the
// gather); a row's texel waits in the row's own place in the operand buffer,
// so the producer warps do not wait for one another.  Every wait is bounded; a
// wait that gives up records CTF_ERR_TIMEOUT and both roles leave.
// The roles share the work so that neither waits long: with the features on
// the producers the consumer stood still for half of the time (4,500 of 8,600
// clocks a group) and a 3840x2160 Mask-11 FP16 view took 198 us, now 193, with
// the consumer the longer role: of 6,500 clocks a group it waits 460, and
// spends 2,100 on features, 2,950 in its 1.23 chains and 950 on the gather; a
// producer warp waits 2,900 and takes 3,450 for step 1 of its two tiles.  In
// the batch kernel, whose parameters are read from shared memory, the features
// stay on the producers (256 views 473 us, on the consumer 493).
// What bounds it: instruction issue (573 warp instructions a tile at 66% of the
// issue slots with 32 warps on an SM) and the latency of the consumer's chain,
// not the tensor pipe and not memory.  So the rows are given out by a counter rather than found by a
// scan, a lane's place in a tile and the tile walk are computed once, FP8 is a
// template parameter, and both roles run in the 64 registers of the launch
// (no register split).  3840x2160 Mask-11 FP16: 276 us with the scan, 72/56
// registers and both operand types in one kernel, 250 us so; 8 producer warps
// at three CTAs per SM 262 us, 6 at four 272 us, 12 at two 304 us, and without
// the producers' two barriers a group (lists handed over by mbarriers) 279 us.
// Each pixel gets the same texels, texel values, image and counts as the
// other learned kernels: the rows of an MMA are independent, so where a
// texel's row sits does not change its value, and an MMA's result does not
// depend on whether its A operand comes from shared or tensor memory.
// Compiled by itself for warp tiles 8 pixels wide; the units that include it
// (the other widths, ctf_mlp_dense.cu) define CTF_MLP_WS2_PART.
#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include "ctf_device.cuh"
#include "ctf_internal.h"
#include "ctf_mlp.cuh"
#include "ctf_select.cuh"
#include "tc_ops.cuh"
#include "ctf_mlp_chain.cuh"
#include "ctf_exact_tile.cuh"
#include "ctf_mlp_pf.h"

namespace ctf {
namespace {

constexpr int kPProducerWarps = 4;
constexpr int kPProducerThreads = 32 * kPProducerWarps;
constexpr int kPThreads = kRows + kPProducerThreads;
constexpr int kPCtasPerSm = 4;
constexpr int kPSlots = 2;                             // pixel tiles of a group per producer warp
constexpr int kPTiles = kPSlots * kPProducerWarps;     // tiles of a group
constexpr int kPGroupRows = 32 * kPTiles;              // pixels of a group, and rows of it at most
constexpr int kPLaunchRegs = (65536 / (kPThreads * kPCtasPerSm)) & ~7;

// Shared memory (bytes).  The operand image sits at 0 with the offsets of
// ctf_mlp.cuh; then the MMA barrier and TMEM slot, the stage hand-over
// barriers, the producers' Mask rank slots and texel lists, in the variant
// with fallbacks C / C+ one texel table per warp, and the stages.
// Tensor memory (128 columns): every layer's accumulator D at columns
// [0, 64), the hidden activations at [64, 96).
constexpr int kPMaxStages = 3;
constexpr int kPBar = kImgBytes;                 // MMA barrier (8 B), TMEM base (4 B)
constexpr int kPTmem = kPBar + 8;
constexpr int kPHand = kPBar + 16;               // full[kPMaxStages], done[kPMaxStages]
// producer warps x 64 rank slots (two texels per lane may rank 64 texels a tile)
constexpr int kPRanks = kPHand + 16 * kPMaxStages;
constexpr int kPRanksEnd = kPRanks + kPProducerWarps * 64 * 4;  // fallback variant: the warps' texel tables; then the stages

// One stage of a group of at most T tiles (offsets in bytes).
template <int T>
struct PStage {
    static constexpr int kPix = 32 * T;              // pixels, and rows at most
    // layer-1 operand, 32 B a row; before it a row's texel (p_texel), after it the row values (16 B each)
    static constexpr int kX = 0;
    static constexpr int kWord = kX + kPix * 32;     // float4 per pixel: s, t, the packed word, unused
    static constexpr int kBase = kWord + kPix * 16;  // int2 per tile: first row, first pixel
    static constexpr int kAlloc = kBase + T * 8;     // int: rows given out so far
    static constexpr int kEnd = kAlloc + 16;
    static constexpr int kQ = kEnd;                  // fallback variant: int2 texel a pixel's lane produces
    static constexpr int kUL = kQ + kPix * 8;        // fallback variant: int2 upper-left texel of the footprint
    static constexpr int kFbEnd = kUL + kPix * 8;
};

// kFb: the variant with fallbacks C / C+ (two stages, to make room for the
// texel tables and the per-pixel texels the blend of eq. 1 needs).
// kBatch: the persistent batch kernel, whose stages also carry the group's
// view (copies of its parameters and network) and whose producer warps keep
// two copies of their own.
constexpr int kPViewBytes = (int)sizeof(ExactParams) + (((int)sizeof(MlpDevice) + 15) & ~15);
template <bool kFb, bool kBatch = false>
struct PLayout {
    static_assert(!(kFb && kBatch), "batches take no fallbacks on learned views");
    using S = PStage<kPTiles>;
    static constexpr int kStages = kFb ? 2 : 3;
    static constexpr int kStage0 = kPRanksEnd + (kFb ? (4 + kPProducerWarps) * (int)sizeof(FbTable) : kBatch ? 2 * kPProducerWarps * kPViewBytes : 0);
    static constexpr int kStageBytes = kFb ? S::kFbEnd : S::kEnd + (kBatch ? kPViewBytes : 0);
    static constexpr int kBytes = kStage0 + kStages * kStageBytes;
    static_assert(kStage0 % 16 == 0 && kStageBytes % 16 == 0 && kPRanksEnd % 16 == 0, "16-byte operand buffers");
    // kPCtasPerSm CTAs per SM fit, and no more than four (4 x 128 TMEM columns)
    static_assert(kPCtasPerSm * (kBytes + 1024 + 128) <= 228 * 1024, "the CTAs of an SM fit in shared memory");
};
static_assert(65536 / (kPThreads * kPLaunchRegs) <= 4, "at most four CTAs share an SM's TMEM");

template <bool kFb, bool kBatch = false>
__device__ __forceinline__ unsigned char *p_stage(unsigned char *sm, int s) {
    return sm + PLayout<kFb, kBatch>::kStage0 + s * PLayout<kFb, kBatch>::kStageBytes;
}
__device__ __forceinline__ uint64_t *p_full(unsigned char *sm, int s) {
    return reinterpret_cast<uint64_t *>(sm + kPHand) + s;
}
__device__ __forceinline__ uint64_t *p_done(unsigned char *sm, int s) {
    return reinterpret_cast<uint64_t *>(sm + kPHand) + kPMaxStages + s;
}

__device__ __forceinline__ void p_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(bar)) : "memory");
}

// Named barriers: 1 among the 128 consumer threads, 2 among the producer
// threads (0 stays __syncthreads).
__device__ __forceinline__ void cons_bar() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// Barrier `id` among n threads, returning whether any of them passed true.
template <int id, int n>
__device__ __forceinline__ bool bar_or(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.or.pred p, %2, %3, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(id), "n"(n)
        : "memory");
    return r != 0;
}

// Hidden epilogue of a warp's 32 rows: TMEM columns [taddr, taddr + 64) of
// this thread's row -> bias, ReLU -> the next layer's A operand, written to
// TMEM columns from hcol on (FP16 pairs, or E4M3 quadruples, per 32-bit
// column in K order).  `bias` and `oscale` point into the kernel's parameters
// (every address is a compile-time offset there, so the packed adds take
// them as constant-bank operands) or, in a batch whose group has another
// network, into the operand image in shared memory.  From shared memory the
// epilogue takes about 490 clocks with four CTAs on the SM, from the
// parameters 270.
template <bool kFp8>
__device__ __forceinline__ void p_hidden_epilogue(uint32_t hcol, uint32_t taddr, const float *bias,
                                                  const float *oscale) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float d[16];
        tc::tmem_ld16(taddr + 16 * q, d);
        tc::tmem_wait_ld();
        tc::regs_after_wait<16>(d);
        if (!kFp8) {
            uint32_t w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int k = 2 * i, c = 16 * q + k;
                const float2 t = __fadd2_rn(make_float2(d[k], d[k + 1]), make_float2(bias[c], bias[c + 1]));
                w[i] = relu_half2(t.x, t.y);
            }
            tc::tmem_st8(hcol + 8 * q, w);
        } else {
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = 4 * i, c = 16 * q + k;
                const float2 t0 = __ffma2_rn(make_float2(d[k], d[k + 1]), make_float2(oscale[c], oscale[c + 1]),
                                             make_float2(bias[c], bias[c + 1]));
                const float2 t1 = __ffma2_rn(make_float2(d[k + 2], d[k + 3]), make_float2(oscale[c + 2], oscale[c + 3]),
                                             make_float2(bias[c + 2], bias[c + 3]));
                w[i] = (uint32_t)relu_e4m3x2(t0.x, t0.y) | ((uint32_t)relu_e4m3x2(t1.x, t1.y) << 16);
            }
            tc::tmem_st4(hcol + 4 * q, w);
        }
    }
    tc::tmem_wait_st();
}

// The end of one MMA layer, for one thread: every consumer thread polls the
// MMA barrier itself.  (One polling thread and a named barrier for the others
// took about 240 clocks longer per layer: 2700 instead of 2130 clocks for a
// chain with four CTAs on the SM.)  Returns false if the MMAs did not
// complete within the bound; the caller goes on and the threads agree on it
// at their next barrier.
__device__ __forceinline__ bool p_layer_wait(uint64_t *bar, uint32_t &phase) {
    const bool ok = tc::mbar_wait(bar, phase, kMaxTries);
    phase ^= 1u;
    __syncwarp();  // the TMEM accesses that follow are .aligned
    tc::fence_after_sync();
    return ok;
}

// The three layers for the 128 rows of chain c of a stage (layer-1 operand
// at sX).  TMEM columns: D (every layer's accumulator) at [0, 64), the
// hidden activations H at [64, 96).  `live`: this warp has rows below the
// group's row count (else it skips its epilogues).  kParam: the network's
// biases and scales are in ep (a kernel parameter), else in the operand
// image.  Consumer threads only.  Returns false (for every consumer thread
// alike) if layer 1 or 2 did not complete within the wait bound; `bad` is
// set in the threads that gave up on layer 3, which the caller's next
// barrier has to collect.
template <bool kParam, bool kFp8>
__device__ __forceinline__ bool p_chain(unsigned char *sm, uint32_t tmem, uint64_t *bar, uint32_t &phase,
                                        uint32_t sX, int warp, bool live, const MlpEpilogue &ep, float4 &out,
                                        bool &bad, int *err) {
    const int tid = threadIdx.x;
    const float *b1 = reinterpret_cast<const float *>(sm + kImgB1);
    const float *b2 = reinterpret_cast<const float *>(sm + kImgB2);
    const float *b3 = reinterpret_cast<const float *>(sm + kImgB3);
    const float *s1 = reinterpret_cast<const float *>(sm + kImgS1);
    const float *s2 = reinterpret_cast<const float *>(sm + kImgS2);
    const float *s3 = reinterpret_cast<const float *>(sm + kImgS3);
    const uint32_t lane_base = tmem + ((uint32_t)(32 * warp) << 16);
    const uint32_t sW1 = tc::smem_addr(sm + kImgW1), sW2 = tc::smem_addr(sm + kImgW2),
                   sW3 = tc::smem_addr(sm + kImgW3);
    const uint32_t kstep = 256;              // 32 bytes of K per 8-row group
    const uint32_t sboX = 256u;              // K = 32 bytes per row, FP16 and E4M3 alike
    constexpr uint32_t sboH = kFp8 ? 512u : 1024u;  // 64 elements per row
    constexpr int nk = kFp8 ? 2 : 4;         // MMAs over K = 64
    constexpr uint32_t id64 = kFp8 ? tc::idesc_e4m3(128, 64) : tc::idesc_f16(128, 64);
    constexpr uint32_t id16 = kFp8 ? tc::idesc_e4m3(128, 16) : tc::idesc_f16(128, 16);
    const uint32_t tH = tmem + 64;

    // ---- layer 1: D = X W1^T
    if (warp == 0 && tc::elect_one()) {
        tc::fence_after_sync();
        const uint64_t a = tc::smem_desc(sX, 128, sboX), b = tc::smem_desc(sW1, 128, sboX);
        if (kFp8) tc::mma_e4m3(tmem, a, b, id64, false);
        else tc::mma_f16(tmem, a, b, id64, false);
        tc::commit(bar);
    }
    bad |= !p_layer_wait(bar, phase);
    if (live) {
        if (kParam) p_hidden_epilogue<kFp8>(lane_base + 64, lane_base + 0, ep.b1, ep.s1);
        else p_hidden_epilogue<kFp8>(lane_base + 64, lane_base + 0, b1, s1);
    }
    tc::fence_before_sync();
    if (bar_or<1, kRows>(bad)) {
        if (tid == 0) atomicExch(err, CTF_ERR_TIMEOUT);
        return false;
    }
    // ---- layer 2: D = H1 W2^T (D1 has been read)
    if (warp == 0 && tc::elect_one()) {
        tc::fence_after_sync();
#pragma unroll
        for (int j = 0; j < nk; ++j) {
            const uint64_t b = tc::smem_desc(sW2 + j * kstep, 128, sboH);
            if (kFp8) tc::mma_e4m3_ts(tmem, tH + 8 * j, b, id64, j > 0);
            else tc::mma_f16_ts(tmem, tH + 8 * j, b, id64, j > 0);
        }
        tc::commit(bar);
    }
    bad |= !p_layer_wait(bar, phase);
    // the layer-2 MMAs have read H1, so H2 may overwrite it
    if (live) {
        if (kParam) p_hidden_epilogue<kFp8>(lane_base + 64, lane_base + 0, ep.b2, ep.s2);
        else p_hidden_epilogue<kFp8>(lane_base + 64, lane_base + 0, b2, s2);
    }
    tc::fence_before_sync();
    if (bar_or<1, kRows>(bad)) {
        if (tid == 0) atomicExch(err, CTF_ERR_TIMEOUT);
        return false;
    }
    // ---- layer 3: D[0..16) = H2 W3^T
    if (warp == 0 && tc::elect_one()) {
        tc::fence_after_sync();
#pragma unroll
        for (int j = 0; j < nk; ++j) {
            const uint64_t b = tc::smem_desc(sW3 + j * kstep, 128, sboH);
            if (kFp8) tc::mma_e4m3_ts(tmem, tH + 8 * j, b, id16, j > 0);
            else tc::mma_f16_ts(tmem, tH + 8 * j, b, id16, j > 0);
        }
        tc::commit(bar);
    }
    bad |= !p_layer_wait(bar, phase);
    if (live) {
        uint32_t r[4];
        tc::tmem_ld4(lane_base + 0, r);
        tc::tmem_wait_ld();
        tc::regs_after_wait<4>(r);
        float o[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float d = __uint_as_float(r[c]);
            const float s = kParam ? ep.s3[c] : s3[c], b = kParam ? ep.b3[c] : b3[c];
            const float v = kFp8 ? __fmaf_rn(d, s, b) : __fadd_rn(d, b);
            o[c] = fminf(fmaxf(v, 0.f), 1.f);
        }
        out = make_float4(o[0], o[1], o[2], o[3]);
    }
    tc::fence_before_sync();
    return true;
}

// The texel of row `row` of a stage waits in the first 16 bytes of the row's
// place in the layer-1 operand: the thread that reads it is the one that
// writes the row's features over it.
template <typename S>
__device__ __forceinline__ int2 *p_texel(unsigned char *st, int row) {
    return reinterpret_cast<int2 *>(st + S::kX + (row >> 3) * 256 + (row & 7) * 16);
}

// n rows of the group for tile slot g whose first pixel is `pixel`; the stage
// keeps both for the gather.  (The rows of the tiles follow one another in
// the order in which the warps come; a row's place does not change its
// value.)
template <typename S>
__device__ __forceinline__ int p_take_rows(unsigned char *st, int g, int n, uint32_t pixel, int lane) {
    int base = 0;
    if (lane == 0) {
        base = atomicAdd(reinterpret_cast<int *>(st + S::kAlloc), n);
        reinterpret_cast<int2 *>(st + S::kBase)[g] = make_int2(base, (int)pixel);
    }
    return __shfl_sync(FULL, base, 0);
}

// The place of a lane in the tiles of a view: its pixel's offset from the
// tile's first pixel, and the bounds below which the tile's column and row
// keep it inside the frame.
template <int TW>
struct LanePlace {
    uint32_t tx, ty, off, lim_x, lim_y;
    __device__ __forceinline__ LanePlace(const ExactParams &p, int lane) {
        constexpr uint32_t TH = 32 / TW;
        tx = (uint32_t)lane % TW;
        ty = (uint32_t)lane / TW;
        off = ty * (uint32_t)p.W + tx;
        lim_x = ((uint32_t)p.W - tx + TW - 1) / TW;
        lim_y = ((uint32_t)p.H - ty + TH - 1) / TH;
    }
};

// The tap indices of a tile whose texels are set bits of a box (Box and Mask
// Sampling) come in pairs: tap k + 1 is the next list entry after tap k = 0, 2.
template <int ALG>
constexpr bool p_tap_pairs() { return ALG == ALG_BOX || ALG == ALG_MASK; }

// The inputs of the lane's pixel of the tile at (bx, by).  Every lane loads
// (lanes outside the frame pixel 0, which exists), so that the loads carry no
// predicates.
template <int ALG, int TW>
__device__ __forceinline__ Inputs p_load(const ExactParams &p, const LanePlace<TW> &lp, uint32_t bx, uint32_t by) {
    constexpr uint32_t TH = 32 / TW;
    return load_inputs_any<(ALG >= ALG_LIST)>(p, bx < lp.lim_x && by < lp.lim_y,
                                              by * (TH * (uint32_t)p.W) + bx * TW + lp.off);
}

// Producer: step 1 on the tile at (bx, by), slot g of the group, into stage
// st: per pixel (s, t) and a packed word (bits 0-19 the list indices of its 4
// taps on success, else of its own texel; 20-22 its count; 23 active; 24
// inside; 25 success), and the tile's texels (clamped) at the rows it takes.
// A tile past the last row of tiles has no pixel inside.
// kStats: the variant that keeps the outcome counters (p.stats set).
// kFb: the variant with fallbacks C / C+: an over-budget magnified tile
// takes its texels from fb_choose (the exact path's choice, with the warp's
// table fbt); each lane's produced texel gets the rank of the lane among
// the producing lanes, and the pixel's word carries bit 26 (fallback tile)
// and bit 27 (this lane produces); the produced texel and the footprint's
// upper-left texel go to the stage for the blend of eq. 1.
// kTwo: the variant with two texels per lane (groups of 4 tiles of up to 64
// texels): the pixel's word holds the 6-bit list indices of its taps (bits
// 0-23, or of its own texel), its count (24-25), active (26), inside (27)
// and success (28).
template <int ALG, int TW, int MD, bool kStats, bool kFb, bool kTwo = false>
__device__ __forceinline__ void p_step1(const ExactParams &p, const LanePlace<TW> &lp, uint32_t bx, uint32_t by,
                                        const Inputs &in, int g, unsigned char *st, int lane, uint32_t lt, int *ranks,
                                        Counters &cnt, FbTable *fbt) {
    using S = typename PLayout<kFb>::S;
    constexpr uint32_t TH = 32 / TW;
    const bool inside = bx < lp.lim_x && by < lp.lim_y;
    const int px = (int)(bx * TW + lp.tx), py = (int)(by * TH + lp.ty);
    const uint32_t pixel = by * (TH * (uint32_t)p.W) + bx * TW;
    PixelSetup ps;
    ps.active = inside && in.cov != 0;
    setup_coords(in.uv, (float)p.Wt, (float)p.Ht, ps);
    Selection sel;
    if (!kStats || by * TH < (uint32_t)p.H) {
        sel = select_tile<ALG, MD, kStats, false, kTwo>(p, ps, in.jac, px, py, lane, lt, ranks, cnt);
    } else {  // no tile: nothing to count
        sel.path = PATH_EMPTY;
        sel.A = 0;
        sel.produce = sel.produce2 = false;
        sel.count = 0;
        sel.my_rank = sel.my_rank2 = 0;
    }
    float4 *word = reinterpret_cast<float4 *>(st + S::kWord) + 32 * g + lane;
    auto put = [&](int row, int x, int y) {
        *p_texel<S>(st, ck(row, kPGroupRows, p.err, kBndTexList)) =
            make_int2(min(max(x, 0), p.Wt - 1), min(max(y, 0), p.Ht - 1));
    };
    if (kFb && p.fallback != 0 && sel.path == PATH_FALLBACK_BUDGET) {  // warp-uniform
        const FbChoice c = fb_choose(p.fallback, p.view, p.y0, p.k0, p.k1, ps.ulx, ps.uly, ps.s, ps.t, ps.active, px,
                                     py, sel.A, lane, lt, fbt);
        const uint32_t pm = __ballot_sync(FULL, c.produce);
        const int rank = __popc(pm & lt), n = __popc(pm);
        const int base = p_take_rows<S>(st, g, n, pixel, lane);
        if (c.produce) put(base + rank, c.qx, c.qy);
        // select_tile counted one evaluation per active lane
        if (kStats) cnt.v[kStatTexelEvals] += n - __popc(sel.A);
        const uint32_t info = (uint32_t)rank | ((c.produce ? 1u : 0u) << 20) | (ps.active ? 1u << 23 : 0u) |
                              (inside ? 1u << 24 : 0u) | (1u << 26) | (c.produce ? 1u << 27 : 0u);
        *word = make_float4(ps.s, ps.t, __uint_as_float(info), 0.f);
        reinterpret_cast<int2 *>(st + S::kQ)[32 * g + lane] = make_int2(c.qx, c.qy);
        reinterpret_cast<int2 *>(st + S::kUL)[32 * g + lane] = make_int2(ps.ulx, ps.uly);
        return;
    }
    const bool succ = sel.path == PATH_SUCCESS;
    const int base = p_take_rows<S>(st, g, succ ? sel.n : __popc(sel.A), pixel, lane);
    if (sel.produce) put(base + sel.my_rank, sel.tx, sel.ty);
    if (kTwo && sel.produce2) put(base + sel.my_rank2, sel.tx2, sel.ty2);
    constexpr int kIdxBits = kTwo ? 6 : 5, kCnt = kTwo ? 24 : 20, kAct = kTwo ? 26 : 23, kIns = kTwo ? 27 : 24,
                  kSucc = kTwo ? 28 : 25;
    constexpr uint32_t kIdxMask = (1u << kIdxBits) - 1u;
    uint32_t info = 0;
#pragma unroll
    for (int k = 0; k < 4; k += p_tap_pairs<ALG>() ? 2 : 1) info |= ((uint32_t)sel.rk[k] & kIdxMask) << (kIdxBits * k);
    info = succ ? info : ((uint32_t)sel.my_rank & kIdxMask);
    info |= ((uint32_t)sel.count << kCnt) | (ps.active ? 1u << kAct : 0u) | (inside ? 1u << kIns : 0u) |
            (succ ? 1u << kSucc : 0u);
    *word = make_float4(ps.s, ps.t, __uint_as_float(info), 0.f);
}

// Consumer: step 3 for tile slot g of the group from stage st (its row values
// in place): gather, filter, store; `off` is the lane's pixel in the tile.
template <int ALG, bool kFb, bool kTwo = false>
__device__ __forceinline__ void p_gather(const ExactParams &p, uint32_t off, int g, const unsigned char *st, int lane,
                                         FbTable *fbt) {
    using S = typename PLayout<kFb>::S;
    const float4 word = reinterpret_cast<const float4 *>(st + S::kWord)[32 * g + lane];
    const int2 tile = reinterpret_cast<const int2 *>(st + S::kBase)[g];
    const uint32_t info = __float_as_uint(word.z);
    const float4 *outrow = reinterpret_cast<const float4 *>(st + S::kX);
    // row of list entry i of this tile (the row values fill half of the operand rows' space)
    auto row_of = [&](uint32_t i) { return ck(tile.x + (int)i, kPGroupRows, p.err, kBndRow); };
    // the word's fields (kTwo: 6-bit list indices)
    constexpr int kIdxBits = kTwo ? 6 : 5, kCnt = kTwo ? 24 : 20, kAct = kTwo ? 26 : 23, kIns = kTwo ? 27 : 24,
                  kSucc = kTwo ? 28 : 25;
    constexpr uint32_t kIdxMask = (1u << kIdxBits) - 1u, kCntMask = kTwo ? 3u : 7u;
    const bool inside = ((info >> kIns) & 1u) != 0;  // (pixels outside the frame take part in the blend only)
    const uint32_t idx = ck(inside ? (uint32_t)tile.y + off : 0u, view_pixels(p), p.err, kBndPixel);
    if (kFb && ((info >> 26) & 1u)) {
        // fallback C / C+ (the whole warp: the blend is warp-collective):
        // eq. 1 over the produced texels of the footprint, their values the
        // rows of the tile's list
        FbChoice c;
        c.produce = ((info >> 27) & 1u) != 0;
        const int2 q = reinterpret_cast<const int2 *>(st + S::kQ)[32 * g + lane];
        const int2 ul = reinterpret_cast<const int2 *>(st + S::kUL)[32 * g + lane];
        c.qx = q.x;
        c.qy = q.y;
        const float4 val = c.produce ? outrow[row_of(info & 31u)] : make_float4(0.f, 0.f, 0.f, 0.f);
        const FallbackOut fo = fb_blend<false>(val, c, ul.x, ul.y, word.x, word.y, ((info >> 23) & 1u) != 0, lane, fbt);
        if (inside) {
            __stcs(p.out + idx, fo.res);
            if (p.evals) p.evals[idx] = (uint8_t)fo.count;
        }
        return;
    }
    if (!inside) return;  // outside the frame (or no tile)
    float4 result = make_float4(0.f, 0.f, 0.f, 0.f);
    uint8_t cv = 0;
    if ((info >> kAct) & 1u) {
        if ((info >> kSucc) & 1u) {
            float w[4];
            bilinear_weights(word.x, word.y, w);
            float2 rg = make_float2(0.f, 0.f), ba = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // (paired taps: the odd one is the next row)
                const bool next = p_tap_pairs<ALG>() && (k & 1);
                const float4 t = outrow[ck(row_of((info >> (kIdxBits * (next ? k - 1 : k))) & kIdxMask) + (next ? 1 : 0),
                                           kPGroupRows, p.err, kBndRow)];
                const float2 wk = make_float2(w[k], w[k]);
                rg = __ffma2_rn(wk, make_float2(t.x, t.y), rg);
                ba = __ffma2_rn(wk, make_float2(t.z, t.w), ba);
            }
            result = make_float4(rg.x, rg.y, ba.x, ba.y);
            cv = (uint8_t)((info >> kCnt) & kCntMask);
        } else {
            result = outrow[row_of(info & kIdxMask)];
            cv = 1;
        }
    }
    __stcs(p.out + idx, result);
    if (p.evals) p.evals[idx] = cv;
}

// The features of rows tid, tid + 128 of the R rows of stage st in the tensor
// cores' operand layout, for thread tid of a role; published to the MMAs.
static_assert(kPProducerThreads == kRows, "either role has a thread per row of a chain");
template <typename S, bool kFp8>
__device__ __forceinline__ void p_features(const MlpDevice &m, unsigned char *st, int R, int tid, const float *inv_a1) {
#pragma unroll 1
    for (int row = tid; row < R; row += kRows) {
        const int2 t = *p_texel<S>(st, row);
        float f[kMlpIn];
        texel_features(m, t.x, t.y, f);
        store_x_row_at(st + S::kX, row, f, kFp8, inv_a1);
    }
    tc::fence_proxy_async();  // generic-proxy writes -> the MMAs' async proxy
}

// Column and row of the tile g places after (bx, by).
__device__ __forceinline__ void p_tile(uint32_t tiles_x, uint32_t &bx, uint32_t &by, uint32_t g) {
    bx += g;
    while (bx >= tiles_x) {
        bx -= tiles_x;
        ++by;
    }
}

template <int ALG, int TW, int MD, bool kStats, bool kFb, bool kTwo, bool kFp8>
__global__ void __launch_bounds__(kPThreads, kPCtasPerSm)
    mlp_filter_pf_kernel(const ExactParams p, const MlpDevice m, const __grid_constant__ MlpEpilogue ep, int *err) {
    static_assert(!(kFb && kTwo), "fallbacks with two texels per lane run on the extension kernel");
    using S = typename PLayout<kFb>::S;
    constexpr int kPStages = PLayout<kFb>::kStages;
    // tiles per group: two texels per lane may need 64 rows a tile
    constexpr int kSlots = kTwo ? kPSlots / 2 : kPSlots;
    constexpr int kGT = kSlots * kPProducerWarps;
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ unsigned long long block_stats[kNumStats];
    const int lane = threadIdx.x & 31;
    const int warp = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0);  // uniform, and known to be
    // fallback variant: warp w's texel table (empty between tiles)
    FbTable *fbt = kFb ? reinterpret_cast<FbTable *>(sm + kPRanksEnd) + warp : nullptr;
    if (kFb) fb_clear(fbt, lane);
    uint64_t *mma_bar = reinterpret_cast<uint64_t *>(sm + kPBar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + kPTmem);
    if (threadIdx.x < kNumStats) block_stats[threadIdx.x] = 0;
    {
        const uint4 *src = m.img;
        uint4 *dst = reinterpret_cast<uint4 *>(sm + kImgW1);
        for (int i = threadIdx.x; i < kImgBytes / 16; i += blockDim.x) dst[i] = __ldg(src + i);
        // every thread's part of the image, written through the generic
        // proxy, ordered before the MMAs that read it through the async proxy
        tc::fence_proxy_async();
    }
    if (threadIdx.x == 0) {
        tc::mbar_init(mma_bar, 1);
        for (int s = 0; s < kPStages; ++s) {
            tc::mbar_init(p_full(sm, s), kPProducerWarps);
            tc::mbar_init(p_done(sm, s), 1);
            *reinterpret_cast<int *>(p_stage<kFb>(sm, s) + S::kAlloc) = 0;
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
    // what comes before overlaps the end of the kernel before this one; the
    // next kernel starts when this one has its TMEM
    grid_wait();
    grid_trigger();
    const uint32_t tmem = *tslot;
    const float *inv_a1 = reinterpret_cast<const float *>(sm + kImgA1);
    Counters cnt;
#pragma unroll
    for (int i = 0; i < kNumStats; ++i) cnt.v[i] = 0;
    const long long n_groups = (p.n_tiles + kGT - 1) / kGT;
    const long long G = gridDim.x;

    if (warp < 4) {
        // ---------------- consumer ----------------
        const int tid = threadIdx.x;
        const uint32_t off = LanePlace<TW>(p, lane).off;
        uint32_t phase = 0;
        for (long long j = 0;; ++j) {
            const long long grp = blockIdx.x + j * G;
            if (grp >= n_groups) break;
            const int s = (int)(j % kPStages);
            const uint32_t par = (uint32_t)((j / kPStages) & 1);
            unsigned char *st = p_stage<kFb>(sm, s);
            bool ok = tc::mbar_wait(p_full(sm, s), par, kMaxTries);
            __syncwarp();
            // the features of rows tid and tid + 128 in the tensor cores' operand layout
            const int R = min(__shfl_sync(FULL, *reinterpret_cast<const int *>(st + S::kAlloc), 0), kPGroupRows);
            if (ok) p_features<S, kFp8>(m, st, R, tid, inv_a1);
            if (bar_or<1, kRows>(!ok)) {
                if (tid == 0) atomicExch(err, CTF_ERR_TIMEOUT);
                break;
            }
            if (kStats && tid == 0) cnt.v[kStatTexelEvalsUnique] += R;
            const int passes = (R + kRows - 1) / kRows;
            float4 *outrow = reinterpret_cast<float4 *>(st + S::kX);
            const uint32_t sX = tc::smem_addr(st + S::kX);
            for (int c = 0; c < passes && ok; ++c) {
                const bool live = kRows * c + 32 * warp < R;
                float4 v;
                bool bad = false;
                ok = p_chain<true, kFp8>(sm, tmem, mma_bar, phase, sX + 4096u * (uint32_t)c, warp, live, ep, v, bad, err);
                if (!ok) break;
                // chain c's outputs overwrite operand rows of chain 0, which its
                // layer-1 MMA has read; chain 1's operand rows (bytes 4096 on)
                // are untouched
                if (live) outrow[ck(kRows * c + tid, kPGroupRows, p.err, kBndRow)] = v;
                ok = !bar_or<1, kRows>(bad);
                if (!ok && tid == 0) atomicExch(err, CTF_ERR_TIMEOUT);
            }
            if (!ok) break;
            {
                // step 3 for the group: warp w the tiles w, 4 + w, ...
#pragma unroll 1
                for (int k = warp; k < kGT; k += 4) p_gather<ALG, kFb, kTwo>(p, off, k, st, lane, fbt);
            }
            __syncwarp();
            cons_bar();  // every consumer warp has read the stage
            if (tid == 0) {
                *reinterpret_cast<int *>(st + S::kAlloc) = 0;
                p_arrive(p_done(sm, s));
            }
        }
    } else {
        // ---------------- producers: kPSlots tile slots per warp ----------------
        const int pw = warp - 4;
        const uint32_t lt = lanemask_lt();
        int *ranks = reinterpret_cast<int *>(sm + kPRanks) + 64 * pw;
        const LanePlace<TW> lp(p, lane);
        // the warp's tiles, advanced by the grid's stride without dividing again
        const uint32_t tiles_x = (uint32_t)p.tiles_x;
        const uint32_t mine = (uint32_t)blockIdx.x * kGT + (uint32_t)(kSlots * pw);
        uint32_t gx = mine % tiles_x, gy = mine / tiles_x;  // the warp's first tile of the group
        const uint32_t step = (uint32_t)G * kGT, step_x = step % tiles_x, step_y = step / tiles_x;
        uint32_t bx = gx, by = gy;
        Inputs in = p_load<ALG, TW>(p, lp, bx, by);
        for (long long j = 0;; ++j) {
            const long long grp = blockIdx.x + j * G;
            const bool have = grp < n_groups;  // uniform over the CTA
            if (!have) break;
            {
                const int s = (int)(j % kPStages);
                unsigned char *st = p_stage<kFb>(sm, s);
                if (j >= kPStages) {  // the consumer has gathered group j - kPStages from this stage
                    const bool okd = tc::mbar_wait(p_done(sm, s), (uint32_t)(((j - kPStages) / kPStages) & 1), kMaxTries);
                    if (!__all_sync(FULL, okd)) {
                        if (lane == 0) atomicExch(err, CTF_ERR_TIMEOUT);
                        break;
                    }
                }
#pragma unroll 1
                for (int k = 0; k < kSlots; ++k) {
                    // the inputs of the warp's next tile come in while this one
                    // is in step 1 (or the warp waits for its next stage)
                    uint32_t nx = bx, ny = by;
                    if (k + 1 < kSlots) {
                        p_tile(tiles_x, nx, ny, 1u);
                    } else {  // first slot of the CTA's next group
                        gx += step_x;
                        gy += step_y;
                        if (gx >= tiles_x) {
                            gx -= tiles_x;
                            ++gy;
                        }
                        nx = gx;
                        ny = gy;
                    }
                    const Inputs next = p_load<ALG, TW>(p, lp, nx, ny);
                    p_step1<ALG, TW, MD, kStats, kFb, kTwo>(p, lp, bx, by, in, kSlots * pw + k, st, lane, lt,
                                                            ranks, cnt, fbt);
                    bx = nx;
                    by = ny;
                    in = next;
                }
                __syncwarp();
                if (lane == 0) p_arrive(p_full(sm, s));
            }
        }
    }

    if (kStats && p.stats && lane == 0) {
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
    if (p.stats && threadIdx.x < kNumStats && block_stats[threadIdx.x])
        atomicAdd(p.stats + threadIdx.x, block_stats[threadIdx.x]);
}

// A producer warp's place in the items of a batch: the view of its current
// item and that view's items [begin, end).
struct BatchPlace {
    int view;
    long long begin, end;
};

// The view of `item`: the last one whose first item is <= item (views without
// items share the next view's first item, so they are skipped).  Items only
// grow, so the search starts at the current view, 32 views at a time.
// Warp-collective.
__device__ __forceinline__ BatchPlace find_batch_view(const long long *begin, int nviews, long long item, int from,
                                                      int lane) {
    int k = from;  // begin[k] <= item
    while (true) {
        const int i = k + 1 + lane;
        const bool le = i < nviews && __ldg(begin + i) <= item;
        const int n = __popc(__ballot_sync(FULL, le));  // (begin is sorted: the first n)
        k += n;
        if (n < 32) break;
    }
    BatchPlace b;
    b.view = k;
    b.begin = __ldg(begin + k);
    b.end = __ldg(begin + k + 1);
    return b;
}

// The learned views of a batch: the packed-group kernel made persistent.  CTA
// c takes the groups (items of 8 tiles) c, c + G, ... of all views, so that
// every producer warp knows its next group and has its next tile's inputs in
// flight, as in the single-view kernel (groups from a global counter, a view
// lookup and a parameter copy between barriers took 579 us for 256 views, of
// which the learned half was 415).  Each producer warp keeps copies of the
// parameters and network of its current and its next group's view; the stage
// carries a copy for the consumer, which reloads the operand image when a
// group's network is not the one in shared memory (between chains, when no
// MMA is in flight).
template <int ALG, int TW, int MD, bool kStats>
__global__ void __launch_bounds__(kPThreads, kPCtasPerSm)
    mlp_batch_pf_kernel(const PfBatch b, const MlpDevice m0, const __grid_constant__ MlpEpilogue ep0) {
    using S = PLayout<false, true>::S;
    constexpr int kPBat = S::kEnd;  // the group's view, after the stage's other fields
    constexpr int kPStages = PLayout<false, true>::kStages;
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ unsigned long long block_stats[kNumStats];
    const int lane = threadIdx.x & 31;
    const int warp = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0);  // uniform, and known to be
    uint64_t *mma_bar = reinterpret_cast<uint64_t *>(sm + kPBar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + kPTmem);
    if (threadIdx.x < kNumStats) block_stats[threadIdx.x] = 0;
    {
        const uint4 *src = m0.img;
        uint4 *dst = reinterpret_cast<uint4 *>(sm + kImgW1);
        for (int i = threadIdx.x; i < kImgBytes / 16; i += blockDim.x) dst[i] = __ldg(src + i);
        // every thread's part of the image, written through the generic
        // proxy, ordered before the MMAs that read it through the async proxy
        tc::fence_proxy_async();
    }
    if (threadIdx.x == 0) {
        tc::mbar_init(mma_bar, 1);
        for (int s = 0; s < kPStages; ++s) {
            tc::mbar_init(p_full(sm, s), kPProducerWarps);
            tc::mbar_init(p_done(sm, s), 1);
            *reinterpret_cast<int *>(p_stage<false, true>(sm, s) + S::kAlloc) = 0;
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
    // what comes before overlaps the end of the kernel before this one; the
    // next kernel starts when this one has its TMEM
    grid_wait();
    grid_trigger();
    const uint32_t tmem = *tslot;
    Counters cnt;
#pragma unroll
    for (int i = 0; i < kNumStats; ++i) cnt.v[i] = 0;
    int *err = b.err;

    if (warp < 4) {
        // ---------------- consumer ----------------
        const int tid = threadIdx.x;
        uint32_t phase = 0;
        const uint4 *loaded = m0.img;
        for (long long j = 0; blockIdx.x + j * (long long)gridDim.x < b.total_items; ++j) {
            const int s = (int)(j % kPStages);
            const uint32_t par = (uint32_t)((j / kPStages) & 1);
            unsigned char *st = p_stage<false, true>(sm, s);
            bool ok = tc::mbar_wait(p_full(sm, s), par, kMaxTries);
            __syncwarp();
            if (bar_or<1, kRows>(!ok)) {
                if (tid == 0) atomicExch(err, CTF_ERR_TIMEOUT);
                break;
            }
            const ExactParams &p = *reinterpret_cast<const ExactParams *>(st + kPBat);
            const MlpDevice &m = *reinterpret_cast<const MlpDevice *>(st + kPBat + sizeof(ExactParams));
            if (m.img != loaded) {
                // another network: its operand image (every MMA of the last chain is done)
                const uint4 *src = m.img;
                uint4 *dst = reinterpret_cast<uint4 *>(sm + kImgW1);
                for (int i = tid; i < kImgBytes / 16; i += kRows) dst[i] = __ldg(src + i);
                tc::fence_proxy_async();  // generic-proxy writes -> the MMAs' async proxy
                cons_bar();
                loaded = m.img;
            }
            const bool fp8 = __shfl_sync(FULL, m.fp8, 0) != 0;
            const int R = min(__shfl_sync(FULL, *reinterpret_cast<const int *>(st + S::kAlloc), 0), kPGroupRows);
            if (kStats && tid == 0) cnt.v[kStatTexelEvalsUnique] += R;
            const int passes = (R + kRows - 1) / kRows;
            float4 *outrow = reinterpret_cast<float4 *>(st + S::kX);
            const uint32_t sX = tc::smem_addr(st + S::kX);
            for (int c = 0; c < passes && ok; ++c) {
                const bool live = kRows * c + 32 * warp < R;
                float4 v;
                bool bad = false;
                const uint32_t sXc = sX + 4096u * (uint32_t)c;
                if (loaded == m0.img)
                    ok = fp8 ? p_chain<true, true>(sm, tmem, mma_bar, phase, sXc, warp, live, ep0, v, bad, err)
                             : p_chain<true, false>(sm, tmem, mma_bar, phase, sXc, warp, live, ep0, v, bad, err);
                else
                    ok = fp8 ? p_chain<false, true>(sm, tmem, mma_bar, phase, sXc, warp, live, ep0, v, bad, err)
                             : p_chain<false, false>(sm, tmem, mma_bar, phase, sXc, warp, live, ep0, v, bad, err);
                if (!ok) break;
                if (live) outrow[ck(kRows * c + tid, kPGroupRows, err, kBndRow)] = v;
                ok = !bar_or<1, kRows>(bad);
                if (!ok && tid == 0) atomicExch(err, CTF_ERR_TIMEOUT);
            }
            if (!ok) break;
            {
                const uint32_t off = LanePlace<TW>(p, lane).off;
#pragma unroll 1
                for (int k = warp; k < kPTiles; k += 4) p_gather<ALG, false>(p, off, k, st, lane, nullptr);
            }
            __syncwarp();
            cons_bar();  // every consumer warp has read the stage
            if (tid == 0) {
                *reinterpret_cast<int *>(st + S::kAlloc) = 0;
                p_arrive(p_done(sm, s));
            }
        }
    } else {
        // ---------------- producers ----------------
        const int pw = warp - 4;
        const uint32_t lt = lanemask_lt();
        int *ranks = reinterpret_cast<int *>(sm + kPRanks) + 64 * pw;
        // this warp's copies of its current and its next group's view
        unsigned char *own = sm + kPRanksEnd + 2 * pw * kPViewBytes;
        auto params = [&](int c) -> const ExactParams & {
            return *reinterpret_cast<const ExactParams *>(own + c * kPViewBytes);
        };
        auto locate = [&](long long it, BatchPlace &at, int c) {
            at = find_batch_view(b.item_begin, b.nkind, it, at.view, lane);
            const BatchViewDev *V =
                b.views + ck(__ldg(b.index + ck(at.view, b.nkind, err, kBndBatch)), b.nviews, err, kBndBatch);
            __syncwarp();
            const uint4 *src = reinterpret_cast<const uint4 *>(&V->p);
            uint4 *dst = reinterpret_cast<uint4 *>(own + c * kPViewBytes);
            if (lane < (int)(sizeof(ExactParams) / 16)) dst[lane] = __ldg(src + lane);
            const uint2 *msrc = reinterpret_cast<const uint2 *>(&V->m);
            uint2 *mdst = reinterpret_cast<uint2 *>(own + c * kPViewBytes + sizeof(ExactParams));
            if (lane < (int)(sizeof(MlpDevice) / 8)) mdst[lane] = __ldg(msrc + lane);
            __syncwarp();
        };
        auto first_tile = [&](long long it, const BatchPlace &at, int c, uint32_t &x, uint32_t &y) {
            const uint32_t t = (uint32_t)((it - at.begin) * kPTiles) + (uint32_t)(kPSlots * pw);
            const uint32_t tiles_x = (uint32_t)params(c).tiles_x;
            x = t % tiles_x;
            y = t / tiles_x;
        };
        BatchPlace at;
        at.view = 0;
        long long item = blockIdx.x;  // (the grid has at most one CTA per item)
        int cur = 0;
        locate(item, at, cur);
        uint32_t bx, by;
        first_tile(item, at, cur, bx, by);
        Inputs in = p_load<ALG, TW>(params(cur), LanePlace<TW>(params(cur), lane), bx, by);
        for (long long j = 0; item < b.total_items; ++j) {
            const int s = (int)(j % kPStages);
            unsigned char *st = p_stage<false, true>(sm, s);
            // the next group's view (a copy into the other slot when it changes)
            const long long next_item = item + gridDim.x;
            const bool more = next_item < b.total_items;
            int nxt = cur;
            if (more && next_item >= at.end) {
                nxt = cur ^ 1;
                locate(next_item, at, nxt);
            }
            // the consumer has gathered group j - kPStages from this stage
            bool okd = true;
            if (j >= kPStages)
                okd = __all_sync(FULL, tc::mbar_wait(p_done(sm, s), (uint32_t)(((j - kPStages) / kPStages) & 1), kMaxTries));
            const ExactParams &p = params(cur);
            if (okd && pw == 0) {  // the view for the consumer
                const uint4 *src = reinterpret_cast<const uint4 *>(own + cur * kPViewBytes);
                if (lane < kPViewBytes / 16) reinterpret_cast<uint4 *>(st + kPBat)[lane] = src[lane];
            }
            const LanePlace<TW> lp(p, lane);
            const uint32_t tiles_x = (uint32_t)p.tiles_x;
#pragma unroll 1
            for (int k = 0; k < kPSlots && okd; ++k) {
                uint32_t nx = bx, ny = by;
                Inputs next;
                if (k + 1 < kPSlots) {
                    p_tile(tiles_x, nx, ny, 1u);
                    next = p_load<ALG, TW>(p, lp, nx, ny);
                } else {
                    // (after the last group: this tile's inputs again, unused)
                    if (more) first_tile(next_item, at, nxt, nx, ny);
                    next = p_load<ALG, TW>(params(nxt), LanePlace<TW>(params(nxt), lane), nx, ny);
                }
                p_step1<ALG, TW, MD, kStats, false>(p, lp, bx, by, in, kPSlots * pw + k, st, lane, lt, ranks,
                                                    cnt, nullptr);
                bx = nx;
                by = ny;
                in = next;
            }
            __syncwarp();
            // every tile's texels are listed (unless a warp gave up its wait)
            if (bar_or<2, kPProducerThreads>(!okd)) {
                if (threadIdx.x == kRows) atomicExch(err, CTF_ERR_TIMEOUT);
                break;
            }
            {
                const MlpDevice &m = *reinterpret_cast<const MlpDevice *>(own + cur * kPViewBytes + sizeof(ExactParams));
                const float *inv_a1 =
                    reinterpret_cast<const float *>(reinterpret_cast<const unsigned char *>(m.img) + kImgA1);
                const int R = *reinterpret_cast<const int *>(st + S::kAlloc), pt = (int)threadIdx.x - kRows;
                if (m.fp8) p_features<S, true>(m, st, R, pt, inv_a1);
                else p_features<S, false>(m, st, R, pt, inv_a1);
            }
            __syncwarp();
            if (lane == 0) p_arrive(p_full(sm, s));
            item = next_item;
            cur = nxt;
        }
    }

    if (kStats && b.stats && lane == 0) {
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
    if (kStats && b.stats && threadIdx.x < kNumStats && block_stats[threadIdx.x])
        atomicAdd(b.stats + threadIdx.x, block_stats[threadIdx.x]);
}

template <int TW, bool kStats, int kVar, bool kFp8>
PfFn pf_pick_alg(int alg, int md) {
    constexpr bool kFb = kVar == kPfFallback, kTwo = kVar == kPfTwoTexels;
    switch (alg) {
    case ALG_STF: return kVar == kPfPlain ? mlp_filter_pf_kernel<ALG_STF, TW, 16, kStats, false, false, kFp8> : nullptr;
    case ALG_LIST: return kFb ? nullptr : mlp_filter_pf_kernel<ALG_LIST, TW, 16, kStats, false, kTwo, kFp8>;
    case ALG_BOX: return mlp_filter_pf_kernel<ALG_BOX, TW, 16, kStats, kFb, kTwo, kFp8>;
    case ALG_MASK:
        return md == 11 ? mlp_filter_pf_kernel<ALG_MASK, TW, 11, kStats, kFb, kTwo, kFp8>
                        : mlp_filter_pf_kernel<ALG_MASK, TW, 16, kStats, kFb, kTwo, kFp8>;
    default: return nullptr;
    }
}

template <int TW, bool kStats, bool kFp8>
PfFn pf_pick_var(int alg, int md, int var) {
    switch (var) {
    case kPfPlain: return pf_pick_alg<TW, kStats, kPfPlain, kFp8>(alg, md);
    case kPfFallback: return pf_pick_alg<TW, kStats, kPfFallback, kFp8>(alg, md);
    case kPfTwoTexels: return pf_pick_alg<TW, kStats, kPfTwoTexels, kFp8>(alg, md);
    default: return nullptr;
    }
}

template <int TW>
PfFn pf_pick(int alg, int md, bool stats, int var, bool fp8) {
    if (stats) return fp8 ? pf_pick_var<TW, true, true>(alg, md, var) : pf_pick_var<TW, true, false>(alg, md, var);
    return fp8 ? pf_pick_var<TW, false, true>(alg, md, var) : pf_pick_var<TW, false, false>(alg, md, var);
}

template <int TW, bool kStats>
BatchPfFn batch_pf_pick_alg(int alg, int md) {
    switch (alg) {
    case ALG_STF: return mlp_batch_pf_kernel<ALG_STF, TW, 16, kStats>;
    case ALG_LIST: return mlp_batch_pf_kernel<ALG_LIST, TW, 16, kStats>;
    case ALG_BOX: return mlp_batch_pf_kernel<ALG_BOX, TW, 16, kStats>;
    case ALG_MASK: return md == 11 ? mlp_batch_pf_kernel<ALG_MASK, TW, 11, kStats> : mlp_batch_pf_kernel<ALG_MASK, TW, 16, kStats>;
    default: return nullptr;
    }
}

template <int TW>
BatchPfFn batch_pf_pick(int alg, int md, bool stats) {
    return stats ? batch_pf_pick_alg<TW, true>(alg, md) : batch_pf_pick_alg<TW, false>(alg, md);
}

// What the host needs to launch the kernels compiled here (one file per tile width).
template <int TW>
PfKernels pf_kernels() {
    PfKernels k;
    k.filter = pf_pick<TW>;
    k.batch = batch_pf_pick<TW>;
    k.threads = kPThreads;
    k.launch_regs = kPLaunchRegs;
    k.ctas_per_sm = kPCtasPerSm;
    k.tiles[kPfPlain] = k.tiles[kPfFallback] = kPTiles;
    k.tiles[kPfTwoTexels] = kPTiles / 2;
    k.smem[kPfPlain] = k.smem[kPfTwoTexels] = PLayout<false>::kBytes;
    k.smem[kPfFallback] = PLayout<true>::kBytes;
    k.batch_smem = PLayout<false, true>::kBytes;
    return k;
}

}  // namespace

#ifndef CTF_MLP_WS2_PART
PfKernels pf_kernels_w8() { return pf_kernels<8>(); }
#endif

}  // namespace ctf
