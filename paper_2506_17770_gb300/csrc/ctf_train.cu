// ctf_train.cu -- training of the learned texel decode on the GPU.
//
// The network of ctf_mlp.cu (two 8-channel latent grids sampled bilinearly,
// 16 -> 64 -> 64 -> 4 with ReLU) is fitted to the exact decode of a block
// texture.  FP32 master parameters live in one device buffer:
//   [w1 1024 | b1 64 | w2 4096 | b2 64 | w3 256 | b3 4 | pad 4 | latent0 | latent1]
// A step samples a batch of texels with Philox4x32-10.  A CTA of 128
// threads takes up to 128 texels per round and runs the forward and
// backward pass as tcgen05 MMAs over them (FP16 operands in shared memory,
// FP32 accumulation in TMEM; bias, ReLU and the loss in FP32): the layer
// products, the input-side gradients and the weight gradients, which it
// sums over its rounds in TMEM and leaves as the CTA's partial sums; the
// latent-grid gradients go to 64-bit fixed-point accumulators (integer
// atomics are order-independent, so a step is deterministic).  A second kernel
// adds the partial sums up and applies Adam to the weights and to the latent
// cells that the next step reads; at the end of a segment of steps all other
// cells take the steps they have missed (advance_kernel, sweep_kernel).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "../../include/ctf.h"
#include "ctf_device.cuh"
#include "ctf_internal.h"
#include "tc_ops.cuh"

namespace ctf {
namespace {

constexpr int kOffW1 = 0, kOffB1 = 1024, kOffW2 = 1088, kOffB2 = 5184, kOffW3 = 5248, kOffB3 = 5504;
constexpr int kWeights = 5508;
constexpr int kOffLat = 5512;
constexpr double kFix = 17592186044416.0;  // 2^44: gradient fixed point
constexpr double kLossFix = 4294967296.0;  // 2^32: loss fixed point
constexpr int kThreads = 128;              // threads of the activation-statistics kernel
constexpr int kT = 128;                    // rows of a round of the gradient kernel (one per thread)
constexpr int kMaxRounds = 4;              // rounds per CTA, at most (unless the batch needs more)
constexpr int kMaxGradCtas = 1024;         // CTAs of the gradient kernel, at most (their partial sums)

struct GradParams {
    const float *params;
    const uint2 *blocks;
    int Wt, Ht, nbx;
    int gw[2], gh[2];
    float sx[2], sy[2];
    const int2 *xy;        // explicit texels, or nullptr: Philox sampling
    int n;                 // texels in this call
    int rounds;            // rounds per CTA
    int per_round;         // texels per round (at most kT; the other rows of the round are empty)
    uint32_t step;         // Philox counter word
    uint32_t k0, k1;       // Philox key
    float dscale;          // 2 / batch
    long long *grad;       // fixed-point gradient accumulators (same layout as params)
    uint32_t *seen;        // per latent cell (grid 0, then grid 1): see advance_kernel
    uint32_t mark;         // the first step of a segment: the value its cells get there, else 0
    long long *loss;       // fixed-point sum of squared errors
    int *err;              // device error word: a wait that gave up records CTF_ERR_TIMEOUT
    unsigned char *wimg;   // the weight image of the gradient kernel (pack_kernel)
    float *partial;        // per-CTA weight-gradient sums [CTA][kWeights], added up in CTA order
};

// v * 2^44 is exact in FP32 (a power-of-two scale), so this rounds the same
// value as the FP64 product would, without FP64 arithmetic.
__device__ __forceinline__ long long to_fix(float v) { return __float2ll_rn(v * 0x1p44f); }

// Shared memory of the gradient kernel (bytes).  Every matrix is an MMA
// operand in FP16, stored K-major in 8-row x 16-byte core matrices (element
// (r, k) at (r/8) * (K/8) * 128 + (k/8) * 128 + (r%8) * 16 + (k%8) * 2):
//   weights as the B operands of the forward and backward products:
//   W1 [64 x 16], W2 [64 x 64], W3 [16 x 64] (rows 4..15 zero), W3^T
//   [64 x 16] (columns 4..15 zero), W2^T [64 x 64], W1^T [16 x 64];
//   AH, one row per texel of the round, 176 channels: H2 (0..63), a ones
//   block (64..79: channel 64 is 1, the rest 0), H1 (80..143), the
//   features F (144..159) and a second ones block (160..175);
//   DH, one row per texel, 128 channels: dH2 (0..63), dH1 (64..127);
//   DE, one row per texel, 16 channels: the output errors (0..3), zeros.
// The weight gradients are products over the round's texels with the
// texel as the reduction index: the same AH and DH buffers, read
// MN-major (channels along MN, texels along K), give
//   [dH2; dH1]^T [H1 | F | 1] -> dW2, dW1 and the bias sums db2, db1 (one
//   MMA chain, M = 128 channels, N = 96), and
//   [H2 | 1 | ...]^T DE -> dW3^T and db3 (M = 128, N = 16),
// accumulated in TMEM over the CTA's rounds.
constexpr int kGW1 = 0;
constexpr int kGW2 = kGW1 + 2048;
constexpr int kGW3 = kGW2 + 8192;
constexpr int kGW3T = kGW3 + 2048;
constexpr int kGW2T = kGW3T + 2048;
constexpr int kGW1T = kGW2T + 8192;
constexpr int kGBias = kGW1T + 2048;              // b1[64], b2[64], b3[4] (FP32)
constexpr int kAHK = 176, kAHGroup = kAHK / 8 * 128;  // channels, bytes per 8-row group
constexpr int kChH2 = 0, kChOnes = 64, kChH1 = 80, kChF = 144, kChOnes2 = 160;
constexpr int kGAH = kGBias + 640;
constexpr int kDHGroup = 128 / 8 * 128;
// after a round's MMAs DH holds the rows' dF (64 B each), then per row and grid
// the four taps' cells and weights (32 B)
constexpr int kDHTaps = 128 * 64;
static_assert(kDHTaps + 128 * 2 * 32 <= 16 * kDHGroup, "inside DH");
constexpr int kGDH = kGAH + 16 * kAHGroup;
constexpr int kGDE = kGDH + 16 * kDHGroup;
constexpr int kGXY = kGDE + 16 * 256;             // int2 [128] texel coordinates
constexpr int kGBar = kGXY + 128 * 8;             // MMA barrier (8 B), TMEM base (4 B)
constexpr int kGSlot = kGBar + 8;
constexpr int kGLoss = kGBar + 16;                // float per warp: squared errors
constexpr int kGradSmemBytes = kGLoss + 16;
static_assert(kGAH % 16 == 0 && kGDH % 16 == 0 && kGDE % 16 == 0, "16-byte operand buffers");
static_assert(2 * (kGradSmemBytes + 1024) <= 228 * 1024 && 3 * (kGradSmemBytes + 1024) > 228 * 1024,
              "exactly two CTAs (2 x 256 TMEM columns) per SM");
constexpr size_t kGradSmem = kGradSmemBytes;
// TMEM columns (FP32, lane = row): forward D1 / backward dE W3^T [0, 64),
// D2 / dH2 W2^T [64, 128), D3 / dH1 W1^T [128, 144), the weight-gradient
// sums [144, 240) and [240, 256).
constexpr uint32_t kTcCols = 256, kColA = 0, kColB = 64, kColC = 128, kColWG1 = 144, kColWG2 = 240;
constexpr uint32_t kGradTries = 1u << 24;

__host__ __device__ constexpr uint32_t idesc_f16_t(int M, int N, int ta, int tb) {
    return (1u << 4) | ((uint32_t)ta << 15) | ((uint32_t)tb << 16) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ uint32_t h2pack(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ uint32_t relu_h2(float a, float b) {
    uint32_t r;
    asm("cvt.rn.relu.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
    return r;
}

// Offset of element (r, k) in a K-major FP16 operand with K channels.
__device__ __forceinline__ int kofs(int r, int k, int K) { return (r >> 3) * (K / 8) * 128 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2; }

__device__ __forceinline__ uint32_t saddr_of(const void *p) { return tc::smem_addr(p); }

// The end of the MMAs committed to `bar`, polled by every thread.  Returns
// false if they did not complete within the bound; the caller goes on and the
// threads agree on it at their next barrier.
__device__ __forceinline__ bool tc_wait(uint64_t *bar, uint32_t &phase) {
    const bool ok = tc::mbar_wait(bar, phase, kGradTries);
    phase ^= 1u;
    __syncwarp();  // the TMEM accesses that follow are .aligned
    tc::fence_after_sync();
    return ok;
}

// Generic-proxy shared-memory writes of every thread made visible to the
// MMAs issued next.  Returns false (for all threads alike) if a thread gave
// up a wait.
__device__ __forceinline__ bool tc_publish(bool bad) {
    tc::fence_proxy_async();
    tc::fence_before_sync();
    const bool any = __syncthreads_or(bad);
    tc::fence_after_sync();
    return !any;
}

__device__ __forceinline__ void tld16(uint32_t taddr, float v[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    // the loaded registers pass through an empty asm after the wait, so that
    // no use of them can be scheduled before it
#pragma unroll
    for (int i = 0; i < 16; ++i) asm volatile("" : "+r"(r[i]));
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void bilinear_taps(const GradParams &g, int grid, int x, int y, int idx[4], float w[4]) {
    // grid is 0 or 1; selecting by value keeps the parameter block out of local memory
    const float sx = grid ? g.sx[1] : g.sx[0], sy = grid ? g.sy[1] : g.sy[0];
    const int gw = grid ? g.gw[1] : g.gw[0], gh = grid ? g.gh[1] : g.gh[0];
    const float gx = __fsub_rn(__fmul_rn(__fadd_rn((float)x, 0.5f), sx), 0.5f);
    const float gy = __fsub_rn(__fmul_rn(__fadd_rn((float)y, 0.5f), sy), 0.5f);
    const float fx0 = floorf(gx), fy0 = floorf(gy);
    const float fx = __fsub_rn(gx, fx0), fy = __fsub_rn(gy, fy0);
    const int x0 = (int)fx0, y0 = (int)fy0;
    const int xa = min(max(x0, 0), gw - 1), xb = min(max(x0 + 1, 0), gw - 1);
    const int ya = min(max(y0, 0), gh - 1), yb = min(max(y0 + 1, 0), gh - 1);
    const long long cells = (long long)gw * gh;
    idx[0] = ck(ya * gw + xa, cells, g.err, kBndLatent);
    idx[1] = ck(ya * gw + xb, cells, g.err, kBndLatent);
    idx[2] = ck(yb * gw + xa, cells, g.err, kBndLatent);
    idx[3] = ck(yb * gw + xb, cells, g.err, kBndLatent);
    const float ofx = __fsub_rn(1.f, fx), ofy = __fsub_rn(1.f, fy);
    w[0] = __fmul_rn(ofx, ofy);
    w[1] = __fmul_rn(fx, ofy);
    w[2] = __fmul_rn(ofx, fy);
    w[3] = __fmul_rn(fx, fy);
}


// Texel i of the step's batch.
__device__ __forceinline__ void sample_texel(const GradParams &g, uint32_t step, uint32_t i, int &x, int &y) {
    const uint4 rr = philox4x32_10(make_uint4(i, step, 0x5A4Du, 0u), g.k0, g.k1);
    x = (int)(((unsigned long long)rr.x * (unsigned)g.Wt) >> 32);
    y = (int)(((unsigned long long)rr.y * (unsigned)g.Ht) >> 32);
}

// A CTA's partial weight-gradient sums, in the order in which its threads
// hold them (thread m row m of the two products), so that a warp stores 32
// neighbours: dW2 [input][output], dW1 [input][output], db2, db1, dW3, db3.
// (In parameter order every lane stored to a sector of its own, 1.6 million
// sectors a step at batch 8,192.)
constexpr int kSlotW1 = 4096, kSlotB = 5120, kSlotW3 = 5248, kSlotB3 = 5504;

// The parameter of slot s.
__device__ __forceinline__ int slot_param(int s) {
    if (s < kSlotW1) return kOffW2 + (s & 63) * 64 + (s >> 6);
    if (s < kSlotB) return kOffW1 + (s & 63) * 16 + ((s - kSlotW1) >> 6);
    if (s < kSlotB + 64) return kOffB2 + s - kSlotB;
    if (s < kSlotW3) return kOffB1 + s - kSlotB - 64;
    return s - kSlotW3 + kOffW3;  // dW3 and db3 follow one another in both
}
static_assert(kSlotB3 - kSlotW3 == kOffB3 - kOffW3 && kSlotB3 + 4 == kWeights, "one slot per parameter");

// Where parameter e of the network goes in the gradient kernel's weight image
// (the first kGAH bytes of its shared memory: W1, W2, W3 and their transposes
// as FP16 operands, the biases in FP32).
__device__ __forceinline__ void put_weight(unsigned char *img, int e, float v) {
    const __half w = __float2half_rn(v);
    if (e < kOffB1) {
        const int o = e >> 4, k = e & 15;
        *reinterpret_cast<__half *>(img + kGW1 + kofs(o, k, 16)) = w;
        *reinterpret_cast<__half *>(img + kGW1T + kofs(k, o, 64)) = w;
    } else if (e < kOffW2) {
        reinterpret_cast<float *>(img + kGBias)[e - kOffB1] = v;
    } else if (e < kOffB2) {
        const int j = e - kOffW2, o = j >> 6, k = j & 63;
        *reinterpret_cast<__half *>(img + kGW2 + kofs(o, k, 64)) = w;
        *reinterpret_cast<__half *>(img + kGW2T + kofs(k, o, 64)) = w;
    } else if (e < kOffW3) {
        reinterpret_cast<float *>(img + kGBias)[64 + e - kOffB2] = v;
    } else if (e < kOffB3) {
        const int j = e - kOffW3, c = j >> 6, k = j & 63;
        *reinterpret_cast<__half *>(img + kGW3 + kofs(c, k, 64)) = w;
        *reinterpret_cast<__half *>(img + kGW3T + kofs(k, c, 16)) = w;
    } else {
        reinterpret_cast<float *>(img + kGBias)[128 + e - kOffB3] = v;
    }
}

// Before the first step of a call: the weight image from the current FP32
// master parameters (the updates keep it current from then on).  One thread
// per element.
__global__ void pack_kernel(const float *params, unsigned char *img) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 1024) {
        const int o = i >> 4, k = i & 15;
        const __half w = __float2half_rn(params[kOffW1 + i]);
        *reinterpret_cast<__half *>(img + kGW1 + kofs(o, k, 16)) = w;
        *reinterpret_cast<__half *>(img + kGW1T + kofs(k, o, 64)) = w;
    } else if (i < 1024 + 4096) {
        const int j = i - 1024, o = j >> 6, k = j & 63;
        const __half w = __float2half_rn(params[kOffW2 + j]);
        *reinterpret_cast<__half *>(img + kGW2 + kofs(o, k, 64)) = w;
        *reinterpret_cast<__half *>(img + kGW2T + kofs(k, o, 64)) = w;
    } else if (i < 1024 + 4096 + 1024) {
        const int j = i - 5120, c = j >> 6, k = j & 63;
        const __half w = __float2half_rn(c < 4 ? params[kOffW3 + j] : 0.f);
        *reinterpret_cast<__half *>(img + kGW3 + kofs(c, k, 64)) = w;   // rows 4..15 zero
        *reinterpret_cast<__half *>(img + kGW3T + kofs(k, c, 16)) = w;  // columns 4..15 zero
    } else if (i < 6144 + 160) {
        const int j = i - 6144;  // biases b1 (64), b2 (64), b3 (4), zero padding
        float v = 0.f;
        if (j < 64) v = params[kOffB1 + j];
        else if (j < 128) v = params[kOffB2 + j - 64];
        else if (j < 132) v = params[kOffB3 + j - 128];
        reinterpret_cast<float *>(img + kGBias)[j] = v;
    }
}
constexpr int kPackThreads = 6144 + 160;
static_assert(kGBias + 160 * 4 == kGAH, "the image ends where the activations begin");

// Forward and backward pass of kT texels per round on the tensor cores:
// thread t owns texel row t of every per-texel operand and TMEM lane t.
// Per round: features (FP32, from the FP32 master latents) and targets;
// H1 = relu(F W1^T + b1), H2 = relu(H1 W2^T + b2), Y = H2 W3^T + b3 (FP16
// operands, FP32 accumulation, bias and ReLU in FP32); e = Y - target;
// dH2 = (e W3) masked by H2 > 0, dH1 = (dH2 W2) masked by H1 > 0,
// dF = dH1 W1; the weight gradients accumulate in TMEM; dF, times the
// bilinear tap weights and 2 / batch, goes to the latent cells.  The CTA's
// weight-gradient sums (times 2 / batch) and its squared errors go to the
// 64-bit fixed-point accumulators at the end.  Rows past the batch carry
// e = 0 and so contribute nothing.
__global__ void __launch_bounds__(kT, 2) grad_kernel(const GradParams g) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x;
    const int warp = __shfl_sync(FULL, tid >> 5, 0);  // uniform, and known to be
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + kGBar);
    uint32_t *slot = reinterpret_cast<uint32_t *>(sm + kGSlot);
    float *sloss = reinterpret_cast<float *>(sm + kGLoss);
    unsigned char *AH = sm + kGAH, *DH = sm + kGDH, *DE = sm + kGDE;
    const float *P = g.params;  // latents (FP32 master values)
    // ---- the constant ones blocks, and zero features in rows that no round uses
    const float *B = reinterpret_cast<const float *>(sm + kGBias);
    {
        // the ones blocks of every row: channels 64 and 160 are 1, the rest of
        // their 16-channel blocks 0 (never written again)
        const uint4 one = make_uint4(0x3C00u, 0u, 0u, 0u), zero = make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4 *>(AH + kofs(tid, kChOnes, kAHK)) = one;
        *reinterpret_cast<uint4 *>(AH + kofs(tid, kChOnes + 8, kAHK)) = zero;
        *reinterpret_cast<uint4 *>(AH + kofs(tid, kChOnes2, kAHK)) = one;
        *reinterpret_cast<uint4 *>(AH + kofs(tid, kChOnes2 + 8, kAHK)) = zero;
        *reinterpret_cast<uint4 *>(AH + kofs(tid, kChF, kAHK)) = zero;
        *reinterpret_cast<uint4 *>(AH + kofs(tid, kChF + 8, kAHK)) = zero;
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr_of(bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        __syncwarp();  // tcgen05.alloc needs the whole warp
        tc::tmem_alloc(slot, kTcCols);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *slot;
    const uint32_t lane_t = tmem + ((uint32_t)(32 * (tid >> 5)) << 16);  // this thread's TMEM lane
    uint32_t phase = 0;
    bool ok = true;
    const size_t lat1 = (size_t)g.gw[0] * g.gh[0] * 8;  // start of the second grid
    const uint32_t sAH = saddr_of(AH), sDH = saddr_of(DH), sDE = saddr_of(DE);
    const uint32_t id64 = idesc_f16_t(128, 64, 0, 0), id16 = idesc_f16_t(128, 16, 0, 0);
    const uint32_t idW1 = idesc_f16_t(128, 96, 1, 1), idW2 = idesc_f16_t(128, 16, 1, 1);
    float loss = 0.f;

    // Half rounds (64 texels): two threads share a texel, one latent grid
    // each, for the features and for the gradient scatter; the rows past the
    // texels keep zero features.
    const bool half = g.per_round <= kT / 2;
    const int row = half ? tid & (kT / 2 - 1) : tid;
    const int g_lo = half ? tid / (kT / 2) : 0, g_hi = half ? g_lo + 1 : 2;
    // This thread's texel of round r (`there`; `valid`: it is row tid's) and
    // its target.
    int x, y;
    bool there, valid;
    float tgt[4];
    auto pick = [&](int r) {
        const int i = (blockIdx.x * g.rounds + r) * g.per_round + row;
        there = row < g.per_round && i < g.n;
        valid = there && row == tid;
        if (g.xy) {
            const int2 c = there ? g.xy[ck(i, g.n, g.err, kBndTrain)] : make_int2(0, 0);
            x = min(max(c.x, 0), g.Wt - 1);
            y = min(max(c.y, 0), g.Ht - 1);
        } else {
            sample_texel(g, g.step, (uint32_t)i, x, y);
        }
        const uint32_t px = fetch_block_texel(g.blocks, g.nbx, g.Wt, g.Ht, x, y, g.err);
#pragma unroll
        for (int c = 0; c < 4; ++c) tgt[c] = __fdiv_rn((float)((px >> (8 * c)) & 0xffu), 255.f);
    };
    pick(0);
    // Launched as the dependent of the previous step's update: what comes
    // before this line (the first texels and their targets too) overlaps its
    // end.  The next update may start from here on (it only loads before it
    // waits for this kernel).
    grid_wait();
    grid_trigger();
    // ---- the weights as FP16 operands and the biases (the image made from
    // the current parameters): in flight together with the first latents
    constexpr int kImg16 = kGAH / 16, kImgLoads = (kImg16 + kT - 1) / kT;
    uint4 img[kImgLoads];
#pragma unroll
    for (int k = 0; k < kImgLoads; ++k)
        img[k] = __ldcg(reinterpret_cast<const uint4 *>(g.wimg) + min(tid + k * kT, kImg16 - 1));
    bool bad = false;
#pragma unroll 1
    for (int r = 0; r < g.rounds && ok; ++r) {
#pragma unroll 1
        for (int gi = g_lo; gi < g_hi; ++gi) {
            int tap[4];
            float tw[4];
            bilinear_taps(g, gi, x, y, tap, tw);
            const float *lg = P + kOffLat + (gi ? lat1 : 0);
            float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            float4 v0[4], v1[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                v0[k] = __ldcg(reinterpret_cast<const float4 *>(lg + (size_t)tap[k] * 8));
                v1[k] = __ldcg(reinterpret_cast<const float4 *>(lg + (size_t)tap[k] * 8 + 4));
            }
            if (r == 0 && gi == g_lo) {
#pragma unroll
                for (int k = 0; k < kImgLoads; ++k)
                    if (tid + k * kT < kImg16) reinterpret_cast<uint4 *>(sm)[tid + k * kT] = img[k];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                acc[0] = __fmaf_rn(tw[k], v0[k].x, acc[0]);
                acc[1] = __fmaf_rn(tw[k], v0[k].y, acc[1]);
                acc[2] = __fmaf_rn(tw[k], v0[k].z, acc[2]);
                acc[3] = __fmaf_rn(tw[k], v0[k].w, acc[3]);
                acc[4] = __fmaf_rn(tw[k], v1[k].x, acc[4]);
                acc[5] = __fmaf_rn(tw[k], v1[k].y, acc[5]);
                acc[6] = __fmaf_rn(tw[k], v1[k].z, acc[6]);
                acc[7] = __fmaf_rn(tw[k], v1[k].w, acc[7]);
            }
            *reinterpret_cast<uint4 *>(AH + kofs(row, kChF + 8 * gi, kAHK)) =
                make_uint4(h2pack(acc[0], acc[1]), h2pack(acc[2], acc[3]), h2pack(acc[4], acc[5]), h2pack(acc[6], acc[7]));
        }
        if (!(ok = tc_publish(bad))) break;
        // ---- H1 = relu(F W1^T + b1)
        if (warp == 0 && tc::elect_one()) {
            tc::mma_f16(tmem + kColA, tc::smem_desc(sAH + kChF / 8 * 128, 128, kAHGroup),
                        tc::smem_desc(saddr_of(sm + kGW1), 128, 256), id64, false);
            tc::commit(bar);
        }
        bad |= !tc_wait(bar, phase);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float d[16];
            tld16(lane_t + kColA + 16 * q, d);
            uint32_t w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                w[j] = relu_h2(__fadd_rn(d[2 * j], B[16 * q + 2 * j]), __fadd_rn(d[2 * j + 1], B[16 * q + 2 * j + 1]));
            *reinterpret_cast<uint4 *>(AH + kofs(tid, kChH1 + 16 * q, kAHK)) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4 *>(AH + kofs(tid, kChH1 + 16 * q + 8, kAHK)) = make_uint4(w[4], w[5], w[6], w[7]);
        }
        if (!(ok = tc_publish(bad))) break;
        // ---- H2 = relu(H1 W2^T + b2)
        if (warp == 0 && tc::elect_one()) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                tc::mma_f16(tmem + kColB, tc::smem_desc(sAH + kChH1 / 8 * 128 + 256 * j, 128, kAHGroup),
                       tc::smem_desc(saddr_of(sm + kGW2) + 256 * j, 128, 1024), id64, j > 0);
            tc::commit(bar);
        }
        bad |= !tc_wait(bar, phase);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float d[16];
            tld16(lane_t + kColB + 16 * q, d);
            uint32_t w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                w[j] = relu_h2(__fadd_rn(d[2 * j], B[64 + 16 * q + 2 * j]),
                               __fadd_rn(d[2 * j + 1], B[64 + 16 * q + 2 * j + 1]));
            *reinterpret_cast<uint4 *>(AH + kofs(tid, kChH2 + 16 * q, kAHK)) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4 *>(AH + kofs(tid, kChH2 + 16 * q + 8, kAHK)) = make_uint4(w[4], w[5], w[6], w[7]);
        }
        if (!(ok = tc_publish(bad))) break;
        // ---- Y = H2 W3^T + b3, e = Y - target (0 past the batch)
        if (warp == 0 && tc::elect_one()) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                tc::mma_f16(tmem + kColC, tc::smem_desc(sAH + kChH2 / 8 * 128 + 256 * j, 128, kAHGroup),
                       tc::smem_desc(saddr_of(sm + kGW3) + 256 * j, 128, 1024), id16, j > 0);
            tc::commit(bar);
        }
        bad |= !tc_wait(bar, phase);
        {
            float d[16];
            tld16(lane_t + kColC, d);
            float e[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                e[c] = valid ? __fsub_rn(__fadd_rn(d[c], B[128 + c]), tgt[c]) : 0.f;
                loss = __fmaf_rn(e[c], e[c], loss);
            }
            *reinterpret_cast<uint4 *>(DE + kofs(tid, 0, 16)) = make_uint4(h2pack(e[0], e[1]), h2pack(e[2], e[3]), 0u, 0u);
            *reinterpret_cast<uint4 *>(DE + kofs(tid, 8, 16)) = make_uint4(0u, 0u, 0u, 0u);
        }
        if (!(ok = tc_publish(bad))) break;
        // ---- dH2 = (e W3) masked by H2 > 0
        if (warp == 0 && tc::elect_one()) {
            tc::mma_f16(tmem + kColA, tc::smem_desc(sDE, 128, 256), tc::smem_desc(saddr_of(sm + kGW3T), 128, 256), id64,
                        false);
            tc::commit(bar);
        }
        bad |= !tc_wait(bar, phase);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float d[16];
            tld16(lane_t + kColA + 16 * q, d);
            const uint4 h0 = *reinterpret_cast<const uint4 *>(AH + kofs(tid, kChH2 + 16 * q, kAHK));
            const uint4 h1 = *reinterpret_cast<const uint4 *>(AH + kofs(tid, kChH2 + 16 * q + 8, kAHK));
            const __half *hh0 = reinterpret_cast<const __half *>(&h0), *hh1 = reinterpret_cast<const __half *>(&h1);
            uint32_t w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const __half a = j < 4 ? hh0[2 * j] : hh1[2 * j - 8], b = j < 4 ? hh0[2 * j + 1] : hh1[2 * j - 7];
                w[j] = h2pack(__half2float(a) > 0.f ? d[2 * j] : 0.f, __half2float(b) > 0.f ? d[2 * j + 1] : 0.f);
            }
            *reinterpret_cast<uint4 *>(DH + kofs(tid, 16 * q, 128)) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4 *>(DH + kofs(tid, 16 * q + 8, 128)) = make_uint4(w[4], w[5], w[6], w[7]);
        }
        if (!(ok = tc_publish(bad))) break;
        // ---- dH1 = (dH2 W2) masked by H1 > 0
        if (warp == 0 && tc::elect_one()) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                tc::mma_f16(tmem + kColB, tc::smem_desc(sDH + 256 * j, 128, kDHGroup),
                            tc::smem_desc(saddr_of(sm + kGW2T) + 256 * j, 128, 1024),
                       id64, j > 0);
            tc::commit(bar);
        }
        bad |= !tc_wait(bar, phase);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float d[16];
            tld16(lane_t + kColB + 16 * q, d);
            const uint4 h0 = *reinterpret_cast<const uint4 *>(AH + kofs(tid, kChH1 + 16 * q, kAHK));
            const uint4 h1 = *reinterpret_cast<const uint4 *>(AH + kofs(tid, kChH1 + 16 * q + 8, kAHK));
            const __half *hh0 = reinterpret_cast<const __half *>(&h0), *hh1 = reinterpret_cast<const __half *>(&h1);
            uint32_t w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const __half a = j < 4 ? hh0[2 * j] : hh1[2 * j - 8], b = j < 4 ? hh0[2 * j + 1] : hh1[2 * j - 7];
                w[j] = h2pack(__half2float(a) > 0.f ? d[2 * j] : 0.f, __half2float(b) > 0.f ? d[2 * j + 1] : 0.f);
            }
            *reinterpret_cast<uint4 *>(DH + kofs(tid, 64 + 16 * q, 128)) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4 *>(DH + kofs(tid, 64 + 16 * q + 8, 128)) = make_uint4(w[4], w[5], w[6], w[7]);
        }
        if (!(ok = tc_publish(bad))) break;
        // ---- dF = dH1 W1; the weight gradients of the round (texels as the
        // reduction index, both operands read MN-major)
        if (warp == 0 && tc::elect_one()) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                tc::mma_f16(tmem + kColC, tc::smem_desc(sDH + 64 / 8 * 128 + 256 * j, 128, kDHGroup),
                       tc::smem_desc(saddr_of(sm + kGW1T) + 256 * j, 128, 1024), id16, j > 0);
            for (int s = 0; s < kT / 16; ++s) {
                const bool acc = r > 0 || s > 0;
                // [dH2 dH1]^T [H1 F 1]: A = DH (channels along MN), B = AH channels 80..175
                tc::mma_f16(tmem + kColWG1, tc::smem_desc(sDH + 2 * kDHGroup * s, kDHGroup, 128),
                       tc::smem_desc(sAH + kChH1 / 8 * 128 + 2 * kAHGroup * s, kAHGroup, 128), idW1, acc);
                // [H2 1 H1]^T e: A = AH channels 0..127, B = DE
                tc::mma_f16(tmem + kColWG2, tc::smem_desc(sAH + 2 * kAHGroup * s, kAHGroup, 128), tc::smem_desc(sDE + 512 * s, 256, 128),
                       idW2, acc);
            }
            tc::commit(bar);
        }
        bad |= !tc_wait(bar, phase);
        // ---- the latent-grid gradient.  The rows' dF, taps and tap weights go
        // through shared memory (DH, which the MMAs have read), and a warp adds
        // one texel and grid at a time: 8 lanes a cell, its four cells side by
        // side, so that a warp's atomics go to 8 sectors and not to 32.
        {
            float df[16];
            tld16(lane_t + kColC, df);  // warp-collective: every lane takes it
#pragma unroll
            for (int c = 0; c < 4; ++c)
                *reinterpret_cast<float4 *>(DH + 64 * tid + 16 * c) =
                    make_float4(df[4 * c], df[4 * c + 1], df[4 * c + 2], df[4 * c + 3]);
            for (int gi = g_lo; gi < g_hi; ++gi) {
                int tap[4];
                float tw[4];
                bilinear_taps(g, gi, x, y, tap, tw);
                *reinterpret_cast<int4 *>(DH + kDHTaps + 32 * (2 * row + gi)) = make_int4(tap[0], tap[1], tap[2], tap[3]);
                *reinterpret_cast<float4 *>(DH + kDHTaps + 32 * (2 * row + gi) + 16) =
                    make_float4(__fmul_rn(tw[0], g.dscale), __fmul_rn(tw[1], g.dscale), __fmul_rn(tw[2], g.dscale),
                                __fmul_rn(tw[3], g.dscale));
            }
        }
        if (!(ok = !__syncthreads_or(bad))) break;
        {
            const int lane = tid & 31, k = lane >> 3, ch = lane & 7, row0 = row - lane;
            const int n = __popc(__ballot_sync(FULL, there));  // (the warp's texels are its first n rows)
            for (int gi = g_lo; gi < g_hi; ++gi) {
                unsigned long long *gl = reinterpret_cast<unsigned long long *>(g.grad + kOffLat + (gi ? lat1 : 0)) + ch;
                const uint32_t cell0 = gi ? (uint32_t)(lat1 / 8) : 0u;
#pragma unroll 4
                for (int t = 0; t < n; ++t) {
                    const unsigned char *rec = DH + kDHTaps + 32 * (2 * (row0 + t) + gi) + 4 * k;
                    const int cell = *reinterpret_cast<const int *>(rec);
                    const float w = *reinterpret_cast<const float *>(rec + 16);
                    const float df = *reinterpret_cast<const float *>(DH + 64 * (row0 + t) + 32 * gi + 4 * ch);
                    if (g.mark && ch == 0) atomicMax(g.seen + cell0 + cell, g.mark);
                    const long long v = to_fix(__fmul_rn(w, df));
                    if (v) atomicAdd(gl + (size_t)cell * 8, (unsigned long long)v);
                }
            }
        }
        if (r + 1 < g.rounds) pick(r + 1);
    }
    if (ok) ok = !__syncthreads_or(bad);
    // ---- the CTA's weight-gradient sums, row m = tid of the two products,
    // stored as this CTA's partial sums (added up in CTA order: no atomics on
    // the few thousand weight entries)
    if (ok) {
        float *W = g.partial + (size_t)ck((int)blockIdx.x, kMaxGradCtas, g.err, kBndTrain) * kWeights;
        const int m = tid;
#pragma unroll 1
        for (int q = 0; q < 6; ++q) {
            float d[16];
            tld16(lane_t + kColWG1 + 16 * q, d);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const int n = 16 * q + j;
                if (m < 64 && n < 64) W[n * 64 + m] = d[j];                              // dW2
                else if (m >= 64 && n >= 64 && n < 80) W[kSlotW1 + (n - 64) * 64 + m - 64] = d[j];  // dW1
                else if (n == 80) W[kSlotB + m] = d[j];                                  // db2, db1
            }
        }
        {
            float d[16];
            tld16(lane_t + kColWG2, d);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (m < 64) W[kSlotW3 + c * 64 + m] = d[c];
                else if (m == 64) W[kSlotB3 + c] = d[c];
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) loss = __fadd_rn(loss, __shfl_xor_sync(FULL, loss, o));
        if ((tid & 31) == 0) sloss[warp] = loss;
    }
    tc::fence_before_sync();
    __syncthreads();
    if (ok && tid == 0) {
        float tot = 0.f;
        for (int s = 0; s < kT / 32; ++s) tot = __fadd_rn(tot, sloss[s]);
        atomicAdd(reinterpret_cast<unsigned long long *>(g.loss), (unsigned long long)__double2ll_rn((double)tot * kLossFix));
    }
    if (!ok && tid == 0 && g.err) atomicExch(g.err, CTF_ERR_TIMEOUT);
    if (warp == 0) {
        __syncwarp();  // tcgen05.dealloc needs the whole warp
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, kTcCols);
    }
}

// The weight gradients (ctf_trainer_gradients; a step's update adds them up the
// same way itself): the CTAs' partial sums added up in CTA order (FP64), times
// 2 / batch, into the fixed-point accumulators.  A block takes 16
// entries; its 16 thread rows each add every 16th CTA in order (loads
// issued 8 at a time), and the 16 row sums are added in row order, so the
// result does not depend on timing.
constexpr int kRedEntries = 16, kRedRows = 16;

// Thread row `row`'s share of slot e: every 16th CTA in order.
__device__ __forceinline__ double partial_sum(const float *partial, int ctas, int e, int row) {
    double acc = 0.0;
    for (int c0 = row; c0 < ctas; c0 += 8 * kRedRows) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = c0 + j * kRedRows;
            v[j] = c < ctas ? __ldcg(partial + (size_t)c * kWeights + e) : 0.f;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) acc += (double)v[j];
    }
    return acc;
}

__global__ void __launch_bounds__(kRedEntries * kRedRows) reduce_kernel(const float *partial, int ctas, double dscale,
                                                                       long long *grad) {
    __shared__ double part[kRedRows][kRedEntries];
    const int e = blockIdx.x * kRedEntries + (threadIdx.x % kRedEntries), row = threadIdx.x / kRedEntries;
    part[row][threadIdx.x % kRedEntries] = e < kWeights ? partial_sum(partial, ctas, e, row) : 0.0;
    __syncthreads();
    if (row == 0 && e < kWeights) {
        double tot = 0.0;
        for (int r = 0; r < kRedRows; ++r) tot += part[r][threadIdx.x];
        grad[slot_param(e)] = __double2ll_rn(tot * dscale * kFix);
    }
}

// Steps of a segment at most (see advance_kernel): 4096^2 texture, 8,192
// texels, 64 steps 2.72 ms with 8, 2.61 with 16, 2.59 with 32, 2.82 with 64.
constexpr int kSegment = 16;

// What a step multiplies: the learning rate over the first bias correction
// (weights, latents) and 1 / (1 - beta2^t).
struct AdamStep {
    float w, lat, inv_bc2;
};

struct AdamParams {
    float *params, *m, *v;
    long long *grad;
    size_t n;
    float beta1, beta2, eps;
    AdamStep st[kSegment];   // the segment's steps
    int j;                   // this step's place in them
    uint32_t base;           // steps before the segment
    uint32_t *seen;          // per latent cell, see advance_kernel
    const float *partial;    // the gradient kernel's weight sums, `ctas` of them
    int ctas;
    double dscale;           // 2 / batch
    unsigned char *wimg;     // the weight image, kept current
    int descending;          // sweep_kernel walks the latents from the last one down
};

__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// p -= step * m / (sqrt(v / (1 - beta2^t)) + eps) after the moment updates
// (bias corrections folded into step and inv_bc2; approximate square root
// and division, as an optimiser needs no correctly rounded update).
__device__ __forceinline__ void adam_update(const AdamParams &a, long long gi, float step, float inv_bc2, float &p,
                                            float &m, float &v) {
    const float gr = __ll2float_rn(gi) * 0x1p-44f;  // fixed point back to FP32 (exact scale)
    m = __fmaf_rn(a.beta1, m, (1.f - a.beta1) * gr);
    v = __fmaf_rn(a.beta2, v, (1.f - a.beta2) * (gr * gr));
    p = __fmaf_rn(-step, __fdividef(m, sqrt_approx(v * inv_bc2) + a.eps), p);
}

__device__ __forceinline__ void adam_quad(const AdamParams &a, const AdamStep &st, float4 &p, float4 &m, float4 &v,
                                          longlong2 g01, longlong2 g23) {
    adam_update(a, g01.x, st.lat, st.inv_bc2, p.x, m.x, v.x);
    adam_update(a, g01.y, st.lat, st.inv_bc2, p.y, m.y, v.y);
    adam_update(a, g23.x, st.lat, st.inv_bc2, p.z, m.z, v.z);
    adam_update(a, g23.y, st.lat, st.inv_bc2, p.w, m.w, v.w);
}

// The weights' share of a step, 16 slots per CTA and turn for CTA `first`, +
// `ctas`, ...: the gradient CTAs' partial sums added in CTA order (as in
// reduce_kernel), Adam, and the operand image.
__device__ __forceinline__ void update_weights(const AdamParams &a, const AdamStep &st, int first, int ctas) {
    __shared__ double part[kRedRows][kRedEntries];
    for (int b = first; b * kRedEntries < kWeights; b += ctas) {
        const int e = b * kRedEntries + (threadIdx.x % kRedEntries), row = threadIdx.x / kRedEntries;
        const int w = e < kWeights ? slot_param(e) : 0;
        float p = 0.f, m = 0.f, v = 0.f;
        if (row == 0) {
            p = __ldcg(a.params + w);
            m = __ldcg(a.m + w);
            v = __ldcg(a.v + w);
        }
        part[row][threadIdx.x % kRedEntries] = e < kWeights ? partial_sum(a.partial, a.ctas, e, row) : 0.0;
        __syncthreads();
        if (row == 0 && e < kWeights) {
            double tot = 0.0;
            for (int r = 0; r < kRedRows; ++r) tot += part[r][threadIdx.x];
            adam_update(a, __double2ll_rn(tot * a.dscale * kFix), st.w, st.inv_bc2, p, m, v);
            a.params[w] = p;
            a.m[w] = m;
            a.v[w] = v;
            put_weight(a.wimg, w, p);
        }
        __syncthreads();
    }
}

// A step's Adam update reaches every cell, but a cell that no texel of the
// step reads takes it with a gradient of zero, which needs nothing but the
// cell itself.  So the steps of a call run in segments of up to kSegment; a
// cell stands still within a segment until a step is about to read it
// (advance_kernel) or the segment ends (sweep_kernel), and then takes the steps
// it has missed one after the other, the same operations in the same order.
// The first of them is the step that read it last, whose gradient waits in the
// accumulators; the others have none.  A segment moves the 24 bytes of a
// parameter once, and once more each time its cell is read, and not once a step.
// seen[cell]: 1 + the steps that the cell had taken when it was last brought
// up to date to be read; a value up to `base` is from before the segment.
//
// advance_kernel, which runs beside the gradients of step j and ends after
// them: the cells that step j + 1 reads take their steps up to j, and the
// weights take step j.  Two threads per cell, sixteen per texel; the first to
// reach a cell claims it.  Only cells that step j reads too (`late`) wait for
// its gradients; the gradient kernel neither reads nor changes the others.
// What it reads and claims before that wait (`seen`, parameters, moments,
// accumulators) the update before wrote.  griddepcontrol.wait would order only
// what the gradient kernel wrote; that the update before is over rests on the
// gradient kernel, which lets this one begin only after its own wait for it, and
// that its results are seen on the loads (__ldcg), stores and atomics, which
// meet in L2 and leave no line of these arrays in an SM's L1.
// 4096^2 texture, 8,192 texels: 34 us a step in a call of 64 (gradients and
// advance 29, a sixteenth of a sweep 6); 66 us in calls of one step, whose
// sweep moves every parameter, and 93 us with an Adam kernel of all cells and
// five more launches a step.  Five CTAs per SM 36 us.
constexpr int kAdvThreads = 256, kAdvCtasPerSm = 4;
__global__ void __launch_bounds__(kAdvThreads, kAdvCtasPerSm) advance_kernel(const GradParams g, const AdamParams a) {
    static_assert(kAdvThreads == kRedEntries * kRedRows, "the weight sums' thread layout");
    float4 *__restrict__ P = reinterpret_cast<float4 *>(a.params + kOffLat);
    float4 *__restrict__ M = reinterpret_cast<float4 *>(a.m + kOffLat);
    float4 *__restrict__ V = reinterpret_cast<float4 *>(a.v + kOffLat);
    longlong2 *__restrict__ G = reinterpret_cast<longlong2 *>(a.grad + kOffLat);
    const longlong2 z = make_longlong2(0, 0);
    const uint32_t j = (uint32_t)a.j, seen = a.base + j + 2;
    const long long items = 16ll * g.n, stride = (long long)gridDim.x * kAdvThreads;
    const int sub = threadIdx.x & 15, gi = sub >> 3, tap = (sub >> 1) & 3;
    bool waited = false;
    for (long long e = (long long)blockIdx.x * kAdvThreads + threadIdx.x; __shfl_sync(FULL, e, 0) < items; e += stride) {
        const bool valid = e < items;  // (the threads of a texel alike)
        int x, y, cells[4];
        float w[4];
        sample_texel(g, g.step + 1u, (uint32_t)(valid ? e >> 4 : 0), x, y);
        bilinear_taps(g, gi, x, y, cells, w);
        const int c01 = tap & 1 ? cells[1] : cells[0], c23 = tap & 1 ? cells[3] : cells[2];
        const uint32_t cell = (uint32_t)(tap & 2 ? c23 : c01) + (gi ? (uint32_t)(g.gw[0] * g.gh[0]) : 0u);
        const size_t q = 2 * (size_t)cell + (sub & 1);
        uint32_t old = seen;
        if (valid && !(sub & 1)) old = atomicMax(a.seen + cell, seen);
        old = __shfl_sync(FULL, old, (int)(threadIdx.x & 30));
        const bool mine = old < seen;
        uint32_t t = max(old, a.base + 1u) - 1u - a.base;  // the first step to take
        const bool late = mine && t == j;
        float4 p, m, v;
        if (mine) {
            p = __ldcg(P + q);
            m = __ldcg(M + q);
            v = __ldcg(V + q);
        }
        if (__any_sync(FULL, late) && !waited) {
            grid_wait();  // the gradients of step j
            waited = true;
        }
        if (mine) {
            const longlong2 g0 = __ldcg(G + 2 * q), g1 = __ldcg(G + 2 * q + 1);
            adam_quad(a, a.st[t], p, m, v, g0, g1);
#pragma unroll 1
            while (++t <= j) adam_quad(a, a.st[t], p, m, v, z, z);
            P[q] = p;
            M[q] = m;
            V[q] = v;
            if (g0.x | g0.y | g1.x | g1.y) {
                G[2 * q] = z;
                G[2 * q + 1] = z;
            }
        }
    }
    grid_wait();
    grid_trigger();
    update_weights(a, a.st[a.j], (int)blockIdx.x, (int)gridDim.x);
}

// The segment's end, after the gradients of its last step j: every cell takes
// the steps it has missed, and the weights step j.  Bound by the instructions
// of the updates in long segments (94 us for 10.5 million parameters and 16
// steps at 85% of the issue slots; 42 us would be the 24 bytes of each), by
// those bytes in short ones, whose cells are walked up and down in turn so that
// a sweep starts with the cells that the last one left in L2 (4096^2 texture,
// 8,192 texels, calls of one step: 78 us a step with one direction, 66 with
// both).  Five or more CTAs per SM are slower by 3%.
constexpr int kSweepThreads = 256, kSweepCtasPerSm = 4;
__global__ void __launch_bounds__(kSweepThreads, kSweepCtasPerSm) sweep_kernel(const AdamParams a) {
    static_assert(kSweepThreads == kRedEntries * kRedRows, "the weight sums' thread layout");
    float4 *__restrict__ P = reinterpret_cast<float4 *>(a.params + kOffLat);
    float4 *__restrict__ M = reinterpret_cast<float4 *>(a.m + kOffLat);
    float4 *__restrict__ V = reinterpret_cast<float4 *>(a.v + kOffLat);
    longlong2 *__restrict__ G = reinterpret_cast<longlong2 *>(a.grad + kOffLat);
    const size_t nq = (a.n - kOffLat) / 4, stride = (size_t)gridDim.x * kSweepThreads;
    const uint32_t j = (uint32_t)a.j;
    const longlong2 z = make_longlong2(0, 0);
    size_t i = blockIdx.x * (size_t)kSweepThreads + threadIdx.x;
    auto quad_at = [&](size_t k) {  // (past the end: the last quad again, not used)
        const size_t c = min(k, nq - 1);
        return a.descending ? nq - 1 - c : c;
    };
    // parameters and moments do not change before the wait (of the cells that
    // step j reads, neither does `seen`, but in a segment's first step); the
    // update before is over by now, as in advance_kernel
    size_t q = quad_at(i);
    float4 p = __ldcg(P + q), m = __ldcg(M + q), v = __ldcg(V + q);
    grid_wait();
    grid_trigger();
    uint32_t old = __ldcg(a.seen + (q >> 1));
    update_weights(a, a.st[j], (int)blockIdx.x, (int)gridDim.x);
    for (; i < nq; i += stride) {
        const size_t qn = quad_at(i + stride);
        const uint32_t oldn = __ldcg(a.seen + (qn >> 1));
        const float4 pn = __ldcg(P + qn), mn = __ldcg(M + qn), vn = __ldcg(V + qn);
        uint32_t t = 0;
        longlong2 g0 = z, g1 = z;
        if (old > a.base) {
            t = old - 1u - a.base;
            g0 = __ldcg(G + 2 * q);
            g1 = __ldcg(G + 2 * q + 1);
        }
        adam_quad(a, a.st[t], p, m, v, g0, g1);
#pragma unroll 1
        while (++t <= j) adam_quad(a, a.st[t], p, m, v, z, z);
        P[q] = p;
        M[q] = m;
        V[q] = v;
        if (g0.x | g0.y | g1.x | g1.y) {
            G[2 * q] = z;
            G[2 * q + 1] = z;
        }
        q = qn;
        old = oldn;
        p = pn;
        m = mn;
        v = vn;
    }
}

__global__ void init_kernel(float *params, size_t n, uint32_t k0, uint32_t k1) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const uint4 r = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)(i >> 32), 0x1A17u, 0u), k0, k1);
        const float u0 = ((float)(r.x >> 8) + 0.5f) * 5.9604644775390625e-08f;
        const float u1 = ((float)(r.y >> 8) + 0.5f) * 5.9604644775390625e-08f;
        float v = 0.f;
        if (i < (size_t)kOffB1) v = (2.f * u0 - 1.f) * sqrtf(6.f / 16.f);
        else if (i >= (size_t)kOffW2 && i < (size_t)kOffB2) v = (2.f * u0 - 1.f) * sqrtf(6.f / 64.f);
        else if (i >= (size_t)kOffW3 && i < (size_t)kOffB3) v = (2.f * u0 - 1.f) * sqrtf(6.f / 64.f);
        else if (i >= (size_t)kOffB3 && i < (size_t)kWeights) v = 0.5f;
        else if (i >= (size_t)kOffLat) v = 0.5f * sqrtf(-2.f * logf(u0)) * cospif(2.f * u1);
        params[i] = v;
    }
}

// Largest |input| of each layer per input channel over every texel (FP8
// scales).  Values are non-negative, so their bit patterns order like ints.
__global__ void __launch_bounds__(kThreads) actstats_kernel(const GradParams g, unsigned *amax) {
    __shared__ float W[kWeights];
    __shared__ unsigned smax[144];
    for (int i = threadIdx.x; i < kWeights; i += kThreads) W[i] = g.params[i];
    for (int i = threadIdx.x; i < 144; i += kThreads) smax[i] = 0u;
    __syncthreads();
    const float *lat[2] = {g.params + kOffLat, g.params + kOffLat + (size_t)g.gw[0] * g.gh[0] * 8};
    const long long total = (long long)g.Wt * g.Ht;
    for (long long t = blockIdx.x * (long long)kThreads + threadIdx.x; t < total; t += (long long)gridDim.x * kThreads) {
        const int x = (int)(t % g.Wt), y = (int)(t / g.Wt);
        float f[16];
#pragma unroll
        for (int gi = 0; gi < 2; ++gi) {
            int tap[4];
            float tw[4];
            bilinear_taps(g, gi, x, y, tap, tw);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                float acc = 0.f;
#pragma unroll
                for (int k = 0; k < 4; ++k) acc = __fmaf_rn(tw[k], __ldg(lat[gi] + (size_t)tap[k] * 8 + c), acc);
                f[gi * 8 + c] = acc;
            }
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) atomicMax(&smax[k], __float_as_uint(fabsf(f[k])));
        float h1[64];
#pragma unroll
        for (int j = 0; j < 64; ++j) {
            float a = W[kOffB1 + j];
#pragma unroll
            for (int k = 0; k < 16; ++k) a = __fmaf_rn(W[kOffW1 + j * 16 + k], f[k], a);
            h1[j] = fmaxf(a, 0.f);
            atomicMax(&smax[16 + j], __float_as_uint(h1[j]));
        }
        for (int j = 0; j < 64; ++j) {
            float a = W[kOffB2 + j];
#pragma unroll
            for (int k = 0; k < 64; ++k) a = __fmaf_rn(W[kOffW2 + j * 64 + k], h1[k], a);
            atomicMax(&smax[80 + j], __float_as_uint(fmaxf(a, 0.f)));
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 144; i += kThreads) atomicMax(amax + i, smax[i]);
}

// Squared RGB error and largest channel error of a learned texture's decoded
// texels against the exact decode, for texels [start, start + n).
__global__ void compare_kernel(const uint2 *blocks, int nbx, int Wt, int Ht, const float4 *dec, long long start, int n,
                               double *sse, unsigned *maxabs) {
    double acc = 0.0;
    float mx = 0.f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const long long t = start + i;
        const int x = (int)(t % Wt), y = (int)(t / Wt);
        const uint32_t px = fetch_block_texel(blocks, nbx, Wt, Ht, x, y);
        const float4 d = dec[i];
        const float e0 = d.x - __fdiv_rn((float)(px & 0xffu), 255.f);
        const float e1 = d.y - __fdiv_rn((float)((px >> 8) & 0xffu), 255.f);
        const float e2 = d.z - __fdiv_rn((float)((px >> 16) & 0xffu), 255.f);
        const float e3 = d.w - __fdiv_rn((float)(px >> 24), 255.f);
        acc += (double)e0 * e0 + (double)e1 * e1 + (double)e2 * e2;
        mx = fmaxf(mx, fmaxf(fmaxf(fabsf(e0), fabsf(e1)), fmaxf(fabsf(e2), fabsf(e3))));
    }
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(FULL, acc, o);
        mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(sse, acc);
        atomicMax(maxabs, __float_as_uint(mx));
    }
}

__global__ void linear_xy_kernel(int2 *xy, long long start, int n, int Wt) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const long long t = start + i;
        xy[i] = make_int2((int)(t % Wt), (int)(t / Wt));
    }
}

}  // namespace
}  // namespace ctf

struct ctf_trainer_s {
    ctf_texture src = nullptr;
    ctf_train_desc desc{};
    int Wt = 0, Ht = 0;
    size_t n_lat[2] = {0, 0};
    size_t nparams = 0;
    float *params = nullptr, *m = nullptr, *v = nullptr;
    long long *grad = nullptr, *loss = nullptr;
    uint32_t *seen = nullptr;       // per latent cell, see advance_kernel
    uint32_t seen_steps = 0;        // the steps that `seen` counts (all of them, but for an overflow)
    unsigned char *wimg = nullptr;  // FP16 weight operands of the gradient kernel
    float *partial = nullptr;       // per-CTA weight-gradient sums of the gradient kernel
    int64_t step = 0;
    uint32_t sweeps = 0;            // sweeps so far: every other one walks down
    // a segment that a refused launch cut short (finish_segment): its step whose
    // launches are not all queued, or -1; whether the gradients are; its base
    int open = -1;
    bool open_grad = false;
    uint32_t open_base = 0;
};

namespace ctf {
namespace {

GradParams grad_params(const ctf_trainer_s *t) {
    GradParams g;
    g.params = t->params;
    g.blocks = static_cast<const uint2 *>(t->src->blocks);
    g.Wt = t->Wt;
    g.Ht = t->Ht;
    g.nbx = t->Wt / 4;
    for (int i = 0; i < 2; ++i) {
        g.gw[i] = t->desc.latent_w[i];
        g.gh[i] = t->desc.latent_h[i];
        g.sx[i] = (float)g.gw[i] / (float)t->Wt;
        g.sy[i] = (float)g.gh[i] / (float)t->Ht;
    }
    g.xy = nullptr;
    g.n = 0;
    g.rounds = 1;
    g.step = 0;
    g.k0 = (uint32_t)(t->desc.seed & 0xffffffffu);
    g.k1 = (uint32_t)(t->desc.seed >> 32);
    g.dscale = 0.f;
    g.grad = t->grad;
    g.seen = t->seen;
    g.mark = 0;
    g.loss = t->loss;
    g.per_round = kT;
    g.wimg = t->wimg;
    g.partial = t->partial;
    g.err = nullptr;
    device_error_word(&g.err);  // a static device word: no allocation; nullptr if it cannot be had
    return g;
}

// The split of a batch over the gradient kernel's CTAs.  Two CTAs fit on an
// SM (TMEM and shared memory).  Small batches take 64 texels per round (the
// other 64 rows of the MMAs stay empty) so that more SMs have work; a CTA's
// fixed costs (weights in, sums out) favour a few rounds each once there are
// 256 CTAs, and at most kMaxGradCtas CTAs hold partial sums.  The split
// depends on the batch alone, so a step gives the same sums on any device.
int split_batch(GradParams &g) {
    g.per_round = g.n >= 32768 ? kT : kT / 2;
    int rounds = g.n / (g.per_round * 256);
    rounds = rounds < 1 ? 1 : (rounds > kMaxRounds ? kMaxRounds : rounds);
    const int need = (g.n + g.per_round * kMaxGradCtas - 1) / (g.per_round * kMaxGradCtas);
    g.rounds = rounds > need ? rounds : need;
    return (g.n + g.per_round * g.rounds - 1) / (g.per_round * g.rounds);
}

// The gradient kernel, after a kernel that left the weight image.
cudaError_t launch_grad(const GradParams &g, int ctas, cudaStream_t s) {
    static std::mutex mu;
    static bool attr[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    {
        std::lock_guard<std::mutex> lk(mu);
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        if (!attr[dev]) {
            cudaError_t e = cudaFuncSetAttribute(grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradSmem);
            if (e != cudaSuccess) return e;
            attr[dev] = true;
        }
    }
    return launch_dependent(grad_kernel, ctas, kT, kGradSmem, s, g);
}

cudaError_t launch_pack(const GradParams &g, cudaStream_t s) {
    return launch_plain(pack_kernel, (kPackThreads + 255) / 256, 256, 0, s, g.params, g.wimg);
}

// A step's gradients, and their split over CTAs.
GradParams step_grad_params(const ctf_trainer_s *t, int &ctas) {
    GradParams g = grad_params(t);
    g.n = t->desc.batch;
    g.dscale = 2.0f / (float)t->desc.batch;
    ctas = split_batch(g);
    return g;
}

AdamParams adam_params(const ctf_trainer_s *t, const GradParams &g, int ctas) {
    AdamParams a;
    a.params = t->params;
    a.m = t->m;
    a.v = t->v;
    a.grad = t->grad;
    a.n = t->nparams;
    a.beta1 = t->desc.beta1;
    a.beta2 = t->desc.beta2;
    a.eps = t->desc.eps;
    a.partial = t->partial;
    a.ctas = ctas;
    a.dscale = (double)g.dscale;
    a.wimg = t->wimg;
    a.seen = t->seen;
    return a;
}

AdamStep adam_step(const ctf_trainer_s *t, int64_t st) {
    const double frac = std::fmin(1.0, (double)st / (double)t->desc.total_steps);
    const double sched = 1.0 - (1.0 - t->desc.lr_final_frac) * frac;
    const double bc1 = 1.0 - std::pow((double)t->desc.beta1, (double)(st + 1));
    const double bc2 = 1.0 - std::pow((double)t->desc.beta2, (double)(st + 1));
    AdamStep r;
    r.w = (float)(t->desc.lr_weights * sched / bc1);
    r.lat = (float)(t->desc.lr_latents * sched / bc1);
    r.inv_bc2 = (float)(1.0 / bc2);
    return r;
}

// A launch refused inside a segment leaves the weights and some cells steps
// ahead of the others.  Every call that reads or changes the trainer first ends
// such a segment with the step that was refused: its gradients, if they are
// not queued yet, and a sweep.  The steps count from then on.  If that is refused
// too, the trainer stays as it was.
int finish_segment(ctf_trainer_s *t, cudaStream_t s) {
    if (t->open < 0) return CTF_OK;
    int ctas = 0;
    GradParams g = step_grad_params(t, ctas);
    AdamParams a = adam_params(t, g, ctas);
    a.base = t->open_base;
    a.j = t->open;
    for (int j = 0; j <= t->open; ++j) a.st[j] = adam_step(t, t->step + j);
    a.descending = (int)(t->sweeps & 1u);
    g.step = (uint32_t)(t->step + t->open);
    cudaError_t e = cudaSuccess;
    if (!t->open_grad) {  // (after a plain launch, so after everything before it)
        e = launch_pack(g, s);
        if (e == cudaSuccess) e = launch_grad(g, ctas, s);
        t->open_grad = e == cudaSuccess;
    }
    if (e == cudaSuccess)
        e = launch_plain(sweep_kernel, device_sm_count() * kSweepCtasPerSm, kSweepThreads, 0, s, a);
    if (e != cudaSuccess) return report_cuda(e, "finishing a training segment");
    ++t->sweeps;
    t->step += t->open + 1;
    t->seen_steps = t->open_base + (uint32_t)t->open + 1;
    t->open = -1;
    return CTF_OK;
}

int check_desc(const ctf_train_desc *d) {
    if (!d) return report(CTF_ERR_ARG, "desc is NULL");
    for (int g = 0; g < 2; ++g)
        if (d->latent_w[g] < 1 || d->latent_h[g] < 1 || d->latent_w[g] > 16384 || d->latent_h[g] > 16384)
            return report(CTF_ERR_ARG, "latent grid %d is %dx%d", g, d->latent_w[g], d->latent_h[g]);
    if (d->batch < 1 || d->batch > 4194304) return report(CTF_ERR_ARG, "batch %d outside [1, 4194304]", d->batch);
    if (d->total_steps < 1) return report(CTF_ERR_ARG, "total_steps must be positive");
    if (!(d->lr_weights > 0.f) || !(d->lr_latents > 0.f) || !(d->lr_final_frac >= 0.f) || !(d->beta1 >= 0.f) ||
        !(d->beta1 < 1.f) || !(d->beta2 >= 0.f) || !(d->beta2 < 1.f) || !(d->eps > 0.f))
        return report(CTF_ERR_ARG, "learning rates / Adam constants out of range");
    return CTF_OK;
}

void free_trainer(ctf_trainer_s *t) {
    if (!t) return;
    ctf::dev_free(t->params);
    ctf::dev_free(t->m);
    ctf::dev_free(t->v);
    ctf::dev_free(t->grad);
    ctf::dev_free(t->seen);
    ctf::dev_free(t->loss);
    ctf::dev_free(t->wimg);
    ctf::dev_free(t->partial);
    delete t;
}

int alloc_trainer(ctf_texture src, const ctf_train_desc *d, ctf_trainer_s **out) {
    if (!src || src->mode != CTF_EVAL_BLOCK) return report(CTF_ERR_ARG, "the source must be an exact block texture");
    int rc = check_desc(d);
    if (rc) return rc;
    ctf_trainer_s *t = new (std::nothrow) ctf_trainer_s();
    if (!t) return report(CTF_ERR_OOM, "host allocation");
    t->src = src;
    t->desc = *d;
    t->Wt = src->width;
    t->Ht = src->height;
    for (int g = 0; g < 2; ++g) t->n_lat[g] = (size_t)d->latent_w[g] * d->latent_h[g] * 8;
    t->nparams = kOffLat + t->n_lat[0] + t->n_lat[1];
    cudaError_t e = ctf::dev_malloc(&t->params, t->nparams * 4);
    if (e == cudaSuccess) e = ctf::dev_malloc(&t->seen, (t->nparams - kOffLat) / 8 * 4);
    if (e == cudaSuccess) e = ctf::dev_malloc(&t->m, t->nparams * 4);
    if (e == cudaSuccess) e = ctf::dev_malloc(&t->v, t->nparams * 4);
    if (e == cudaSuccess) e = ctf::dev_malloc(&t->grad, t->nparams * 8);
    if (e == cudaSuccess) e = ctf::dev_malloc(&t->loss, 8);
    if (e == cudaSuccess) e = ctf::dev_malloc(&t->wimg, kGAH);
    if (e == cudaSuccess) e = ctf::dev_malloc(&t->partial, (size_t)kMaxGradCtas * kWeights * 4);
    if (e == cudaSuccess) e = cudaMemset(t->m, 0, t->nparams * 4);
    if (e == cudaSuccess) e = cudaMemset(t->v, 0, t->nparams * 4);
    if (e == cudaSuccess) e = cudaMemset(t->grad, 0, t->nparams * 8);
    if (e == cudaSuccess) e = cudaMemset(t->params, 0, t->nparams * 4);
    if (e == cudaSuccess) e = cudaMemset(t->loss, 0, 8);
    if (e == cudaSuccess) e = cudaMemset(t->seen, 0, (t->nparams - kOffLat) / 8 * 4);
    if (e != cudaSuccess) {
        free_trainer(t);
        return report_cuda(e, "trainer allocation");
    }
    *out = t;
    return CTF_OK;
}

// Array order of ctf_mlp_arrays and their offsets / sizes in the parameter buffer.
void layout(const ctf_trainer_s *t, size_t off[8], size_t cnt[8]) {
    const size_t o[8] = {kOffLat, kOffLat + t->n_lat[0], kOffW1, kOffB1, kOffW2, kOffB2, kOffW3, kOffB3};
    const size_t c[8] = {t->n_lat[0], t->n_lat[1], 1024, 64, 4096, 64, 256, 4};
    for (int i = 0; i < 8; ++i) {
        off[i] = o[i];
        cnt[i] = c[i];
    }
}

void arrays_of(const ctf_mlp_arrays *a, float *p[8]) {
    p[0] = a->latent[0];
    p[1] = a->latent[1];
    p[2] = a->w1;
    p[3] = a->b1;
    p[4] = a->w2;
    p[5] = a->b2;
    p[6] = a->w3;
    p[7] = a->b3;
}

constexpr char kMagic[8] = {'C', 'T', 'F', 'T', 'R', 'N', '0', '1'};
constexpr uint32_t kVersion = 1;

}  // namespace
}  // namespace ctf

extern "C" {

int ctf_trainer_create(ctf_texture exact_src, const ctf_train_desc *desc, ctf_trainer *out) {
    using namespace ctf;
    clear_error();
    if (!out) return report(CTF_ERR_ARG, "out is NULL");
    *out = nullptr;
    ctf_trainer_s *t = nullptr;
    int rc = alloc_trainer(exact_src, desc, &t);
    if (rc) return rc;
    cudaError_t e = launch_plain(init_kernel, 1024, 256, 0, nullptr, t->params, t->nparams,
                                 (uint32_t)(desc->seed & 0xffffffffu), (uint32_t)(desc->seed >> 32));
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        free_trainer(t);
        return report_cuda(e, "parameter initialisation");
    }
    *out = t;
    return CTF_OK;
}

int ctf_trainer_destroy(ctf_trainer t) {
    ctf::clear_error();
    if (!t) return CTF_OK;
    cudaDeviceSynchronize();
    ctf::free_trainer(t);
    return CTF_OK;
}

int64_t ctf_trainer_steps_done(ctf_trainer t) { return t ? t->step : -1; }

int ctf_trainer_step(ctf_trainer t, int64_t steps, void *stream) {
    ctf::NvtxRange nvtx_range("ctf_trainer_step");
    using namespace ctf;
    clear_error();
    if (!t) return report(CTF_ERR_ARG, "trainer is NULL");
    if (steps < 0) return report(CTF_ERR_ARG, "negative step count");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int ctas = 0;
    GradParams g = step_grad_params(t, ctas);
    AdamParams a = adam_params(t, g, ctas);
    // A captured call runs whenever its graph does, after other replays and
    // calls: its segments count from zero in cells that it clears itself.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    uint32_t seen_steps = t->seen_steps;
    if (steps > 0) {
        cudaError_t e = cudaStreamIsCapturing(s, &capture);
        if (e != cudaSuccess) cudaGetLastError();
        if (e == cudaSuccess && capture != cudaStreamCaptureStatusNone) {
            if (t->open >= 0)
                return report(CTF_ERR_UNSUPPORTED, "steps cut short by a refused launch are finished outside a capture");
            seen_steps = 0;
            e = cudaMemsetAsync(t->seen, 0, (t->nparams - kOffLat) / 8 * 4, s);
        }
        if (e == cudaSuccess && t->open >= 0) {
            const int rc = finish_segment(t, s);
            if (rc) return rc;
            seen_steps = t->seen_steps;
        }
        if (e == cudaSuccess) e = launch_pack(g, s);
        if (e != cudaSuccess) return report_cuda(e, "training step");
    }
    // Segments of equal length, to one step; of one step where a step's texels
    // reach more cells (eight each) than there are, since nothing stands still
    // then: 4096^2 with 262,144 texels 281 us a step against 302 in segments,
    // 2048^2 with 65,536 63 against 66; below the line, 4096^2 with 65,536
    // texels, 124 against 105.
    const int sms = device_sm_count();
    const int64_t longest = 64ll * g.n > (int64_t)(t->nparams - kOffLat) ? 1 : kSegment;
    for (int64_t left = (steps + longest - 1) / longest, k = 0; k < steps; --left) {
        const int len = (int)((steps - k + left - 1) / left);
        a.base = seen_steps;
        for (int j = 0; j < len; ++j) a.st[j] = adam_step(t, t->step + j);
        cudaError_t e = cudaSuccess;
        if (a.base > 0xffffff00u) {
            e = cudaMemsetAsync(t->seen, 0, (t->nparams - kOffLat) / 8 * 4, s);
            a.base = 0;
        }
        for (int j = 0; j < len && e == cudaSuccess; ++j) {
            g.step = (uint32_t)(t->step + j);
            g.mark = j == 0 ? a.base + 1u : 0u;
            a.j = j;
            e = launch_grad(g, ctas, s);
            const bool grad = e == cudaSuccess;
            if (grad && j + 1 < len) {
                const long long need = (16ll * g.n + kAdvThreads - 1) / kAdvThreads, cap = 8ll * sms * kAdvCtasPerSm;
                const long long grid = std::max<long long>(std::min(need, cap), (kWeights + kRedEntries - 1) / kRedEntries);
                e = launch_dependent(advance_kernel, (int)grid, kAdvThreads, 0, s, g, a);
            } else if (grad) {
                a.descending = (int)(t->sweeps & 1u);
                e = launch_dependent(sweep_kernel, sms * kSweepCtasPerSm, kSweepThreads, 0, s, a);
                if (e == cudaSuccess) ++t->sweeps;
            }
            // (of a capture that fails nothing will run)
            if (e != cudaSuccess && (grad || j > 0) && capture == cudaStreamCaptureStatusNone) {
                t->open = j;
                t->open_grad = grad;
                t->open_base = a.base;
            }
        }
        if (e != cudaSuccess) return report_cuda(e, "training step");
        t->step += len;
        seen_steps = a.base + (uint32_t)len;
        // (the marks that a captured call leaves lie below either count)
        t->seen_steps = capture == cudaStreamCaptureStatusNone ? seen_steps : std::max(t->seen_steps, seen_steps);
        k += len;
    }
    return CTF_OK;
}

int ctf_trainer_gradients(ctf_trainer t, const int32_t *xy, int n, double *loss, const ctf_mlp_arrays *grads,
                          void *stream) {
    using namespace ctf;
    clear_error();
    if (!t) return report(CTF_ERR_ARG, "trainer is NULL");
    if (n < 1 || !xy) return report(CTF_ERR_ARG, "need n >= 1 texels");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int rc = finish_segment(t, s);
    if (rc) return rc;
    GradParams g = grad_params(t);
    g.xy = reinterpret_cast<const int2 *>(xy);
    g.n = n;
    g.dscale = 2.0f / (float)n;
    // the accumulators are zero between steps; use them and clear them again
    const int ctas = split_batch(g);
    cudaError_t e = cudaMemsetAsync(t->loss, 0, 8, s);
    if (e == cudaSuccess) e = launch_pack(g, s);
    if (e == cudaSuccess) e = launch_grad(g, ctas, s);
    if (e == cudaSuccess) {
        e = launch_plain(reduce_kernel, (kWeights + kRedEntries - 1) / kRedEntries, kRedEntries * kRedRows, 0, s,
                         g.partial, ctas, (double)g.dscale, g.grad);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return report_cuda(e, "gradient kernel");
    std::vector<long long> h(t->nparams);
    long long hl = 0;
    e = cudaMemcpy(h.data(), t->grad, t->nparams * 8, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&hl, t->loss, 8, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemset(t->grad, 0, t->nparams * 8);
    if (e != cudaSuccess) return report_cuda(e, "reading gradients");
    if (loss) *loss = (double)hl / kLossFix / (double)n;
    if (grads) {
        size_t off[8], cnt[8];
        float *p[8];
        layout(t, off, cnt);
        arrays_of(grads, p);
        for (int i = 0; i < 8; ++i)
            if (p[i])
                for (size_t k = 0; k < cnt[i]; ++k) p[i][k] = (float)((double)h[off[i] + k] / kFix);
    }
    return CTF_OK;
}

int ctf_trainer_get_params(ctf_trainer t, const ctf_mlp_arrays *out) {
    using namespace ctf;
    clear_error();
    if (!t || !out) return report(CTF_ERR_ARG, "trainer and out must not be NULL");
    size_t off[8], cnt[8];
    float *p[8];
    layout(t, off, cnt);
    arrays_of(out, p);
    cudaDeviceSynchronize();
    const int rc = finish_segment(t, nullptr);
    if (rc) return rc;
    for (int i = 0; i < 8; ++i)
        if (p[i]) {
            cudaError_t e = cudaMemcpy(p[i], t->params + off[i], cnt[i] * 4, cudaMemcpyDefault);
            if (e != cudaSuccess) return report_cuda(e, "copying parameters out");
        }
    return CTF_OK;
}

int ctf_trainer_set_params(ctf_trainer t, const ctf_mlp_arrays *in) {
    using namespace ctf;
    clear_error();
    if (!t || !in) return report(CTF_ERR_ARG, "trainer and in must not be NULL");
    size_t off[8], cnt[8];
    float *p[8];
    layout(t, off, cnt);
    arrays_of(in, p);
    cudaDeviceSynchronize();
    const int rc = finish_segment(t, nullptr);
    if (rc) return rc;
    for (int i = 0; i < 8; ++i)
        if (p[i]) {
            cudaError_t e = cudaMemcpy(t->params + off[i], p[i], cnt[i] * 4, cudaMemcpyDefault);
            if (e != cudaSuccess) return report_cuda(e, "copying parameters in");
        }
    return CTF_OK;
}

int ctf_trainer_export(ctf_trainer t, ctf_eval_mode mode, ctf_texture *out) {
    using namespace ctf;
    clear_error();
    if (!t || !out) return report(CTF_ERR_ARG, "trainer and out must not be NULL");
    if (t->open >= 0) {
        cudaDeviceSynchronize();
        const int rc = finish_segment(t, nullptr);
        if (rc) return rc;
    }
    ctf_mlp_desc d;
    std::memset(&d, 0, sizeof(d));
    d.width = t->Wt;
    d.height = t->Ht;
    d.mode = mode;
    for (int g = 0; g < 2; ++g) {
        d.latent_w[g] = t->desc.latent_w[g];
        d.latent_h[g] = t->desc.latent_h[g];
    }
    d.latent[0] = t->params + kOffLat;
    d.latent[1] = t->params + kOffLat + t->n_lat[0];
    d.w1 = t->params + kOffW1;
    d.b1 = t->params + kOffB1;
    d.w2 = t->params + kOffW2;
    d.b2 = t->params + kOffB2;
    d.w3 = t->params + kOffW3;
    d.b3 = t->params + kOffB3;
    std::vector<float> amax(144, 0.f);
    if (mode == CTF_EVAL_MLP_FP8) {
        unsigned *dmax = nullptr;
        cudaError_t e = ctf::dev_malloc(&dmax, 144 * 4);
        if (e == cudaSuccess) e = cudaMemset(dmax, 0, 144 * 4);
        if (e == cudaSuccess) {
            GradParams g = grad_params(t);
            e = launch_plain(actstats_kernel, device_sm_count() * 4, kThreads, 0, nullptr, g, dmax);
        }
        if (e == cudaSuccess) e = cudaMemcpy(amax.data(), dmax, 144 * 4, cudaMemcpyDeviceToHost);
        ctf::dev_free(dmax);
        if (e != cudaSuccess) return report_cuda(e, "activation statistics");
        d.act_absmax[0] = amax.data();
        d.act_absmax[1] = amax.data() + 16;
        d.act_absmax[2] = amax.data() + 80;
    } else {
        cudaDeviceSynchronize();
    }
    return ctf_texture_create_mlp(&d, out);
}

int ctf_trainer_save(ctf_trainer t, const char *path) {
    using namespace ctf;
    clear_error();
    if (!t || !path) return report(CTF_ERR_ARG, "trainer and path must not be NULL");
    cudaDeviceSynchronize();
    const int rc = finish_segment(t, nullptr);
    if (rc) return rc;
    std::vector<float> buf(3 * t->nparams);
    cudaError_t e = cudaMemcpy(buf.data(), t->params, t->nparams * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(buf.data() + t->nparams, t->m, t->nparams * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(buf.data() + 2 * t->nparams, t->v, t->nparams * 4, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return report_cuda(e, "reading the training state");
    FILE *f = std::fopen(path, "wb");
    if (!f) return report(CTF_ERR_ARG, "cannot open %s for writing", path);
    uint64_t h = 1469598103934665603ull;
    const uint32_t ver = kVersion;
    const int32_t dims[6] = {t->Wt, t->Ht, t->desc.latent_w[0], t->desc.latent_h[0], t->desc.latent_w[1],
                             t->desc.latent_h[1]};
    const uint64_t np = t->nparams;
    const int64_t step = t->step;
    bool ok = true;
    auto put = [&](const void *p, size_t n) {
        ok = ok && std::fwrite(p, 1, n, f) == n;
        h = fnv1a(p, n, h);
    };
    put(kMagic, 8);
    put(&ver, 4);
    put(dims, sizeof(dims));
    put(&np, 8);
    put(&step, 8);
    put(&t->desc, sizeof(t->desc));
    put(buf.data(), buf.size() * 4);
    ok = ok && std::fwrite(&h, 1, 8, f) == 8;
    ok = (std::fclose(f) == 0) && ok;
    if (!ok) return report(CTF_ERR_ARG, "writing %s failed", path);
    return CTF_OK;
}

int ctf_trainer_load(ctf_texture exact_src, const char *path, ctf_trainer *out) {
    using namespace ctf;
    clear_error();
    if (!out || !path) return report(CTF_ERR_ARG, "path and out must not be NULL");
    *out = nullptr;
    FILE *f = std::fopen(path, "rb");
    if (!f) return report(CTF_ERR_ARG, "cannot open %s", path);
    std::vector<unsigned char> all;
    unsigned char tmp[65536];
    size_t k;
    while ((k = std::fread(tmp, 1, sizeof(tmp), f)) > 0) all.insert(all.end(), tmp, tmp + k);
    std::fclose(f);
    const size_t head = 8 + 4 + 24 + 8 + 8 + sizeof(ctf_train_desc);
    if (all.size() < head + 8 || std::memcmp(all.data(), kMagic, 8) != 0)
        return report(CTF_ERR_CORRUPT, "%s is not a training checkpoint", path);
    uint64_t stored = 0;
    std::memcpy(&stored, all.data() + all.size() - 8, 8);
    if (fnv1a(all.data(), all.size() - 8, 1469598103934665603ull) != stored)
        return report(CTF_ERR_CORRUPT, "checksum mismatch in %s", path);
    uint32_t ver;
    int32_t dims[6];
    uint64_t np;
    int64_t step;
    ctf_train_desc d;
    const unsigned char *p = all.data() + 8;
    std::memcpy(&ver, p, 4);
    p += 4;
    std::memcpy(dims, p, 24);
    p += 24;
    std::memcpy(&np, p, 8);
    p += 8;
    std::memcpy(&step, p, 8);
    p += 8;
    std::memcpy(&d, p, sizeof(d));
    p += sizeof(d);
    if (ver != kVersion) return report(CTF_ERR_CORRUPT, "checkpoint version %u, expected %u", ver, kVersion);
    if (!exact_src || exact_src->width != dims[0] || exact_src->height != dims[1])
        return report(CTF_ERR_CORRUPT, "checkpoint is for a %dx%d texture", dims[0], dims[1]);
    ctf_trainer_s *t = nullptr;
    int rc = alloc_trainer(exact_src, &d, &t);
    if (rc) return rc;
    if (t->nparams != np || all.size() != head + 12 * np + 8) {
        free_trainer(t);
        return report(CTF_ERR_CORRUPT, "checkpoint sizes do not match its description");
    }
    const float *fp = reinterpret_cast<const float *>(p);
    cudaError_t e = cudaMemcpy(t->params, fp, np * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(t->m, fp + np, np * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(t->v, fp + 2 * np, np * 4, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        free_trainer(t);
        return report_cuda(e, "uploading the training state");
    }
    t->step = step;
    *out = t;
    return CTF_OK;
}

int ctf_texture_compare(ctf_texture ref, ctf_texture learned, double *mse_rgb, double *max_abs, void *stream) {
    using namespace ctf;
    clear_error();
    if (!ref || !learned || ref->mode != CTF_EVAL_BLOCK || learned->mode == CTF_EVAL_BLOCK)
        return report(CTF_ERR_ARG, "need an exact block texture and a learned-decode texture");
    if (ref->width != learned->width || ref->height != learned->height)
        return report(CTF_ERR_ARG, "texture sizes differ");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int *err = nullptr;
    int rc = device_error_word(&err);
    if (rc) return rc;
    const long long total = (long long)ref->width * ref->height;
    const int chunk = 1 << 22;
    int2 *xy = nullptr;
    float4 *dec = nullptr;
    double *sse = nullptr;
    unsigned *mx = nullptr;
    cudaError_t e = ctf::dev_malloc(&xy, (size_t)chunk * 8);
    if (e == cudaSuccess) e = ctf::dev_malloc(&dec, (size_t)chunk * 16);
    if (e == cudaSuccess) e = ctf::dev_malloc(&sse, 8);
    if (e == cudaSuccess) e = ctf::dev_malloc(&mx, 4);
    if (e == cudaSuccess) e = cudaMemsetAsync(sse, 0, 8, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(mx, 0, 4, s);
    const MlpDevice m = mlp_device_view(learned);
    for (long long st = 0; st < total && e == cudaSuccess; st += chunk) {
        const int n = (int)std::min<long long>(chunk, total - st);
        e = launch_plain(linear_xy_kernel, 1024, 256, 0, s, xy, st, n, ref->width);
        if (e == cudaSuccess) e = launch_mlp_decode(m, learned->epi, learned->width, learned->height, xy, n, dec, err, s);
        if (e == cudaSuccess) {
            e = launch_plain(compare_kernel, 1024, 256, 0, s, static_cast<const uint2 *>(ref->blocks), ref->width / 4,
                             ref->width, ref->height, dec, st, n, sse, mx);
        }
    }
    double h_sse = 0.0;
    unsigned h_mx = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h_sse, sse, 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h_mx, mx, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    ctf::dev_free(xy);
    ctf::dev_free(dec);
    ctf::dev_free(sse);
    ctf::dev_free(mx);
    if (e != cudaSuccess) return report_cuda(e, "texture comparison");
    if (mse_rgb) *mse_rgb = h_sse / (3.0 * (double)total);
    if (max_abs) {
        float f;
        std::memcpy(&f, &h_mx, 4);
        *max_abs = f;
    }
    return CTF_OK;
}

}  // extern "C"
