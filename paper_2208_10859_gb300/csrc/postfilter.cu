// postfilter.cu -- residual CNN post-filter on the decoded viewport's luma.
//
// The paper has no learned component; this network extends the decoder: it
// removes quantisation artefacts from the viewport's luma.  Five 3x3
// convolutions with zero padding: 1 -> 32 channels (ReLU), three 32 -> 32
// (ReLU), 32 -> 1; the output is the input luma plus that residual.  Weights
// are bf16 (fp32 master copies for training), activations bf16 between
// layers, every product accumulated in fp32 on the tensor cores.
//
// Convolutions are implicit GEMMs on tcgen05 (one elected thread issues the
// MMAs, operands in shared memory, accumulator in TMEM):
//   forward / input gradient: M = 128 pixels of one image row, N = 32 output
//     channels (16 for the last layer) of three output rows, K = 3 column taps
//     x 32 channels.  An input row lies in shared memory as 8-channel columns
//     of 130 pixels (16 bytes per pixel), so the A operand of column tap dx is
//     the row shifted by dx pixels: only the descriptor's start address
//     changes (SBO = 128 bytes, LBO = one column).  All layers run in one
//     kernel (k_net).
//   1 input channel: K = the 9 taps (padded to 16).
//   weight gradient, 32 -> 32: D[dy, ci][dx, co] = sum over pixels of
//     input[p + (dy, dx)][ci] * dZ[p][co]: M = (dy, ci), N = co, K = pixels,
//     one accumulator per dx, both operands read channel-major.
//   The input gradient of a layer is a forward convolution of the output
//   gradient with the spatially flipped, channel-transposed weights; the
//   ReLU of the layer below gates it in the epilogue.
// The weight gradients of the first and last layers (1 channel on one side,
// 1/32 of the work) run on CUDA cores.
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <initializer_list>
#include <new>
#include <vector>

#include "umma.h"
#include "wv_impl.h"

namespace wv {
namespace {

using bf16 = __nv_bfloat16;

constexpr int kC = 32;                  // channels of the hidden layers
constexpr int kLayers = 5;
constexpr int kTilePx = 128;            // pixels per MMA tile (M)
constexpr int kRowPx = kTilePx + 2;     // input pixels of one row slot (1-pixel halo)
constexpr int kLbo = kRowPx * 16;       // bytes between the 8-channel columns of a slot
constexpr int kSlot = 4 * kLbo;         // one input row: 4 columns of 8 channels
constexpr int kStep32 = 32 * 32;        // bytes of one K-step of a 32-row operand
constexpr int kBMid = 18 * kStep32;     // 32 x 288
constexpr int kBLast = 18 * 16 * 32;    // 16 x 288 (row 0 real)
constexpr int kBIn1 = kStep32;          // 32 x 16 (taps 0..8)

__host__ __device__ constexpr int layer_co(int l) { return l == kLayers - 1 ? 1 : kC; }
__host__ __device__ constexpr int layer_ci(int l) { return l == 0 ? 1 : kC; }
__host__ __device__ constexpr int off_w(int l) {
    int o = 0;
    for (int k = 0; k < l; ++k) o += layer_co(k) * layer_ci(k) * 9 + layer_co(k);
    return o;
}
__host__ __device__ constexpr int off_b(int l) { return off_w(l) + layer_co(l) * layer_ci(l) * 9; }
constexpr int kParams = off_w(kLayers);

// packed bf16 B operands: forward of layers 0..4, input gradient of 4..1
enum Pack { kPF0 = 0, kPF1 = kPF0 + kBIn1, kPF2 = kPF1 + kBMid, kPF3 = kPF2 + kBMid, kPF4 = kPF3 + kBMid,
            kPB4 = kPF4 + kBLast, kPB3 = kPB4 + kBIn1, kPB2 = kPB3 + kBMid, kPB1 = kPB2 + kBMid,
            kPackBytes = kPB1 + kBMid };

enum Mode { kTrain = 0, kOut = 1, kRgba = 2 };   // the last layer's epilogue

// ---- the chain of convolutions, fused --------------------------------------
//
// One CTA runs a chain of stages over a column tile of 128 pixels, row by
// row: stage 0 (one input channel: layer 0, or the input gradient of layer
// 4), three 32 -> 32 stages (layers 1-3, or their input gradients), and in the
// forward pass the last layer (32 -> 1).  The rows between the stages stay in
// shared memory; only the input plane, the output and, for training, the
// activations or gradients the weight gradients need touch HBM.  Each stage
// loses a pixel on either side, so a tile yields kTileOut = 120 columns, and
// a segment of S rows costs 2 T more rows in stage 0 (T stages after it).
//
// MMAs: an input row (A: 128 pixels x 32 channels, one 8-channel column per
// 16 bytes, shifted by dx pixels through the descriptor's start) takes part
// in three output rows.  Their accumulators are three 32-column TMEM slots
// (row index mod 3), all three updated by one MMA of N = 96 per K-step: B
// holds the weights of dy = 1, 0, 2, 1, 0 side by side, and a window of three
// starting at the right one fits any rotation of the slots.  So a row is 6
// MMAs instead of 18 and reads A a third as often, and each output sums its
// products in the same order (dy, dx, channel) as 18 would.  A drained slot is
// zeroed by its reader, so every MMA accumulates.
//
// Roles: per stage one warp that issues its MMAs and one warpgroup that reads
// its accumulator, applies bias and ReLU (or the ReLU gate of the backward
// pass) and writes the next stage's input row into a ring of kRings slots.
// (One warp issuing for all stages in turn took 3.2 us per row: a stage
// waited for the issue and the waits of the four others.)  Every wait is an
// mbarrier wait with a limit; one that gives up sets a flag that ends all
// roles.
//
// Bound: the MMAs, which take about one cycle per accumulator column here (by
// count of columns, 290 us of a 2160^2 plane's 306), and that is half the
// tensor pipe's rate: its counter shows 43 % active, with 54 % of the issue
// slots and 38 % of the shared-memory wavefronts used, and DRAM idle.  Why an
// MMA of N = 96 does not take half the cycles is not known.  Layer by layer,
// 2.4 GB of activations through HBM, the plane took 887 us.  Training adds 512 bytes a
// pixel of activations and gradients kept: 144 us forward and 155 us for the
// input gradients of 16 x 256^2 pixels (270 and 230 layer by layer).

constexpr int kTileOut = 120;           // output columns per tile
constexpr int kRings = 3;               // input rows in flight per stage
constexpr int kStages = 5;
// threads of a chain of T + 1 stages: a warpgroup and an issuing warp each
__host__ __device__ constexpr int net_threads(bool bwd) { return 32 * 5 * (bwd ? 4 : kStages); }
constexpr int kSeq = 5;                 // B blocks: dy = 1, 0, 2, 1, 0
constexpr int kBBlock = 4 * 256;        // 32 output channels x 16 K
constexpr int kBMidF = 6 * kSeq * kBBlock;
constexpr int kBLastF = 6 * kSeq * (kBBlock / 2);
constexpr int kA0 = 128 * 32;           // stage 0's operand: 128 pixels x 16 taps
constexpr int kWaitRound = 1 << 14, kWaitRounds = 64;   // polls between looks at the stop flag; default limit
constexpr int kNetRing = 4 * kRings * kSlot;
constexpr int kNetSmem = kNetRing + 3 * kBMidF + kBLastF + kBIn1 + 2 * kA0;

struct NetArgs {
    const float *in_plane;              // stage 0: one-channel input
    const uint8_t *pack[kStages];       // packed B operand of each stage
    const float *bias[kStages];         // forward
    const bf16 *gate[kStages];          // backward: ReLU outputs of the layer below (NHWC)
    bf16 *out[kStages];                 // NHWC outputs kept for the weight gradients, or null
    int n, h, w;
    int seg;                            // rows per segment
    int mode;                           // last layer's epilogue
    const float *x, *t;                 // last layer: input luma, target (kTrain)
    float *y;                           // output plane (kOut; kTrain: optional)
    float *dz;                          // kTrain: dL/dr plane
    float *loss;                        // kTrain: sum of squared errors
    float grad_scale;                   // kTrain: 2 / pixel count
    const uint8_t *cb, *cr;             // kRgba: chroma planes of the viewport
    uint8_t *rgba;
    size_t pitch;
    int *err;
    int wait_rounds;                    // rounds of kWaitRound polls before a wait gives up
};

struct NetBars {
    uint64_t in_full[kStages][kRings], in_free[kStages][kRings];   // stages 1..: input rows
    uint64_t acc_full[kStages], drained[kStages];
    uint64_t a0_full[2], acc0_full[2];
    uint64_t idle[kStages];   // every MMA the stage issued has completed
};

// Waits for the phase; false (and the flag set) when the limit is reached or
// another role has given up.
// LIMIT: the caller's limit (kernels of their own: read at run time it cost the
// forward pass 4 %), else the default.
template <bool LIMIT>
__device__ __forceinline__ bool net_wait(const NetArgs &a, uint64_t *bar, uint32_t parity, volatile int *stop) {
    for (int k = 0; k < (LIMIT ? a.wait_rounds : kWaitRounds); ++k) {
        if (umma::mbar_wait(bar, parity, kWaitRound)) return true;
        if (*stop) return false;
    }
    *stop = 1;
    return false;
}

// The same for a whole warp, with one answer for all its lanes.
template <bool LIMIT>
__device__ __forceinline__ bool net_wait_warp(const NetArgs &a, uint64_t *bar, uint32_t parity, volatile int *stop) {
    return __all_sync(0xffffffffu, net_wait<LIMIT>(a, bar, parity, stop));
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// First column of a stage's accumulators: stages 1-3 three slots of 32
// columns, stage 4 three of 16, stage 0 two of 32.
__device__ __forceinline__ uint32_t acc_col(int stage) { return stage == 0 ? 384 : stage == 4 ? 288 : 96 * (stage - 1); }

struct NetTask {
    int img, x0, y0, y1;   // output columns from x0, rows y0 .. y1 - 1
};
__device__ __forceinline__ NetTask net_task(const NetArgs &a, int it) {
    const int tx = (a.w + kTileOut - 1) / kTileOut, ty = (a.h + a.seg - 1) / a.seg;
    NetTask t;
    t.img = it / (tx * ty);
    t.x0 = (it % tx) * kTileOut;
    t.y0 = ((it / tx) % ty) * a.seg;
    t.y1 = min(t.y0 + a.seg, a.h);
    return t;
}
__device__ __forceinline__ int net_tasks(const NetArgs &a) {
    return a.n * ((a.w + kTileOut - 1) / kTileOut) * ((a.h + a.seg - 1) / a.seg);
}

// The warp that issues stage 0's MMAs (control flow and operands uniform).
template <int T, bool LIMIT>
__device__ __forceinline__ void net_issue0(const NetArgs &a, const uint8_t *sB, const uint8_t *sA0, NetBars *bars,
                                           uint32_t tmem, volatile int *stop) {
    const uint64_t bd = umma::desc(umma::smem_addr(sB) + 3 * kBMidF + kBLastF, 128, 256);
    const uint64_t ad = umma::desc(umma::smem_addr(sA0), 128, 256);
    int r = 0;
    for (int it = blockIdx.x; it < net_tasks(a); it += gridDim.x) {
        const NetTask k = net_task(a, it);
        for (int j = 0; j < k.y1 - k.y0 + 2 * T; ++j, ++r) {
            const int b = r & 1;
            if (!net_wait_warp<LIMIT>(a, &bars->a0_full[b], (r >> 1) & 1, stop)) return;
            umma::fence_after_sync();
            if (umma::elect_one()) {
                umma::mma(tmem + acc_col(0) + 32 * b, ad + b * (kA0 >> 4), bd, umma::idesc_bf16(128, 32), false);
                umma::commit(&bars->acc0_full[b]);
            }
            __syncwarp();
        }
    }
}

// The warp that issues stage l's MMAs (BLK: bytes of one B block,
// NC: accumulator columns per slot).  Input row j of a task takes part in
// the output rows j - 2 .. j (counted from the task's first), which live in
// the slots of their index mod 3.
template <int T, int BLK, int NC, bool LIMIT>
__device__ __forceinline__ void net_issue(const NetArgs &a, int l, const uint8_t *rings, const uint8_t *sB,
                                          NetBars *bars, uint32_t tmem, volatile int *stop) {
    const uint64_t ad = umma::desc(umma::smem_addr(rings) + (l - 1) * kRings * kSlot, kLbo, 128);
    const uint64_t bd = umma::desc(umma::smem_addr(sB) + (l - 1) * kBMidF, 128, 256);
    const uint32_t d = tmem + acc_col(l);
    int u = 0, drains = 0;
    for (int it = blockIdx.x; it < net_tasks(a); it += gridDim.x) {
        const NetTask k = net_task(a, it);
        const int rows = k.y1 - k.y0 + 2 * (T - l + 1);
        for (int j = 0; j < rows; ++j, ++u) {
            const int b = u % kRings;
            if (!net_wait_warp<LIMIT>(a, &bars->in_full[l][b], (u / kRings) & 1, stop)) return;
            if (j == 0 || j >= 3) {   // output row j's slot is free
                if (!net_wait_warp<LIMIT>(a, &bars->drained[l], drains & 1, stop)) return;
                ++drains;
            }
            umma::fence_after_sync();
            const int rot = j % 3;
            const uint32_t idesc = umma::idesc_bf16(128, NC) + ((uint32_t)(min(j, 2) * NC / 8) << 17);
            const uint64_t as = ad + b * (kSlot >> 4), bs = bd + (rot == 0 ? BLK >> 4 : rot == 1 ? 0 : BLK >> 3);
            if (umma::elect_one()) {
#pragma unroll
                for (int s = 0; s < 6; ++s)   // K-step: dx = s / 2, channels 16 (s & 1) ..
                    umma::mma(d, as + (s >> 1) + (s & 1) * (2 * kLbo >> 4), bs + s * (kSeq * BLK >> 4), idesc, true);
                umma::commit(&bars->in_free[l][b]);
                if (j >= 2) umma::commit(&bars->acc_full[l]);
            }
            __syncwarp();
        }
    }
}

// Bias and ReLU, or the ReLU gate, of one pixel's 32 channels; `in`: the
// pixel lies in the image (outside it every stage's output is the zero
// padding).
template <bool BWD>
__device__ __forceinline__ void net_act(const float (&v)[32], const float *bias, const uint4 (&gate)[4], bool in,
                                        uint4 (&o)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float f[8], bv[8] = {};
        if constexpr (!BWD) {
            const float4 b0 = reinterpret_cast<const float4 *>(bias)[2 * q], b1 = reinterpret_cast<const float4 *>(bias)[2 * q + 1];
            bv[0] = b0.x, bv[1] = b0.y, bv[2] = b0.z, bv[3] = b0.w;
            bv[4] = b1.x, bv[5] = b1.y, bv[6] = b1.z, bv[7] = b1.w;
        }
        const uint32_t gw[4] = {gate[q].x, gate[q].y, gate[q].z, gate[q].w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if constexpr (BWD) {
                const float g = __uint_as_float(e & 1 ? gw[e >> 1] & 0xffff0000u : gw[e >> 1] << 16);
                f[e] = g > 0.f ? v[8 * q + e] : 0.f;
            } else {
                f[e] = fmaxf(v[8 * q + e] + bv[e], 0.f);
            }
        }
        o[q] = make_uint4(pack2(f[0], f[1]), pack2(f[2], f[3]), pack2(f[4], f[5]), pack2(f[6], f[7]));
        if (!in) o[q] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// Epilogue of the last layer (residual r).
__device__ __forceinline__ float store_last(const NetArgs &a, size_t p, float r, float bias, float x, float t) {
    const float yv = x + r + bias;
    if (a.y) a.y[p] = yv;
    if (a.mode == kTrain) {
        const float e = yv - t;
        a.dz[p] = a.grad_scale * e;
        return e * e;
    }
    if (a.mode == kRgba) {
        const int yy = min(max(__float2int_rd(fmaf(yv, 255.f, 0.5f)), 0), 255);
        const uchar4 c = to_rgba(yy, a.cb[p], a.cr[p]);
        const int xw = (int)(p % a.w), yh = (int)(p / a.w);
        *reinterpret_cast<uchar4 *>(a.rgba + (size_t)yh * a.pitch + 4 * (size_t)xw) = c;
    }
    return 0.f;
}

// A stage's warpgroup (thread = pixel of the tile).  T: the last stage.
template <bool BWD, int T, bool LIMIT>
__device__ __forceinline__ void net_stage(const NetArgs &a, int l, uint8_t *rings, uint8_t *sA0, const float *bias,
                                          NetBars *bars, uint32_t tmem, volatile int *stop) {
    const int px = threadIdx.x & 127, lane = threadIdx.x & 31;
    const uint32_t acc = tmem + acc_col(l) + ((uint32_t)(px & 96) << 16);
    int outs = 0;       // rows completed by this stage (all tasks)
    float e2 = 0.f;
    if (l > 0) {        // zeroed accumulators
        if (l == 4) {
            for (int k = 0; k < 3; ++k) umma::zero16(acc + 16 * k);
        } else {
            for (int k = 0; k < 3; ++k) umma::zero32(acc + 32 * k);
        }
        umma::fence_before_sync();
        __syncwarp();
        if (lane == 0) umma::mbar_arrive(&bars->drained[l]);
    }
    for (int it = blockIdx.x; it < net_tasks(a); it += gridDim.x) {
        const NetTask k = net_task(a, it);
        const int rows = k.y1 - k.y0 + 2 * (T - l);
        const int gx = k.x0 - 4 + px;
        const bool xin = gx >= 0 && gx < a.w, xown = px >= 4 && px < 4 + kTileOut && xin;
        const size_t img = (size_t)k.img * a.h;
        float win[9], nxt[3];
        // stage 0: the window's next row, columns gx - 1 .. gx + 1
        auto fetch = [&](int y) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int xx = gx + c - 1;
                nxt[c] = y >= 0 && y < a.h && xx >= 0 && xx < a.w ? __ldg(a.in_plane + (img + y) * a.w + xx) : 0.f;
            }
        };
        auto slide = [&]() {
#pragma unroll
            for (int c = 0; c < 6; ++c) win[c] = win[c + 3];
#pragma unroll
            for (int c = 0; c < 3; ++c) win[6 + c] = nxt[c];
        };
        // stage 0: the operand row of its output row `r` (counted over all tasks), then the next fetch
        auto build = [&](int r, int y) {
            slide();
            fetch(y + 2);
            uint8_t *d = sA0 + (r & 1) * kA0 + (px >> 3) * 256 + (px & 7) * 16;
            *reinterpret_cast<uint4 *>(d) = make_uint4(pack2(win[0], win[1]), pack2(win[2], win[3]),
                                                       pack2(win[4], win[5]), pack2(win[6], win[7]));
            *reinterpret_cast<uint4 *>(d + 128) = make_uint4(pack2(win[8], 0.f), 0u, 0u, 0u);
            umma::fence_smem_to_async();
            umma::fence_before_sync();
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&bars->a0_full[r & 1]);
        };
        if (l == 0) {
            const int y = k.y0 - T;
#pragma unroll
            for (int c = 0; c < 9; ++c) win[c] = 0.f;
            fetch(y - 1);
            slide();
            fetch(y);
            slide();
            fetch(y + 1);
            build(outs, y);
        }
        uint4 gate[4] = {};   // fetched a row ahead
        auto load_gate = [&](int y) {
            if (BWD && xin && y >= 0 && y < a.h) {
                const uint4 *src = reinterpret_cast<const uint4 *>(a.gate[l] + ((img + y) * a.w + gx) * kC);
#pragma unroll
                for (int c = 0; c < 4; ++c) gate[c] = __ldg(src + c);
            }
        };
        load_gate(k.y0 - (T - l));
        for (int q = 0; q < rows; ++q) {
            const int y = k.y0 - (T - l) + q;
            const bool in = xin && y >= 0 && y < a.h, own = xown && y >= k.y0 && y < k.y1;
            const size_t p = (img + y) * a.w + gx;
            if (l == 0 && q + 1 < rows) build(outs + 1, y + 1);
            float xv = 0.f, tv = 0.f;
            if (!BWD && l == 4 && own) {
                xv = __ldg(a.x + p);
                if (a.mode == kTrain) tv = __ldg(a.t + p);
            }
            if (l == 0) {
                if (!net_wait_warp<LIMIT>(a, &bars->acc0_full[outs & 1], (outs >> 1) & 1, stop)) return;
            } else {
                if (!net_wait_warp<LIMIT>(a, &bars->acc_full[l], outs & 1, stop)) return;
            }
            umma::fence_after_sync();
            if (!BWD && l == 4) {
                const float r = umma::ld1(acc + 16 * (q % 3));
                if (q + 1 < rows) {
                    umma::zero16(acc + 16 * (q % 3));
                } else {   // the task's MMAs of this stage are done: the rows past its end leave nothing behind
                    for (int c = 0; c < 3; ++c) umma::zero16(acc + 16 * c);
                }
                umma::fence_before_sync();
                __syncwarp();
                if (lane == 0) umma::mbar_arrive(&bars->drained[l]);
                if (own) e2 += store_last(a, p, r, bias[0], xv, tv);
                ++outs;
                continue;
            }
            float v[32];
            if (l == 0) {
                umma::ld32(acc + 32 * (outs & 1), v);
                umma::fence_before_sync();
            } else {
                umma::ld32(acc + 32 * (q % 3), v);
                if (q + 1 < rows) {
                    umma::zero32(acc + 32 * (q % 3));
                } else {
                    for (int c = 0; c < 3; ++c) umma::zero32(acc + 32 * c);
                }
                umma::fence_before_sync();
                __syncwarp();
                if (lane == 0) umma::mbar_arrive(&bars->drained[l]);
            }
            uint4 o[4];
            net_act<BWD>(v, bias, gate, in, o);
            if (q + 1 < rows) load_gate(y + 1);
            // into the next stage's ring (the last stage's rows only pass
            // through it on their way to memory)
            const int b = outs % kRings;
            if (l < T && outs >= kRings && !net_wait_warp<LIMIT>(a, &bars->in_free[l + 1][b], (outs / kRings - 1) & 1, stop)) return;
            uint8_t *row = rings + (l * kRings + b) * kSlot + 16;
#pragma unroll
            for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4 *>(row + px * 16 + c * kLbo) = o[c];
            if (l < T) {
                umma::fence_smem_to_async();
                __syncwarp();
                if (lane == 0) umma::mbar_arrive(&bars->in_full[l + 1][b]);
            }
            if (a.out[l] && y >= k.y0 && y < k.y1) {
                // whole 64-byte pixels by four lanes each: a warp writes 512 contiguous bytes
                __syncwarp();
                uint4 *dst = reinterpret_cast<uint4 *>(a.out[l] + ((img + y) * a.w + k.x0 - 4) * kC);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int i = 128 * (px >> 5) + 32 * c + lane, x = i >> 2;
                    if (x >= 4 && x < 4 + kTileOut && k.x0 - 4 + x < a.w)
                        dst[i] = *reinterpret_cast<const uint4 *>(row + x * 16 + (i & 3) * kLbo);
                }
            }
            ++outs;
        }
    }
    if (!BWD && l == 4 && a.mode == kTrain) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, o);
        if (lane == 0 && e2 != 0.f) atomicAdd(a.loss, e2);
    }
}

template <bool BWD, bool LIMIT>
__global__ void __launch_bounds__(net_threads(BWD), 1) k_net(NetArgs a) {
    constexpr int T = BWD ? 3 : 4, kNetThreads = net_threads(BWD);
    extern __shared__ __align__(128) uint8_t sm[];
    uint8_t *rings = sm, *sB = sm + kNetRing, *sA0 = sB + 3 * kBMidF + kBLastF + kBIn1;
    __shared__ NetBars bars;
    __shared__ uint32_t tmem_base;
    __shared__ int stop;
    __shared__ __align__(16) float sBias[kStages][kC];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // uniform
    // B of the 32-channel stages: per K-step (dx, half of the channels) the
    // blocks of dy = 1, 0, 2, 1, 0
    for (int l = 1; l <= T; ++l) {
        const int blk = l == 4 ? kBBlock / 2 : kBBlock;
        uint8_t *dst = sB + (l - 1) * kBMidF;
        for (int i = 16 * tid; i < 6 * kSeq * blk; i += 16 * kNetThreads) {
            const int s = i / (kSeq * blk), r = (i / blk) % kSeq;
            const int dy = r == 2 ? 2 : (r == 0 || r == 3) ? 1 : 0;
            const int step = (dy * 3 + (s >> 1)) * 2 + (s & 1);
            *reinterpret_cast<uint4 *>(dst + i) = __ldg(reinterpret_cast<const uint4 *>(a.pack[l] + step * blk + i % blk));
        }
    }
    for (int i = 16 * tid; i < kBIn1; i += 16 * kNetThreads)
        *reinterpret_cast<uint4 *>(sB + 3 * kBMidF + kBLastF + i) = __ldg(reinterpret_cast<const uint4 *>(a.pack[0] + i));
    // the pixels left and right of the tile's 128 (read by its outermost,
    // invalid columns)
    for (int i = tid; i < 4 * kRings * 8; i += kNetThreads) {
        const int c = i & 3, e = (i >> 2) & 1;
        *reinterpret_cast<uint4 *>(rings + (i >> 3) * kSlot + c * kLbo + (e ? kRowPx - 1 : 0) * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
    if (!BWD)
        for (int i = tid; i < kStages * kC; i += kNetThreads) {
            const int l = i / kC;
            sBias[l][i % kC] = l < 4 || i % kC == 0 ? __ldg(a.bias[l] + i % kC) : 0.f;
        }
    if (tid == 0) {
        stop = 0;
        for (int l = 0; l < kStages; ++l) {
            for (int b = 0; b < kRings; ++b) {
                umma::mbar_init(&bars.in_full[l][b], 4);
                umma::mbar_init(&bars.in_free[l][b], 1);
            }
            umma::mbar_init(&bars.acc_full[l], 1);
            umma::mbar_init(&bars.drained[l], 4);
            umma::mbar_init(&bars.idle[l], 1);
        }
        for (int b = 0; b < 2; ++b) {
            umma::mbar_init(&bars.a0_full[b], 4);
            umma::mbar_init(&bars.acc0_full[b], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4 * (T + 1)) umma::tmem_alloc<512>(&tmem_base);
    umma::fence_smem_to_async();
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t tmem = tmem_base;
    if (warp >= 4 * (T + 1)) {
        const int l = warp - 4 * (T + 1);
        if (l == 0) net_issue0<T, LIMIT>(a, sB, sA0, &bars, tmem, &stop);
        else if (l < 4) net_issue<T, kBBlock, 32, LIMIT>(a, l, rings, sB, &bars, tmem, &stop);
        else net_issue<T, kBBlock / 2, 16, LIMIT>(a, l, rings, sB, &bars, tmem, &stop);
        if (umma::elect_one()) {
            umma::commit(&bars.idle[l]);
            umma::mbar_wait(&bars.idle[l], 0);
        }
        __syncwarp();
    } else {
        net_stage<BWD, T, LIMIT>(a, warp >> 2, rings, sA0, sBias[warp >> 2], &bars, tmem, &stop);
    }
    umma::fence_before_sync();
    __syncthreads();
    if (tid == 0 && stop) record_error(a.err, WV_ERR_TIMEOUT);
    if (warp == 4 * (T + 1)) umma::tmem_free<512>(tmem);
}

// Weight gradient of a 32 -> 32 layer on the tensor cores:
// dW[tap][ci][co] = sum over pixels of act[p + tap][ci] dz[p][co].  The sum
// runs over pixels, so both operands are read with their channels along the
// MMA's M or N and pixels along K: exactly how the channel-last rows lie in
// shared memory as 8-channel columns (16 bytes a pixel), with the descriptor's
// "MN-major" form; nothing is transposed.  A tile is kWRowsT rows x 128 pixels
// of dz with the kWRowsT + 2 rows of act around them.  For row y and shift dx,
// A starts at act row y - 1, pixel dx: consecutive row slots continue the
// 8-channel columns, so its M = 128 holds (dy, ci) for dy = 0..2 (the fourth
// row's products land in accumulator rows that are never read).  The three dx
// accumulate in three 32-column TMEM ranges over all tiles of the CTA, which
// adds them to the global gradient once at its end, in the gradient's order.
// The bias gradient is summed from the dz rows in shared memory meanwhile.
//
// Bound: the MMAs' reads of A (4 KB per 16 pixels and dx) and the 128 bytes
// per pixel from HBM, about 20 us each for 16 x 256^2 pixels of a layer, and
// the waits of a CTA between its loads and its MMAs; two CTAs per SM so that
// one's loads run under the other's MMAs (one CTA with two operand buffers:
// 88 us, too few warps issuing loads).  Counters of the three layers' launch:
// tensor pipe 18 % active, DRAM 27 %, warps stalled on their loads.  One
// layer alone takes 70 us (with both operands transposed through shared memory
// by the threads 434), the three of a step in one launch 190: a third of the
// CTAs' fills, drains and gradient additions, which go out four floats at a
// time.
constexpr int kWRowsT = 4;                              // dz rows per tile
constexpr int kWThreads = 256;
constexpr int kWAct = (kWRowsT + 3) * kSlot;            // kWRowsT + 2 rows, one more that the last M reads
constexpr int kWDz = kWRowsT * kSlot;                   // dz rows in the same layout (pixels 0..127)
constexpr int kWSmem = kWAct + kWDz;
static_assert(kC * kC * 9 * 4 <= kWSmem, "the gradient is staged in the operand buffers");

__device__ __forceinline__ void cp_async16(uint8_t *dst, const void *src, bool fill) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(umma::smem_addr(dst)), "l"(src),
                 "r"(fill ? 16 : 0)
                 : "memory");
}

// The three layers of a step, one of them per CTA: layer blockIdx.x % layers.
constexpr int kMidLayers = 3;
struct WgradArgs {
    const bf16 *act[kMidLayers], *dz[kMidLayers];
    float *dW[kMidLayers], *db[kMidLayers];   // dW 16-byte aligned
    int layers, n, h, w;
    int *err;
    int polls;   // of a wait for the MMAs before it gives up
};

__global__ void __launch_bounds__(kWThreads, 2) k_wgrad_mid(WgradArgs args) {
    extern __shared__ __align__(128) uint8_t sm[];
    const int layer = blockIdx.x % args.layers, cta = blockIdx.x / args.layers, ctas = gridDim.x / args.layers;
    const bf16 *__restrict__ act = args.act[layer], *__restrict__ dz = args.dz[layer];
    float *dW = args.dW[layer], *db = args.db[layer];
    int *err = args.err;
    const int n = args.n, h = args.h, w = args.w;
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ float sBias[kC];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // uniform
    if (tid == 0) umma::mbar_init(&mbar, 3);
    if (tid < kC) sBias[tid] = 0.f;
    if (warp == 0) umma::tmem_alloc<128>(&tmem_base);
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t tmem = tmem_base;
    const uint32_t idesc = umma::idesc_bf16(128, 32) | umma::kAMnMajor | umma::kBMnMajor;
    const int tx = (w + kTilePx - 1) / kTilePx, ty = (h + kWRowsT - 1) / kWRowsT;
    const int total = n * tx * ty;
    const int q = tid & 3, p0 = tid >> 2;   // this thread's 8 channels and first pixel of a row
    uint8_t *buf = sm;
    auto load = [&](int it) {
        const int x0 = (it % tx) * kTilePx, y0 = ((it / tx) % ty) * kWRowsT, img = it / (tx * ty);
        const int rows = min(kWRowsT, h - y0), px = (min(kTilePx, w - x0) + 15) & ~15;
        for (int r = 0; r < rows + 2; ++r) {
            const int yy = y0 + r - 1;
            const bool yin = yy >= 0 && yy < h;
            const bf16 *src = act + ((long long)img * h + yy) * w * kC + q * 8;
            for (int i = p0; i < px + 2; i += kWThreads / 4) {
                const int xx = x0 - 1 + i;
                const bool in = yin && xx >= 0 && xx < w;
                cp_async16(buf + r * kSlot + q * kLbo + i * 16, in ? src + (long long)xx * kC : act, in);
            }
        }
        for (int r = 0; r < rows; ++r) {
            const bf16 *src = dz + ((long long)img * h + y0 + r) * w * kC + q * 8;
            for (int i = p0; i < px; i += kWThreads / 4)
                cp_async16(buf + kWAct + r * kSlot + q * kLbo + i * 16, x0 + i < w ? src + (long long)(x0 + i) * kC : dz,
                           x0 + i < w);
        }
    };
    uint32_t phase = 0;
    bool first = true, ok = true;
    float bsum[8] = {};   // channels 8 q ..
    auto wait_mma = [&]() {
        const bool got = __syncthreads_and(umma::mbar_wait(&mbar, phase, args.polls));
        if (!got) {
            ok = false;
            if (tid == 0) record_error(err, WV_ERR_TIMEOUT);
            umma::mbar_wait(&mbar, phase);   // no MMA in flight when the CTA ends
        }
        phase ^= 1;
    };
    for (int it = cta; it < total; it += ctas) {
        if (!first) wait_mma();
        if (!ok) break;
        load(it);
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
        umma::fence_smem_to_async();
        umma::fence_before_sync();
        __syncthreads();
        umma::fence_after_sync();
        const int x0 = (it % tx) * kTilePx, y0 = ((it / tx) % ty) * kWRowsT;
        const int rows = min(kWRowsT, h - y0);
        const int steps = (min(kTilePx, w - x0) + 15) / 16;   // K-steps of 16 pixels
        if (warp < 3) {   // dx = warp: its own accumulator, its own issuing warp
            const uint64_t a0 = umma::desc(umma::smem_addr(buf) + warp * 16, 128, kLbo);
            const uint64_t b0 = umma::desc(umma::smem_addr(buf + kWAct), 128, kLbo);
            const uint32_t d = tmem + 32 * warp;
#pragma unroll 1
            for (int r = 0; r < rows; ++r) {
                const uint64_t ar = a0 + r * (kSlot >> 4), br = b0 + r * (kSlot >> 4);
                if (umma::elect_one()) {
#pragma unroll
                    for (int s = 0; s < kTilePx / 16; ++s)
                        if (s < steps) umma::mma(d, ar + 16 * s, br + 16 * s, idesc, !first || r > 0 || s > 0);
                }
                __syncwarp();
            }
            if (umma::elect_one()) umma::commit(&mbar);
            __syncwarp();
        }
        first = false;
        for (int r = 0; r < rows; ++r)
            for (int i = p0; i < 16 * steps; i += kWThreads / 4) {
                const uint4 v = *reinterpret_cast<const uint4 *>(buf + kWAct + r * kSlot + q * kLbo + i * 16);
                const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    bsum[2 * e] += __uint_as_float(u[e] << 16);
                    bsum[2 * e + 1] += __uint_as_float(u[e] & 0xffff0000u);
                }
            }
    }
    if (!first && ok) wait_mma();
    if (!first && ok) {
        // the accumulators, reordered to the gradient's [co][ci][tap] in the
        // operand buffers (the MMAs have completed), then one coalesced pass
        umma::fence_after_sync();
        float *out = reinterpret_cast<float *>(sm);
        const int m = (warp & 3) * 32 + (tid & 31), dy = m >> 5, ci = m & 31;
        for (int dx = warp >> 2; dx < 3; dx += kWThreads / 128) {
            float v[32];
            umma::ld32(tmem + 32 * dx + ((uint32_t)((warp & 3) * 32) << 16), v);
            if (dy < 3)
#pragma unroll
                for (int co = 0; co < 32; ++co) out[(co * kC + ci) * 9 + dy * 3 + dx] = v[co];
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float v = bsum[e];
#pragma unroll
            for (int o = 4; o < 32; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
            if ((tid & 31) < 4) atomicAdd(&sBias[8 * (tid & 3) + e], v);
        }
        __syncthreads();
        for (int i = tid; i < kC * kC * 9 / 4; i += kWThreads)
            atomicAdd(reinterpret_cast<float4 *>(dW) + i, reinterpret_cast<const float4 *>(out)[i]);
        if (tid < kC) atomicAdd(db + tid, sBias[tid]);
    }
    umma::fence_before_sync();
    __syncthreads();
    if (warp == 0) umma::tmem_free<128>(tmem);
}

// Weight gradients of the first (1 -> 32) and last (32 -> 1) layers on CUDA
// cores, in fp32: G[tap][c] = sum over pixels q of T[q][c] P[q + tap - 1],
// with T the layer's 32-channel tensor and P its one-channel plane.  First
// layer: T = dZ, P = the input, tap as is; last layer: T = the input, P = dZ,
// tap flipped (T[p + tap - 1] P[p] = T[q] P[q - (tap - 1)]).  Four lanes hold a
// pixel's channels (one 16-byte load each) and walk along a run of a row, eight
// runs side by side in a warp, with the 3 x 3 window of P sliding in registers:
// 4 loads and 36 packed FMAs for 8 pixels.
// Bound: latency.  With the tensor's loads in the loop (no registers left to
// fetch ahead) it took 47 us for 16 x 256^2 pixels, 2 us for every three pixels
// of a lane; each lane now copies its own pixels to shared memory kEStages - 1
// steps of three ahead: 39 us.  (Staged in shared memory per CTA, with two loads
// per FMA, 138 and 153 us.)
constexpr int kEWarps = 8;
constexpr int kERunMax = 33;     // pixels per run, a multiple of the window's 3 columns
constexpr int kEStages = 6;
constexpr int kEStage = 3 * 32 * 16;                      // bytes of a warp's step
constexpr int kESmem = kEWarps * kEStages * kEStage;

__global__ void __launch_bounds__(32 * kEWarps, 2) k_wgrad_edge(const float *__restrict__ plane,
                                                               const bf16 *__restrict__ act, int first_layer, int n, int h,
                                                               int w, int run, int runs, float *dW, float *db) {
    __shared__ float sum[kEWarps][kC * 10];   // [c][tap], then the bias
    extern __shared__ __align__(128) uint8_t sm[];
    const int tid = threadIdx.x, lane = tid & 31, q = lane & 3, warp = tid >> 5;
    float2 acc[9][4] = {}, bias[4] = {};
    float centre = 0.f;
    const int total = n * h * runs;
    for (int it = blockIdx.x * kEWarps + warp; it < total; it += gridDim.x * kEWarps) {
        const int y = (it / runs) % h, img = it / (runs * h);
        const int xa = ((it % runs) * 8 + (lane >> 2)) * run, xe = min(xa + run, w);
        const float *row = plane + ((size_t)img * h + y) * w;
        const uint4 *t = reinterpret_cast<const uint4 *>(act + ((size_t)img * h + y) * w * kC) + q;
        const bool up = y > 0, dn = y + 1 < h;
        auto load = [&](int x, float (&v)[3]) {
            const bool in = (unsigned)x < (unsigned)w;
            v[0] = in && up ? __ldg(row - w + x) : 0.f;
            v[1] = in ? __ldg(row + x) : 0.f;
            v[2] = in && dn ? __ldg(row + w + x) : 0.f;
        };
        // the lane's pixels xa + 3 g .. + 2 into its slots of stage g mod kEStages
        uint8_t *ring = sm + (size_t)warp * kEStages * kEStage + lane * 16;
        auto fetch = [&](int g) {
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const int x = xa + 3 * g + r;
                const bool in = 3 * g < run && x < xe;
                cp_async16(ring + (g % kEStages) * kEStage + r * 512, reinterpret_cast<const uint8_t *>(in ? t + 4 * (size_t)x : t), in);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        for (int g = 0; g < kEStages - 1; ++g) fetch(g);
        float p[3][3];   // window columns x - 1, x, x + 1 (rotating)
        load(xa - 1, p[0]);
        load(xa, p[1]);
#pragma unroll 1
        for (int k0 = 0, g = 0; k0 < run; k0 += 3, ++g) {
            fetch(g + kEStages - 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(kEStages - 1) : "memory");
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const int x = xa + k0 + r;
                load(x + 1, p[(r + 2) % 3]);
                const uint4 u = *reinterpret_cast<const uint4 *>(ring + (g % kEStages) * kEStage + r * 512);
                const uint32_t uw[4] = {u.x, u.y, u.z, u.w};
                float2 tv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    tv[e] = make_float2(__uint_as_float(uw[e] << 16), __uint_as_float(uw[e] & 0xffff0000u));
                    if (first_layer) bias[e] = __fadd2_rn(bias[e], tv[e]);
                }
                if (x < xe) centre += p[(r + 1) % 3][1];
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    const float pv = p[(r + k % 3) % 3][k / 3];
                    const float2 p2 = make_float2(pv, pv);
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[k][e] = __ffma2_rn(tv[e], p2, acc[k][e]);
                }
            }
        }
        // the fills past the run's end, before the next run's copies into the same slots
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    // over the warp's eight runs, then over the CTA's warps
    auto reduce = [&](float v) {
#pragma unroll
        for (int o = 4; o < 32; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
#pragma unroll
    for (int e = 0; e < 4; ++e) {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int tap = first_layer ? k : 8 - k;
            const float s0 = reduce(acc[k][e].x), s1 = reduce(acc[k][e].y);
            if (lane < 4) {
                sum[warp][(8 * q + 2 * e) * 9 + tap] = s0;
                sum[warp][(8 * q + 2 * e + 1) * 9 + tap] = s1;
            }
        }
        const float b0 = reduce(bias[e].x), b1 = reduce(bias[e].y);
        if (lane < 4) {
            sum[warp][kC * 9 + 8 * q + 2 * e] = b0;
            sum[warp][kC * 9 + 8 * q + 2 * e + 1] = b1;
        }
    }
    centre = reduce(centre);
    if (!first_layer && lane == 0) sum[warp][kC * 9] = centre;
    __syncthreads();
    // dW0[co][0][tap], dW4[0][ci][tap]; the bias gradient is the sum of dZ:
    // the tensor's (first layer) or the plane's (last layer)
    for (int i = tid; i < kC * 9 + (first_layer ? kC : 1); i += 32 * kEWarps) {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < kEWarps; ++k) v += sum[k][i];
        atomicAdd(i < kC * 9 ? dW + i : db + i - kC * 9, v);
    }
}

// bf16 B operands from the fp32 master parameters (one thread per element).
__global__ void k_pack(const float *__restrict__ P, uint8_t *pack) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;   // bf16 element index
    const int byte = 2 * e;
    if (byte >= kPackBytes) return;
    float v = 0.f;
    auto mid = [&](int base, int layer, bool bwd) {
        // K index k = tap * 32 + c, K-step t = k / 16; 32 rows
        const int o = byte - base, t = o / kStep32, in = o % kStep32;
        const int rg = in / 256, kc = (in % 256) / 128, r8 = (in % 128) / 16, k8 = (in % 16) / 2;
        const int r = rg * 8 + r8, kk = kc * 8 + k8, k = t * 16 + kk, tap = k >> 5, c = k & 31;
        // forward: row = co, K = (tap, ci); input gradient: row = ci, K = (flipped tap, co)
        const int co = bwd ? c : r, ci = bwd ? r : c, tp = bwd ? 8 - tap : tap;
        return P[off_w(layer) + (co * kC + ci) * 9 + tp];
    };
    auto in1 = [&](int base, int layer, bool bwd) {
        const int in = byte - base;
        const int rg = in / 256, kc = (in % 256) / 128, r8 = (in % 128) / 16, k8 = (in % 16) / 2;
        const int r = rg * 8 + r8, k = kc * 8 + k8;
        if (k >= 9) return 0.f;
        // forward layer 0: row = co, K = tap; input gradient of layer 4: row = ci, K = flipped tap
        return bwd ? P[off_w(layer) + r * 9 + (8 - k)] : P[off_w(layer) + r * 9 + k];
    };
    if (byte < kPF1) v = in1(kPF0, 0, false);
    else if (byte < kPF2) v = mid(kPF1, 1, false);
    else if (byte < kPF3) v = mid(kPF2, 2, false);
    else if (byte < kPF4) v = mid(kPF3, 3, false);
    else if (byte < kPB4) {
        const int o = byte - kPF4, t = o / 512, in = o % 512;
        const int rg = in / 256, kc = (in % 256) / 128, r8 = (in % 128) / 16, k8 = (in % 16) / 2;
        const int r = rg * 8 + r8, k = t * 16 + kc * 8 + k8;
        v = r == 0 ? P[off_w(4) + (k & 31) * 9 + (k >> 5)] : 0.f;
    } else if (byte < kPB3) v = in1(kPB4, 4, true);
    else if (byte < kPB2) v = mid(kPB3, 3, true);
    else if (byte < kPB1) v = mid(kPB2, 2, true);
    else v = mid(kPB1, 1, true);
    reinterpret_cast<bf16 *>(pack)[e] = __float2bfloat16_rn(v);
}

__global__ void k_adam(float *P, const float *G, float *M, float *V, int n, float lr, float b1, float b2,
                       float c1, float c2, float eps) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float g = G[i];
    const float m = b1 * M[i] + (1.f - b1) * g;
    const float v = b2 * V[i] + (1.f - b2) * g * g;
    M[i] = m;
    V[i] = v;
    P[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

int sm_count() {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

}  // namespace
}  // namespace wv

using namespace wv;

struct wv_cnn {
    int device = 0;
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    uint8_t *pack = nullptr;
    bool packed = false;
    int step = 0;
    bf16 *act[4] = {};                 // training: layer outputs
    bf16 *g[4] = {};                   // training: gradients of the layers' outputs
    float *dz5 = nullptr, *loss = nullptr, *xbuf = nullptr;
    uint8_t *cb = nullptr, *cr = nullptr;
    size_t cap_train = 0, cap_view = 0;
    std::vector<void *> owned_train, owned_view;
    int *err = nullptr;
    int wait_rounds = kWaitRounds;     // limit of the tensor-core kernels' bounded waits
};

namespace {

// Device buffers for px pixels; `ptr` gets the addresses of `bytes` per pixel.
struct Buffer {
    void **p;
    size_t bytes;
};
int ensure_buffers(std::vector<void *> &owned, size_t &cap, size_t px, std::initializer_list<Buffer> list) {
    if (px <= cap) return WV_OK;
    for (void *p : owned) cudaFree(p);
    owned.clear();
    cap = 0;
    const size_t want = px + px / 8;
    for (const Buffer &b : list) {
        *b.p = nullptr;
        if (cudaMalloc(b.p, want * b.bytes) != cudaSuccess) {
            cudaGetLastError();
            return WV_ERR_OOM;
        }
        owned.push_back(*b.p);
    }
    cap = want;
    return WV_OK;
}
// A training step keeps every layer's output and its gradient.
int ensure_train(wv_cnn *c, size_t px) {
    const size_t row = kC * sizeof(bf16);
    return ensure_buffers(c->owned_train, c->cap_train, px,
                          {{(void **)&c->act[0], row}, {(void **)&c->act[1], row}, {(void **)&c->act[2], row},
                           {(void **)&c->act[3], row}, {(void **)&c->g[0], row}, {(void **)&c->g[1], row},
                           {(void **)&c->g[2], row}, {(void **)&c->g[3], row}, {(void **)&c->dz5, 4}});
}
// A filtered viewport: its luma and chroma planes.
int ensure_view(wv_cnn *c, size_t px) {
    return ensure_buffers(c->owned_view, c->cap_view, px,
                          {{(void **)&c->xbuf, 4}, {(void **)&c->cb, 1}, {(void **)&c->cr, 1}});
}

void pack_params(wv_cnn *c, cudaStream_t cs) {
    const int elems = kPackBytes / 2;
    k_pack<<<(elems + 255) / 256, 256, 0, cs>>>(c->params, c->pack);
    c->packed = true;
}

// Rows per segment: the least time over all SMs.  A CTA computes S + 2 T rows
// in stage 0 for S rows and spends about 3 T more row times filling and draining
// its stages, so whole waves of long segments win on large images and short ones on small
// images that would leave SMs idle.
int seg_rows(int n, int h, int w, int T) {
    const long long tiles = (long long)n * ((w + kTileOut - 1) / kTileOut), sms = sm_count();
    long long best = -1;
    int seg = h;
    for (int k = 1; k <= 128 && k <= h; ++k) {
        const int s = (h + k - 1) / k;
        const long long waves = (tiles * ((h + s - 1) / s) + sms - 1) / sms, cost = waves * (s + 5 * T);
        if (best < 0 || cost < best) {
            best = cost;
            seg = s;
        }
    }
    return seg;
}

template <bool BWD, bool LIMIT>
cudaError_t launch_net_as(const NetArgs &a, int grid, cudaStream_t cs) {
    const cudaError_t e = opt_in_smem(reinterpret_cast<const void *>(k_net<BWD, LIMIT>), kNetSmem);
    if (e != cudaSuccess) return e;
    k_net<BWD, LIMIT><<<grid, net_threads(BWD), kNetSmem, cs>>>(a);
    return cudaGetLastError();
}

template <bool BWD>
cudaError_t launch_net(NetArgs &a, cudaStream_t cs) {
    a.seg = seg_rows(a.n, a.h, a.w, BWD ? 3 : 4);
    const long long tasks = (long long)a.n * ((a.w + kTileOut - 1) / kTileOut) * ((a.h + a.seg - 1) / a.seg);
    const int grid = (int)std::min<long long>(tasks, sm_count());
    return a.wait_rounds == kWaitRounds ? launch_net_as<BWD, false>(a, grid, cs) : launch_net_as<BWD, true>(a, grid, cs);
}

cudaError_t launch_wgrad_mid(const WgradArgs &a, cudaStream_t cs) {
    cudaError_t e = opt_in_smem(reinterpret_cast<const void *>(k_wgrad_mid), kWSmem);
    if (e != cudaSuccess) return e;
    const int total = a.n * ((a.h + kWRowsT - 1) / kWRowsT) * ((a.w + kTilePx - 1) / kTilePx);
    const int ctas = std::max(1, std::min(total, 2 * sm_count() / a.layers));   // of one layer
    k_wgrad_mid<<<ctas * a.layers, kWThreads, kWSmem, cs>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_wgrad_edge(const float *plane, const bf16 *act, int first, int n, int h, int w, float *dW,
                              float *db, cudaStream_t cs) {
    // equal runs that cover a row with the fewest warps
    const int runs = (w + 8 * kERunMax - 1) / (8 * kERunMax);
    const int run = 3 * ((w + 24 * runs - 1) / (24 * runs));
    const int total = n * h * runs;
    const int grid = std::max(1, std::min((total + kEWarps - 1) / kEWarps, 2 * sm_count()));
    const cudaError_t e = opt_in_smem(reinterpret_cast<const void *>(k_wgrad_edge), kESmem);
    if (e != cudaSuccess) return e;
    k_wgrad_edge<<<grid, 32 * kEWarps, kESmem, cs>>>(plane, act, first, n, h, w, run, runs, dW, db);
    return cudaGetLastError();
}

// Forward pass; the last layer's epilogue and outputs are set in `a`.
cudaError_t forward(wv_cnn *c, const float *x, int n, int h, int w, NetArgs &a, cudaStream_t cs) {
    if (!c->packed) pack_params(c, cs);
    const int packs[kStages] = {kPF0, kPF1, kPF2, kPF3, kPF4};
    a.in_plane = a.x = x;
    a.n = n;
    a.h = h;
    a.w = w;
    a.err = c->err;
    a.wait_rounds = c->wait_rounds;
    for (int l = 0; l < kStages; ++l) {
        a.pack[l] = c->pack + packs[l];
        a.bias[l] = c->params + off_b(l);
    }
    return launch_net<false>(a, cs);
}

// Forward with the training epilogue, then every gradient into c->grads.
cudaError_t forward_backward(wv_cnn *c, const float *x, const float *t, int n, int h, int w, cudaStream_t cs) {
    cudaError_t e = cudaMemsetAsync(c->grads, 0, sizeof(float) * kParams, cs);
    if (e == cudaSuccess) e = cudaMemsetAsync(c->loss, 0, sizeof(float), cs);
    if (e != cudaSuccess) return e;
    NetArgs a;
    memset(&a, 0, sizeof(a));
    a.mode = kTrain;
    a.t = t;
    a.dz = c->dz5;
    a.loss = c->loss;
    a.grad_scale = 2.f / (float)((double)n * h * w);
    for (int l = 0; l < 4; ++l) a.out[l] = c->act[l];
    e = forward(c, x, n, h, w, a, cs);
    if (e != cudaSuccess) return e;
    // gradients of the outputs of layers 3..0: stage s yields layer 3 - s's,
    // gated by that layer's output
    const int packs[4] = {kPB4, kPB3, kPB2, kPB1};
    memset(&a, 0, sizeof(a));
    a.in_plane = c->dz5;
    a.n = n;
    a.h = h;
    a.w = w;
    a.err = c->err;
    a.wait_rounds = c->wait_rounds;
    for (int s = 0; s < 4; ++s) {
        a.pack[s] = c->pack + packs[s];
        a.gate[s] = c->act[3 - s];
        a.out[s] = c->g[3 - s];
    }
    e = launch_net<true>(a, cs);
    if (e != cudaSuccess) return e;
    float *G = c->grads;
    WgradArgs m;
    memset(&m, 0, sizeof(m));
    m.layers = kMidLayers;
    m.n = n;
    m.h = h;
    m.w = w;
    m.err = c->err;
    m.polls = c->wait_rounds * kWaitRound;
    for (int l = 1; l <= kMidLayers; ++l) {
        m.act[l - 1] = c->act[l - 1];
        m.dz[l - 1] = c->g[l];
        m.dW[l - 1] = G + off_w(l);
        m.db[l - 1] = G + off_b(l);
    }
    e = launch_wgrad_edge(c->dz5, c->act[3], 0, n, h, w, G + off_w(4), G + off_b(4), cs);
    if (e == cudaSuccess) e = launch_wgrad_mid(m, cs);
    if (e == cudaSuccess) e = launch_wgrad_edge(x, c->g[0], 1, n, h, w, G + off_w(0), G + off_b(0), cs);
    return e;
}

int check_dims(int n, int h, int w) {
    return (n >= 1 && h >= 1 && w >= 1 && (double)n * h * w < 2e9 && h <= 65535 * 16 && n <= 65535)
               ? WV_OK
               : WV_ERR_ARG;
}

}  // namespace

extern "C" {

size_t wv_cnn_param_count(void) { return (size_t)kParams; }

int wv_cnn_create(const float *params_host, wv_cnn **out) {
    if (!params_host || !out) return WV_ERR_ARG;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        cudaGetLastError();
        return WV_ERR_CUDA;
    }
    wv_cnn *c = new (std::nothrow) wv_cnn();
    if (!c) return WV_ERR_OOM;
    cudaGetDevice(&c->device);
    bool ok = cudaMalloc(&c->params, sizeof(float) * kParams) == cudaSuccess &&
              cudaMalloc(&c->grads, sizeof(float) * kParams) == cudaSuccess &&
              cudaMalloc(&c->m, sizeof(float) * kParams) == cudaSuccess &&
              cudaMalloc(&c->v, sizeof(float) * kParams) == cudaSuccess &&
              cudaMalloc(&c->pack, kPackBytes) == cudaSuccess && cudaMalloc(&c->loss, 64) == cudaSuccess &&
              cudaMalloc(&c->err, 64) == cudaSuccess;
    if (ok)
        ok = cudaMemcpy(c->params, params_host, sizeof(float) * kParams, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemset(c->m, 0, sizeof(float) * kParams) == cudaSuccess &&
             cudaMemset(c->v, 0, sizeof(float) * kParams) == cudaSuccess &&
             cudaMemset(c->err, 0, 64) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        wv_cnn_close(c);
        return WV_ERR_OOM;
    }
    *out = c;
    return WV_OK;
}

void wv_cnn_close(wv_cnn *c) {
    if (!c) return;
    cudaDeviceSynchronize();
    for (void *p : c->owned_train) cudaFree(p);
    for (void *p : c->owned_view) cudaFree(p);
    cudaFree(c->params);
    cudaFree(c->grads);
    cudaFree(c->m);
    cudaFree(c->v);
    cudaFree(c->pack);
    cudaFree(c->loss);
    cudaFree(c->err);
    delete c;
}

int wv_cnn_get_params(wv_cnn *c, float *host) {
    if (!c || !host) return WV_ERR_ARG;
    return cudaMemcpy(host, c->params, sizeof(float) * kParams, cudaMemcpyDeviceToHost) == cudaSuccess ? WV_OK
                                                                                                       : WV_ERR_CUDA;
}

int wv_cnn_set_params(wv_cnn *c, const float *host) {
    if (!c || !host) return WV_ERR_ARG;
    c->packed = false;
    c->step = 0;
    if (cudaMemset(c->m, 0, sizeof(float) * kParams) != cudaSuccess ||
        cudaMemset(c->v, 0, sizeof(float) * kParams) != cudaSuccess)
        return WV_ERR_CUDA;
    return cudaMemcpy(c->params, host, sizeof(float) * kParams, cudaMemcpyHostToDevice) == cudaSuccess ? WV_OK
                                                                                                       : WV_ERR_CUDA;
}

int wv_cnn_get_state(wv_cnn *c, float *m_host, float *v_host, int *steps) {
    if (!c || !m_host || !v_host || !steps) return WV_ERR_ARG;
    if (cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy(m_host, c->m, sizeof(float) * kParams, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(v_host, c->v, sizeof(float) * kParams, cudaMemcpyDeviceToHost) != cudaSuccess)
        return WV_ERR_CUDA;
    *steps = c->step;
    return WV_OK;
}

int wv_cnn_set_state(wv_cnn *c, const float *m_host, const float *v_host, int steps) {
    if (!c || !m_host || !v_host || steps < 0) return WV_ERR_ARG;
    if (cudaMemcpy(c->m, m_host, sizeof(float) * kParams, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(c->v, v_host, sizeof(float) * kParams, cudaMemcpyHostToDevice) != cudaSuccess)
        return WV_ERR_CUDA;
    c->step = steps;
    return WV_OK;
}

int wv_cnn_forward(wv_cnn *c, const float *x_dev, float *y_dev, int n, int h, int w, void *cuda_stream) {
    if (!c || !x_dev || !y_dev || check_dims(n, h, w) != WV_OK) return WV_ERR_ARG;
    cudaStream_t cs = (cudaStream_t)cuda_stream;
    // Filtering in place: a CTA stores y while others still read x around
    // their own tiles, so where the planes overlap the network reads a copy of
    // x.  The copy is the call's own (stream-ordered memory), so that calls on
    // several streams do not share it and a captured call holds it itself.
    const size_t bytes = sizeof(float) * (size_t)n * h * w;
    const uintptr_t xa = (uintptr_t)x_dev, ya = (uintptr_t)y_dev;
    float *copy = nullptr;
    if (xa < ya + bytes && ya < xa + bytes) {
        if (cudaMallocAsync((void **)&copy, bytes, cs) != cudaSuccess) {
            cudaGetLastError();
            return WV_ERR_OOM;
        }
    }
    NetArgs fin;
    memset(&fin, 0, sizeof(fin));
    fin.mode = kOut;
    fin.y = y_dev;
    cudaError_t e = copy ? cudaMemcpyAsync(copy, x_dev, bytes, cudaMemcpyDeviceToDevice, cs) : cudaSuccess;
    if (e == cudaSuccess) e = forward(c, copy ? copy : x_dev, n, h, w, fin, cs);
    if (copy) {
        const cudaError_t ef = cudaFreeAsync(copy, cs);
        if (e == cudaSuccess) e = ef;
    }
    return e == cudaSuccess ? WV_OK : WV_ERR_CUDA;
}

int wv_cnn_gradients(wv_cnn *c, const float *x_dev, const float *t_dev, int n, int h, int w, float *grads_host,
                     float *loss_host, void *cuda_stream) {
    if (!c || !x_dev || !t_dev || check_dims(n, h, w) != WV_OK) return WV_ERR_ARG;
    if (ensure_train(c, (size_t)n * h * w) != WV_OK) return WV_ERR_OOM;
    cudaStream_t cs = (cudaStream_t)cuda_stream;
    if (forward_backward(c, x_dev, t_dev, n, h, w, cs) != cudaSuccess) return WV_ERR_CUDA;
    float loss = 0.f;
    cudaError_t e = cudaMemcpyAsync(&loss, c->loss, 4, cudaMemcpyDeviceToHost, cs);
    if (e == cudaSuccess && grads_host)
        e = cudaMemcpyAsync(grads_host, c->grads, sizeof(float) * kParams, cudaMemcpyDeviceToHost, cs);
    if (e == cudaSuccess) e = cudaStreamSynchronize(cs);
    if (loss_host) *loss_host = loss / (float)((double)n * h * w);
    return e == cudaSuccess ? WV_OK : WV_ERR_CUDA;
}

int wv_cnn_train_step(wv_cnn *c, const float *x_dev, const float *t_dev, int n, int h, int w, float lr,
                      float *loss_host, void *cuda_stream) {
    if (!c || !x_dev || !t_dev || check_dims(n, h, w) != WV_OK || !(lr > 0.f)) return WV_ERR_ARG;
    if (ensure_train(c, (size_t)n * h * w) != WV_OK) return WV_ERR_OOM;
    cudaStream_t cs = (cudaStream_t)cuda_stream;
    if (forward_backward(c, x_dev, t_dev, n, h, w, cs) != cudaSuccess) return WV_ERR_CUDA;
    c->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)c->step), c2 = 1.f - powf(b2, (float)c->step);
    k_adam<<<(kParams + 255) / 256, 256, 0, cs>>>(c->params, c->grads, c->m, c->v, kParams, lr, b1, b2, c1, c2,
                                                  1e-8f);
    pack_params(c, cs);
    if (cudaGetLastError() != cudaSuccess) return WV_ERR_CUDA;
    if (loss_host) {
        float loss = 0.f;
        if (cudaMemcpyAsync(&loss, c->loss, 4, cudaMemcpyDeviceToHost, cs) != cudaSuccess ||
            cudaStreamSynchronize(cs) != cudaSuccess)
            return WV_ERR_CUDA;
        *loss_host = loss / (float)((double)n * h * w);
    }
    return WV_OK;
}

int wv_cnn_set_wait_limit(wv_cnn *c, int polls) {
    if (!c || polls < 0) return WV_ERR_ARG;
    c->wait_rounds = std::min(polls / kWaitRound + (polls % kWaitRound != 0), kWaitRounds);
    return WV_OK;
}

int wv_cnn_sync_status(wv_cnn *c) {
    if (!c) return WV_ERR_ARG;
    if (cudaDeviceSynchronize() != cudaSuccess) return WV_ERR_CUDA;
    int err = 0;
    if (cudaMemcpy(&err, c->err, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return WV_ERR_CUDA;
    if (err) cudaMemset(c->err, 0, 4);
    return err;
}

// Viewport decode with the post-filter: the steps of wv_decode_viewport up
// to the decoded region, reprojection into luma / chroma planes, the network
// on the luma, colour conversion in the last layer's epilogue.
int wv_decode_viewport_filtered(wv_stream *s, int frame, float yaw, float pitch, float fov, wv_cnn *c,
                                const wv_image *out) {
    if (!s || !c || !out || !out->dptr || out->width <= 0 || out->height <= 0 ||
        out->pitch_bytes < (size_t)out->width * 4 || (out->pitch_bytes % 4) != 0)
        return WV_ERR_ARG;
    if (frame < 0 || frame >= s->g.num_frames || !(fov > 0.f && fov < 3.14159f)) return WV_ERR_ARG;
    const size_t px = (size_t)out->width * out->height;
    if (ensure_view(c, px) != WV_OK) return WV_ERR_OOM;
    // the region decode of the plain path, then the planes instead of RGBA
    int rc = wv::decode_region(s, frame, yaw, pitch, fov, out->width, out->height);
    if (rc != WV_OK) return rc;
    int row0, rows;
    eye_view(s->g, 0, &row0, &rows);   // eye 0 (the top half of a stereo frame)
    const View v = make_view(yaw, pitch, fov, out->width, out->height, s->g.p[0].w, rows, row0);
    launch_resample(s->g, v, recon_planes(s), nullptr, nullptr, 0, s->cs, c->xbuf, c->cb, c->cr, recon_pairs(s),
                    s->err);
    release_recon(s);
    NetArgs fin;
    memset(&fin, 0, sizeof(fin));
    fin.mode = kRgba;
    fin.cb = c->cb;
    fin.cr = c->cr;
    fin.rgba = (uint8_t *)out->dptr;
    fin.pitch = out->pitch_bytes;
    return forward(c, c->xbuf, 1, out->height, out->width, fin, s->cs) == cudaSuccess ? WV_OK : WV_ERR_CUDA;
}

}  // extern "C"
