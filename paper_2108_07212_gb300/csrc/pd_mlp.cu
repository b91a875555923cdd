// pd_mlp.cu -- the surrogate's multilayer perceptron on the tensor cores.
//
// y = W3 gelu(W2 gelu(W1 x + b1) + b2) + b3, 32 -> 128 -> 128 -> 32, with
// BF16 weights and activations as MMA operands and FP32 accumulation in tensor
// memory (tcgen05.mma kind::f16).  The forward pass of a 128-sample tile is
// one fused kernel: the three layers chain through shared memory and TMEM
// without touching global memory.  A training step is two: the forward and
// backward pass of a tile, whose activations never leave the SM, and the sum
// of the tiles' gradients with Adam and the BF16 copies; FP32 master weights,
// BF16 copies for the MMAs.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "pd_internal.h"
#include "pd_mlp_tile.cuh"
#include "pd_tc.cuh"
#include "peridem.h"

namespace pd {
namespace mlp {
constexpr long long kSpins = 1LL << 24;      // bounded mbarrier waits (~0.5 s)
constexpr int kFwdSmem = 104 * 1024;        // 88 KB of operands and the inference's input rows
constexpr int kTrainSmem = 216 * 1024;
constexpr int kParts = 152;                 // gradient partials at most: one per SM
constexpr int kPartStride = NPARAM + 32;    // a partial: the parameters' gradients, then the loss

struct Net {
    float *p, *g, *m, *v;                       // FP32 parameters, gradients, Adam moments
    __nv_bfloat16 *W1, *W2, *W3, *W2t, *W3t;    // BF16 weights [out][in] and transposed [in][out]
    float *parts;                               // gradient partials of a training step, kPartStride each
    float *loss;                                // [0] loss, [1] the error word (one copy to the host)
    int *err;
};

__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * __expf(-0.5f * z * z);
}

// ---------------------------------------------------------------------------
// pieces of a tile of R = 32, 64 or 128 samples on 512 threads: warp w reads
// TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31 (its quarter of the samples) and
// warpgroup w / 4 takes a quarter of a layer's columns.  The products always
// have 128 sample rows (rows from R on hold whatever shared memory does and are
// not read); a tile's time is that of its activations, so a small batch is cut
// into small tiles that more SMs share.

constexpr int kTileThreads = 512;
constexpr int kGroups = kTileThreads / TILE, kGroupCols = HID / kGroups;

// Columns 8 g .. 8 g + 7 of input row `row` (zero from B on).
__device__ __forceinline__ void load_row8(const float *__restrict__ X, int row, int g, int B, bool x16, float (&x)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = 0.f;
    if (row >= B) return;
    const float *src = X + (size_t)row * IN + 8 * g;
    if (x16) {
        const float4 a = *reinterpret_cast<const float4 *>(src), b = *reinterpret_cast<const float4 *>(src + 4);
        x[0] = a.x, x[1] = a.y, x[2] = a.z, x[3] = a.w, x[4] = b.x, x[5] = b.y, x[6] = b.z, x[7] = b.w;
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = src[q];
    }
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16(a)) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16(b)) << 16);
}
// N (a multiple of 8) consecutive columns c0.. of sample `row` as BF16 into the
// K-major operand [samples][features] at dst ...
template <int N>
__device__ __forceinline__ void store_row(uint8_t *dst, int row, int c0, const float (&v)[N]) {
#pragma unroll
    for (int q = 0; q < N; q += 8)
        *reinterpret_cast<uint4 *>(dst + tc::kmajor_off(row, c0 + q, TILE)) =
            make_uint4(pack_bf16(v[q], v[q + 1]), pack_bf16(v[q + 2], v[q + 3]), pack_bf16(v[q + 4], v[q + 5]),
                       pack_bf16(v[q + 6], v[q + 7]));
}
// ... and into its transpose, the K-major operand [features][samples] of `rows`
// features (neighbouring lanes hold neighbouring samples: they swap every other
// column, so that each stores two samples of one feature at once).
template <int N>
__device__ __forceinline__ void store_col(uint8_t *dst, int rows, int row, int c0, const float (&v)[N]) {
    const bool odd = row & 1;
#pragma unroll
    for (int q = 0; q < N; q += 2) {
        const float other = __shfl_xor_sync(0xffffffffu, odd ? v[q] : v[q + 1], 1);
        const uint32_t w = odd ? pack_bf16(other, v[q + 1]) : pack_bf16(v[q], other);
        *reinterpret_cast<uint32_t *>(dst + tc::kmajor_off(c0 + q + (odd ? 1 : 0), row & ~1, rows)) = w;
    }
}
// D[tmem] = A B^T over K, issued by one thread.
__device__ __forceinline__ void issue(uint32_t tmem, const uint8_t *a, int arows, const uint8_t *b, int brows, int K) {
    const uint32_t lbo_a = tc::kmajor_lbo(arows), lbo_b = tc::kmajor_lbo(brows);
    const uint32_t idesc = tc::idesc_bf16(arows, brows);
    for (int ks = 0; ks < K / 16; ++ks)
        tc::mma_bf16(tmem, tc::smem_desc(tc::smem_addr(a) + ks * 2 * lbo_a, lbo_a, tc::kSbo),
                     tc::smem_desc(tc::smem_addr(b) + ks * 2 * lbo_b, lbo_b, tc::kSbo), idesc, ks > 0 ? 1u : 0u);
}
// Shared-memory writes of all threads become visible to the tensor cores.
__device__ __forceinline__ void publish() {
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
}
// The MMAs committed on the phase have completed (uniform over the block).
__device__ __forceinline__ bool arrived(uint64_t *mbar, uint32_t &phase) {
    const bool ok = __syncthreads_and(tc::mbar_wait(mbar, phase, kSpins)) != 0;
    phase ^= 1;
    tc::fence_after_sync();
    return ok;
}
// Hidden activations gelu(acc + bias) of columns c0.. (kGroupCols) of the thread's row.
__device__ __forceinline__ void hidden(uint32_t taddr, const float *__restrict__ bias, int c0, float (&h)[kGroupCols]) {
#pragma unroll
    for (int c = 0; c < kGroupCols; c += 16) {
        float acc[16];
        tc::tmem_ld16(taddr + (uint32_t)(c0 + c), acc);
#pragma unroll
        for (int q = 0; q < 16; ++q) h[c + q] = gelu(acc[q] + __ldg(bias + c0 + c + q));
    }
}

// Forward pass of pd_mlp_forward: each block stages the weights once and works
// through tiles blockIdx.x, blockIdx.x + gridDim.x, ...; two blocks share an
// SM, so that one's loads and activations cover the other's waits.  (128
// threads a tile, the weights staged for each: 49 us for 20,001 samples.)
__global__ void __launch_bounds__(kTileThreads, 2) k_mlp_fwd(Net n, const float *__restrict__ X, float *__restrict__ Y,
                                                            int B, int R) {
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_base;
    uint8_t *sA = sm;                     // X tile   128 x 32  (8 KB)
    uint8_t *sW1 = sm + 8 * 1024;         // W1       128 x 32  (8 KB)
    uint8_t *sH = sm + 16 * 1024;         // H tile   128 x 128 (32 KB)
    uint8_t *sW2 = sm + 48 * 1024;        // W2       128 x 128 (32 KB)
    uint8_t *sW3 = sm + 80 * 1024;        // W3        32 x 128 (8 KB)
    const int tid = threadIdx.x, warp = tid >> 5, wg = warp >> 2, lrow = tid & 127;
    const bool x16 = (reinterpret_cast<uintptr_t>(X) & 15) == 0, y16 = (reinterpret_cast<uintptr_t>(Y) & 15) == 0;
    const bool mine = 32 * (warp & 3) < R;      // the warp's samples belong to the tile
    float x[8];
    if (mine) load_row8(X, blockIdx.x * R + lrow, wg, B, x16, x);
    {
        WeightStage<IN, HID, kTileThreads> w1;
        WeightStage<HID, HID, kTileThreads> w2;
        WeightStage<HID, OUT, kTileThreads> w3;
        w1.load(n.W1, tid);
        w2.load(n.W2, tid);
        w3.load(n.W3, tid);
        if (warp == 0) tc::tmem_alloc(&tmem_base, 128);
        if (tid == 0) tc::mbar_init(&mbar, 1);
        w1.store(sW1, tid);
        w2.store(sW2, tid);
        w3.store(sW3, tid);
    }
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile * R < B && ok; tile += gridDim.x) {
        const int row = tile * R + lrow;
        if (mine) store_row(sA, lrow, 8 * wg, x);
        publish();
        const uint32_t tmem = tmem_base, lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        if (tid == 0) {
            issue(tmem, sA, TILE, sW1, HID, IN);
            tc::mma_commit(&mbar);
        }
        // the next tile's rows meanwhile
        if (mine) load_row8(X, (tile + gridDim.x) * R + lrow, wg, B, x16, x);
        float h[kGroupCols];
        if (!(ok = arrived(&mbar, phase))) break;
        if (mine) {
            hidden(lanes, n.p + OB1, kGroupCols * wg, h);
            store_row(sH, lrow, kGroupCols * wg, h);
        }
        publish();
        if (tid == 0) {
            issue(tmem, sH, TILE, sW2, HID, HID);
            tc::mma_commit(&mbar);
        }
        if (!(ok = arrived(&mbar, phase))) break;
        if (mine) {
            hidden(lanes, n.p + OB2, kGroupCols * wg, h);
            store_row(sH, lrow, kGroupCols * wg, h);
        }
        publish();
        if (tid == 0) {
            issue(tmem, sH, TILE, sW3, OUT, HID);
            tc::mma_commit(&mbar);
        }
        if (!(ok = arrived(&mbar, phase))) break;
        if (mine) {
            float acc[8];
            tc::tmem_ld8(lanes + (uint32_t)(8 * wg), acc);
    #pragma unroll
            for (int q = 0; q < 8; ++q) acc[q] += __ldg(n.p + OB3 + 8 * wg + q);
            if (row < B) {
                float *dst = Y + (size_t)row * OUT + 8 * wg;
                if (y16) {
                    *reinterpret_cast<float4 *>(dst) = make_float4(acc[0], acc[1], acc[2], acc[3]);
                    *reinterpret_cast<float4 *>(dst + 4) = make_float4(acc[4], acc[5], acc[6], acc[7]);
                } else {
    #pragma unroll
                    for (int q = 0; q < 8; ++q) dst[q] = acc[q];
                }
            }
        }
        tc::fence_before_sync();        // (the accumulators are read before the next tile's MMAs, behind publish())
    }
    if (!ok) {
        // the MMAs committed on the phase that timed out may still be writing the
        // accumulator: one more bounded wait on that phase before the columns are
        // released (the outputs of a timed-out tile are invalid either way: err is set)
        tc::mbar_wait(&mbar, phase ^ 1, kSpins);
        if (tid == 0) atomicExch(n.err, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem_base, 128);
}

// ---------------------------------------------------------------------------
// training

// Sums of v[0..31] over the 32 lanes of the warp: lane l gets the sum of v[l].
// Halving exchange: 31 shuffles instead of 32 butterflies of five.
__device__ __forceinline__ float transpose_sum(float (&v)[32]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int half = 16; half > 0; half >>= 1) {
        const bool up = lane & half;
#pragma unroll
        for (int q = 0; q < half; ++q) {
            const float send = up ? v[q] : v[q + half];
            const float keep = up ? v[q + half] : v[q];
            v[q] = keep + __shfl_xor_sync(0xffffffffu, send, half);
        }
    }
    return v[0];
}

// g (+)= v at n consecutive places (first: overwrite).
template <int N>
__device__ __forceinline__ void add_grad(float *g, const float (&v)[N], bool first) {
#pragma unroll
    for (int q = 0; q < N; q += 4) {
        float4 *at = reinterpret_cast<float4 *>(g + q);
        float4 o = first ? make_float4(0.f, 0.f, 0.f, 0.f) : *at;
        *at = make_float4(o.x + v[q], o.y + v[q + 1], o.z + v[q + 2], o.w + v[q + 3]);
    }
}

// Loss mean((net(X) - T)^2) and its parameter gradients of tiles blockIdx.x,
// blockIdx.x + gridDim.x, ... into this block's partial.  Per tile a chain of
// eight products with nothing in global memory between them: the layers' sums
// stay in tensor memory for the activations' derivatives (columns 0 layer 1,
// 128 layer 2, 256 output, 288 backward signal, 416 dW3, 448 dW1; dW2 takes
// layer 2's once it is used up), activations and signals are kept in shared
// memory both ways round, as the products over features and over samples need
// them (the transposed copies are written from the same registers).  Every
// operand is rounded to BF16 where the separate kernels before rounded it.
// (Those, 25 launches a step with element-wise atomics and 2-byte gathers:
// 915 us a step of 1024 samples.)
__global__ void __launch_bounds__(kTileThreads, 1) k_mlp_grad(Net n, const float *__restrict__ X,
                                                             const float *__restrict__ T, int B, int R) {
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ float s_bias[4][HID];             // per quarter of the samples
    __shared__ float s_loss[kTileThreads / 32];
    uint8_t *sX = sm, *sXt = sm + 8 * 1024;                       // X both ways (8 KB each)
    uint8_t *sW1 = sm + 16 * 1024, *sW3 = sm + 24 * 1024, *sW3t = sm + 32 * 1024;
    uint8_t *sD = sm + 40 * 1024, *sDt = sm + 48 * 1024;          // output signal both ways (8 KB each)
    uint8_t *sW2 = sm + 56 * 1024, *sW2t = sm + 88 * 1024;
    uint8_t *sH = sm + 120 * 1024;               // H1, H2, then the layer-2 signal, sample rows
    uint8_t *sT1 = sm + 152 * 1024;              // H1 transposed, then the layer-1 signal
    uint8_t *sT2 = sm + 184 * 1024;              // H2 transposed, then the layer-2 signal
    const int tid = threadIdx.x, warp = tid >> 5, wg = warp >> 2, lrow = tid & 127, lane = tid & 31, quarter = warp & 3;
    const bool x16 = ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(T)) & 15) == 0;
    const int c0 = kGroupCols * wg;
    float *const part = n.parts + (size_t)blockIdx.x * kPartStride;
    const bool mine = 32 * quarter < R;         // the warp's samples belong to the tile
    float x[8], t[8];
    if (mine) {
        load_row8(X, blockIdx.x * R + lrow, wg, B, x16, x);
        load_row8(T, blockIdx.x * R + lrow, wg, B, x16, t);
    }
    s_bias[quarter][kGroupCols * wg + lane] = 0.f;
    {
        WeightStage<IN, HID, kTileThreads> w1;
        WeightStage<HID, HID, kTileThreads> w2, w2t;
        WeightStage<HID, OUT, kTileThreads> w3;
        WeightStage<OUT, HID, kTileThreads> w3t;
        w1.load(n.W1, tid);
        w2.load(n.W2, tid);
        w3.load(n.W3, tid);
        w2t.load(n.W2t, tid);
        w3t.load(n.W3t, tid);
        if (warp == 0) tc::tmem_alloc(&tmem_base, 512);
        if (tid == 0) tc::mbar_init(&mbar, 1);
        w1.store(sW1, tid);
        w2.store(sW2, tid);
        w3.store(sW3, tid);
        w2t.store(sW2t, tid);
        w3t.store(sW3t, tid);
    }
    tc::grid_dep_launch();
    uint32_t phase = 0;
    bool ok = true, first = true;
    float loss = 0.f;
    const float scale = (float)(B * OUT);
    for (int tile = blockIdx.x; tile * R < B && ok; tile += gridDim.x, first = false) {
        const int row = tile * R + lrow;
        if (mine) {
            store_row(sX, lrow, 8 * wg, x);
            store_col(sXt, IN, lrow, 8 * wg, x);
        }
        publish();
        const uint32_t tmem = tmem_base, lanes = tmem + ((uint32_t)(quarter * 32) << 16);
        float h[kGroupCols], d8[8];
        auto run = [&](auto mmas) {
            if (tid == 0) {
                mmas();
                tc::mma_commit(&mbar);
            }
            return ok = arrived(&mbar, phase);
        };
        // forward
        if (!run([&] { issue(tmem, sX, TILE, sW1, HID, IN); })) break;
        if (mine) {
            hidden(lanes, n.p + OB1, c0, h);
            store_row(sH, lrow, c0, h);
            store_col(sT1, HID, lrow, c0, h);
        }
        publish();
        if (!run([&] { issue(tmem + 128, sH, TILE, sW2, HID, HID); })) break;
        if (mine) {
            hidden(lanes + 128, n.p + OB2, c0, h);
            store_row(sH, lrow, c0, h);
            store_col(sT2, HID, lrow, c0, h);
        }
        publish();
        if (!run([&] { issue(tmem + 256, sH, TILE, sW3, OUT, HID); })) break;
        // output signal dL/dY, loss
        if (mine) {
            tc::tmem_ld8(lanes + 256u + (uint32_t)(8 * wg), d8);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float e = row < B ? (d8[q] + __ldg(n.p + OB3 + 8 * wg + q)) - t[q] : 0.f;
                d8[q] = 2.f * e / scale;
                loss += e * e;
            }
            store_row(sD, lrow, 8 * wg, d8);
            store_col(sDt, OUT, lrow, 8 * wg, d8);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float v = d8[q];
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                if (lane == 0) s_bias[quarter][8 * wg + q] = v;
            }
        }
        publish();
        if (tid < OUT) {
            const float v[4] = {s_bias[0][tid], s_bias[1][tid], s_bias[2][tid], s_bias[3][tid]};
            float *g = part + OB3 + tid;
            *g = (first ? 0.f : *g) + ((v[0] + v[1]) + (v[2] + v[3]));
        }
        // the next tile's rows meanwhile
        if (mine) {
            load_row8(X, (tile + gridDim.x) * R + lrow, wg, B, x16, x);
            load_row8(T, (tile + gridDim.x) * R + lrow, wg, B, x16, t);
        }
        // dW3^T = H2^T dY and dH2 = dY W3; dZ2 = dH2 gelu'(Z2)
        if (!run([&] {
                issue(tmem + 416, sT2, HID, sDt, OUT, R);
                issue(tmem + 288, sD, TILE, sW3t, HID, OUT);
            }))
            break;
        auto signal = [&](uint32_t zcol, const float *__restrict__ bias) {
#pragma unroll
            for (int c = 0; c < kGroupCols; c += 16) {
                float z[16], g[16];
                tc::tmem_ld16(lanes + zcol + (uint32_t)(c0 + c), z);
                tc::tmem_ld16(lanes + 288u + (uint32_t)(c0 + c), g);
#pragma unroll
                for (int q = 0; q < 16; ++q)
                    h[c + q] = row < B ? g[q] * gelu_grad(z[q] + __ldg(bias + c0 + c + q)) : 0.f;
            }
        };
        static_assert(kGroupCols == 32, "one column a lane in the bias sums");
        auto bias_add = [&](float *g) {
            if (tid < HID) g[tid] = (first ? 0.f : g[tid]) + ((s_bias[0][tid] + s_bias[1][tid]) + (s_bias[2][tid] + s_bias[3][tid]));
        };
        if (mine) {
            signal(128u, n.p + OB2);
            store_row(sH, lrow, c0, h);
            store_col(sT2, HID, lrow, c0, h);
            s_bias[quarter][c0 + lane] = transpose_sum(h);
        }
        publish();
        bias_add(part + OB2);
        // dW2 = dZ2^T H1 and dH1 = dZ2 W2; dZ1 = dH1 gelu'(Z1)
        if (!run([&] {
                issue(tmem + 128, sT2, HID, sT1, HID, R);
                issue(tmem + 288, sH, TILE, sW2t, HID, HID);
            }))
            break;
        if (mine) {
            signal(0u, n.p + OB1);
            store_col(sT1, HID, lrow, c0, h);
            s_bias[quarter][c0 + lane] = transpose_sum(h);
        }
        publish();
        bias_add(part + OB1);
        // dW1 = dZ1^T X
        if (!run([&] { issue(tmem + 448, sT1, HID, sXt, IN, R); })) break;
        // the weight gradients: TMEM lane = row of the product
        {
            float v[16];
#pragma unroll
            for (int c = 0; c < kGroupCols; c += 16) {
                tc::tmem_ld16(lanes + 128u + (uint32_t)(c0 + c), v);
                add_grad(part + OW2 + lrow * HID + c0 + c, v, first);
            }
            float w[8];
            tc::tmem_ld8(lanes + 448u + (uint32_t)(8 * wg), w);
            add_grad(part + OW1 + lrow * IN + 8 * wg, w, first);
            tc::tmem_ld8(lanes + 416u + (uint32_t)(8 * wg), w);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float *g = part + OW3 + (8 * wg + q) * HID + lrow;
                *g = (first ? 0.f : *g) + w[q];
            }
        }
        tc::fence_before_sync();        // (behind publish() before the next tile's MMAs)
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
    if (lane == 0) s_loss[warp] = loss;
    if (!ok) {
        tc::mbar_wait(&mbar, phase ^ 1, kSpins);     // as in k_mlp_fwd
        if (tid == 0) atomicExch(n.err, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem_base, 512);
    if (tid == 0) {
        float l = 0.f;
        for (int w = 0; w < kTileThreads / 32; ++w) l += s_loss[w];
        part[NPARAM] = l / scale;
    }
}

// BF16 copies of parameter i for the MMAs: [out][in] and transposed [in][out].
__device__ __forceinline__ void store_bf16(const Net &n, int i, float p) {
    const __nv_bfloat16 w = __float2bfloat16(p);
    if (i < OB1) {
        n.W1[i - OW1] = w;
    } else if (i >= OW2 && i < OB2) {
        const int e = i - OW2;
        n.W2[e] = w;
        n.W2t[(e % HID) * HID + e / HID] = w;
    } else if (i >= OW3 && i < OB3) {
        const int e = i - OW3;
        n.W3[e] = w;
        n.W3t[(e % HID) * OUT + e / HID] = w;
    }
}

// The tiles' gradients (n_parts partials, in order) and loss summed; with adam,
// the parameter update and its BF16 copies, else the gradient into n.g.
__global__ void __launch_bounds__(128) k_mlp_update(Net n, int n_parts, int adam, float lr, float b1, float b2, float eps,
                                                    float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    float p = 0.f, m = 0.f, v = 0.f;
    if (adam && i < NPARAM) {
        p = n.p[i];
        m = n.m[i];
        v = n.v[i];
    }
    tc::grid_dep_wait();
    if (i > NPARAM) return;
    float g = 0.f;
    constexpr int kBatch = 8;
    for (int q0 = 0; q0 < n_parts; q0 += kBatch) {
        float a[kBatch];
#pragma unroll
        for (int q = 0; q < kBatch; ++q) a[q] = q0 + q < n_parts ? n.parts[(size_t)(q0 + q) * kPartStride + i] : 0.f;
#pragma unroll
        for (int q = 0; q < kBatch; ++q) g += a[q];
    }
    if (i == NPARAM) {
        n.loss[0] = g;
        return;
    }
    if (!adam) {
        n.g[i] = g;
        return;
    }
    m = b1 * m + (1.f - b1) * g;
    v = b2 * v + (1.f - b2) * g * g;
    n.m[i] = m;
    n.v[i] = v;
    p -= lr * (m / c1) / (sqrtf(v / c2) + eps);
    n.p[i] = p;
    store_bf16(n, i, p);
}

__global__ void k_to_bf16(Net n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NPARAM) store_bf16(n, i, n.p[i]);
}

// Inference of several networks in one launch (the surrogate's step): tile
// blockIdx.x is rows [w.y, min(w.y + 128, w.z)) of X / Y through network
// refs[w.x].  The MMAs are those of fwd_tile; operand staging and the layer
// epilogues are spread over four warpgroups: warp w reads TMEM lanes
// 32 (w % 4) .. 32 (w % 4) + 31 (its quarter of the rows) and warpgroup g
// takes the g-th quarter of a hidden layer's columns, so four warps per
// scheduler hide the latency of the activation chains and of the loads.  The
// activation is the GELU with the error function of Abramowitz & Stegun
// 7.1.26 (branch-free; its 1.5e-7 error is far below the BF16 rounding of
// the activations).  With r.lin the output is the surrogate's modal force
// f = net(q) - Lambda q.
constexpr int kInferThreads = 512;
constexpr int kInferGroups = kInferThreads / TILE;

__global__ void __launch_bounds__(kInferThreads) k_mlp_infer(const MlpRef *__restrict__ refs,
                                                             const int4 *__restrict__ work,
                                                             const float *__restrict__ X, float *__restrict__ Y,
                                                             int *err) {
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_base;
    uint8_t *sA = sm;                     // X tile   128 x 32  (8 KB)
    uint8_t *sW1 = sm + 8 * 1024;         // W1       128 x 32  (8 KB)
    uint8_t *sH = sm + 16 * 1024;         // H tile   128 x 128 (32 KB)
    uint8_t *sW2 = sm + 48 * 1024;        // W2       128 x 128 (32 KB)
    uint8_t *sW3 = sm + 80 * 1024;        // W3        32 x 128 (8 KB)
    const int4 wk = work[blockIdx.x];
    const MlpRef r = refs[wk.x];
    const float *P = r.p, *lin = r.lin;
    const int B = wk.z;
    const int tid = threadIdx.x, warp = tid >> 5, wg = warp >> 2;
    const int lrow = tid & 127;           // = 32 (warp % 4) + lane: the TMEM lane of the thread
    const int row = wk.y + lrow;
    if (tid == 0) tc::mbar_init(&mbar, 1);
    static_assert(IN == 8 * kInferGroups, "one 8-column piece of the input row per warpgroup");
    float *sX = reinterpret_cast<float *>(sm + 88 * 1024);   // input rows in FP32, 128 x 32 (16 KB)
    {
        // every load first: the thread's pieces of the three weight matrices
        // (while the kernel that writes the inputs may still run), then the
        // row's input columns 8 wg .. 8 wg + 7; then the stores
        WeightStage<IN, HID, kInferThreads> w1;
        WeightStage<HID, HID, kInferThreads> w2;
        WeightStage<HID, OUT, kInferThreads> w3;
        w1.load(static_cast<const __nv_bfloat16 *>(r.W1), tid);
        w2.load(static_cast<const __nv_bfloat16 *>(r.W2), tid);
        w3.load(static_cast<const __nv_bfloat16 *>(r.W3), tid);
        tc::grid_dep_wait();
        if (warp == 0) tc::tmem_alloc(&tmem_base, 128);
        float4 x0 = make_float4(0.f, 0.f, 0.f, 0.f), x1 = x0;
        if (row < B) {
            const float4 *src = reinterpret_cast<const float4 *>(X + (size_t)row * IN + 8 * wg);
            x0 = src[0];
            x1 = src[1];
        }
        const float x[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
        __align__(16) __nv_bfloat16 xb[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            xb[q] = __float2bfloat16(x[q]);
            sX[lrow * IN + 8 * wg + q] = x[q];
        }
        *reinterpret_cast<uint4 *>(sA + tc::kmajor_off(lrow, 8 * wg, TILE)) = *reinterpret_cast<const uint4 *>(xb);
        w1.store(sW1, tid);
        w2.store(sW2, tid);
        w3.store(sW3, tid);
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    tc::grid_dep_launch();
    const uint32_t tmem = tmem_base;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    constexpr int kCols = HID / kInferGroups;            // hidden columns per warpgroup
    static_assert(kCols % 16 == 0 && OUT / 16 <= kInferGroups, "16-column TMEM loads");
    bool ok = true;
    uint32_t phase = 0;
    for (int layer = 0; layer < 3 && ok; ++layer) {
        const int K = layer == 0 ? IN : HID;
        const int N = layer == 2 ? OUT : HID;
        uint8_t *a = layer == 0 ? sA : sH;
        uint8_t *b = layer == 0 ? sW1 : (layer == 1 ? sW2 : sW3);
        if (tid == 0) {
            const uint32_t lbo_a = tc::kmajor_lbo(TILE), lbo_b = tc::kmajor_lbo(N);
            const uint32_t idesc = tc::idesc_bf16(TILE, N);
            for (int ks = 0; ks < K / 16; ++ks) {
                const uint64_t ad = tc::smem_desc(tc::smem_addr(a) + ks * 2 * lbo_a, lbo_a, tc::kSbo);
                const uint64_t bd = tc::smem_desc(tc::smem_addr(b) + ks * 2 * lbo_b, lbo_b, tc::kSbo);
                tc::mma_bf16(tmem, ad, bd, idesc, ks > 0 ? 1u : 0u);
            }
            tc::mma_commit(&mbar);
        }
        ok = __syncthreads_and(tc::mbar_wait(&mbar, phase, kSpins)) != 0;   // uniform outcome
        phase ^= 1;
        if (!ok) break;
        tc::fence_after_sync();
        const float *bias = P + (layer == 0 ? OB1 : (layer == 1 ? OB2 : OB3));
        if (layer < 2) {
            // hidden layer: columns kCols wg .. kCols (wg + 1) of the thread's row
#pragma unroll
            for (int c0 = kCols * wg; c0 < kCols * (wg + 1); c0 += 16) {
                float acc[16];
                tc::tmem_ld16(tmem + lane_base + (uint32_t)c0, acc);
                __align__(16) __nv_bfloat16 hb[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) hb[q] = __float2bfloat16(gelu_fast(acc[q] + bias[c0 + q]));
                *reinterpret_cast<uint4 *>(sH + tc::kmajor_off(lrow, c0, TILE)) = *reinterpret_cast<const uint4 *>(hb);
                *reinterpret_cast<uint4 *>(sH + tc::kmajor_off(lrow, c0 + 8, TILE)) =
                    *reinterpret_cast<const uint4 *>(hb + 8);
            }
        } else if (wg < OUT / 16) {
            // output layer: 16 columns per warpgroup (the first OUT / 16 groups; warp-uniform)
            const int c0 = 16 * wg;
            float acc[16];
            tc::tmem_ld16(tmem + lane_base + (uint32_t)c0, acc);
            if (row < B) {
                // y = z - lin (.) x with x from the staged rows; 16-byte stores
                float y[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const int c = c0 + q;
                    const float z = acc[q] + bias[c];
                    y[q] = lin ? z - lin[c] * sX[lrow * IN + c] : z;
                }
                float4 *dst = reinterpret_cast<float4 *>(Y + (size_t)row * OUT + c0);
#pragma unroll
                for (int q = 0; q < 16; q += 4) dst[q / 4] = make_float4(y[q], y[q + 1], y[q + 2], y[q + 3]);
            }
        }
        tc::fence_before_sync();
        tc::fence_async_smem();
        __syncthreads();
        tc::fence_after_sync();
    }
    if (!ok) {
        // the MMAs committed on the phase that timed out may still be writing the
        // accumulator: one more bounded wait on that phase before the columns are
        // released (the outputs of a timed-out tile are invalid either way: err is set)
        tc::mbar_wait(&mbar, phase ^ 1, kSpins);
        if (tid == 0) atomicExch(err, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem_base, 128);
}

}  // namespace mlp
}  // namespace pd

// ===========================================================================
// host side

using namespace pd::mlp;

struct pd_mlp {
    cudaStream_t stream = nullptr;
    int max_batch = 0, Bp = 0;
    Net n{};
    bool bound = false;
    int adam_t = 0;
    float *got = nullptr;       // page-locked: the loss and error word on the host
};

namespace {

size_t al(size_t x) { return (x + 255) & ~size_t(255); }

template <class T>
void carve(char *base, size_t &off, T *&p, size_t count) {
    p = base ? reinterpret_cast<T *>(base + off) : nullptr;
    off = al(off + sizeof(T) * std::max<size_t>(count, 1));
}

size_t mlp_layout(pd_mlp *m, char *base) {
    size_t off = 0;
    Net &n = m->n;
    carve(base, off, n.p, NPARAM);
    carve(base, off, n.g, NPARAM);
    carve(base, off, n.m, NPARAM);
    carve(base, off, n.v, NPARAM);
    carve(base, off, n.W1, HID * IN);
    carve(base, off, n.W2, HID * HID);
    carve(base, off, n.W3, OUT * HID);
    carve(base, off, n.W2t, HID * HID);
    carve(base, off, n.W3t, OUT * HID);
    carve(base, off, n.parts, (size_t)std::min(m->Bp / 32, kParts) * kPartStride);
    carve(base, off, n.loss, 2);
    n.err = reinterpret_cast<int *>(n.loss + 1);
    return off;
}

#define MLP_CUDA(call)                                                                          \
    do {                                                                                        \
        cudaError_t e_ = (call);                                                                \
        if (e_ != cudaSuccess) return pd::set_error(PD_ECUDA, cudaGetErrorString(e_));          \
    } while (0)

// Waits for the stream; loss (nullable) and the error word in one copy.
int finish(pd_mlp *m, float *loss) {
    static_assert(sizeof(int) == sizeof(float), "error word beside the loss");
    MLP_CUDA(cudaMemcpyAsync(m->got, m->n.loss, 2 * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
    MLP_CUDA(cudaStreamSynchronize(m->stream));
    int err;
    std::memcpy(&err, &m->got[1], sizeof(err));
    if (loss) *loss = m->got[0];
    if (err) return pd::set_error(PD_ETIMEOUT, "tensor-core wait timed out");
    return PD_OK;
}

// Samples per tile: the fewest (32, 64, .. most) with which `blocks` tiles take the batch.
int tile_rows(int batch, int blocks, int most) {
    int rows = 32;
    while (rows < most && (long long)rows * blocks < batch) rows *= 2;
    return rows;
}

int forward(pd_mlp *m, const float *x, float *y, int batch, cudaStream_t s) {
    if (batch < 0 || batch > m->max_batch) return pd::set_error(PD_EINVAL, "batch exceeds max_batch");
    if (batch == 0) return PD_OK;
    // (one tile a block, two blocks an SM, up to 128 samples a tile, then several:
    // 50,001 samples take 29 us so, 46 and 56 us with 64 and 32 at most)
    const int rows = tile_rows(batch, 2 * kParts, TILE), tiles = (batch + rows - 1) / rows;
    pd::mlp::k_mlp_fwd<<<std::min(tiles, 2 * kParts), kTileThreads, kFwdSmem, s>>>(m->n, x, y, batch, rows);
    MLP_CUDA(cudaGetLastError());
    return PD_OK;
}

// Loss and gradients of a batch, then the Adam step (adam_t > 0) or n.g.
int backward(pd_mlp *m, const float *x, const float *t, int batch, float lr, int adam_t) {
    // (one tile a block up to 128 samples a tile, then several)
    const int rows = tile_rows(batch, kParts, TILE), parts = std::min((batch + rows - 1) / rows, kParts);
    pd::mlp::k_mlp_grad<<<parts, kTileThreads, kTrainSmem, m->stream>>>(m->n, x, t, batch, rows);
    MLP_CUDA(cudaGetLastError());
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)adam_t), c2 = 1.f - std::pow(b2, (float)adam_t);
    MLP_CUDA(pd::launch_ex(pd::mlp::k_mlp_update, dim3((NPARAM + 1 + 127) / 128), dim3(128), 0, m->stream, true, m->n,
                           parts, adam_t > 0 ? 1 : 0, lr, b1, b2, 1e-8f, c1, c2));
    return PD_OK;
}

}  // namespace

int pd::mlp_ref(pd_mlp *m, MlpRef *out) {
    if (!m || !m->bound || !out) return pd::set_error(PD_ESTATE, "mlp not bound");
    out->W1 = m->n.W1;
    out->W2 = m->n.W2;
    out->W3 = m->n.W3;
    out->p = m->n.p;
    out->lin = nullptr;
    return PD_OK;
}

cudaError_t pd::launch_mlp_grouped(const MlpRef *refs, const int4 *work, int n_work, const float *x, float *y,
                                   int *err, cudaStream_t s, bool pdl) {
    if (n_work == 0) return cudaSuccess;
    static_assert(sizeof(MlpRef) == 40, "MlpRef layout");
    static_assert(88 * 1024 + 128 * PD_MLP_IN * 4 <= kFwdSmem, "inference tile and its input rows fit");
    // rows of 32 floats: 16-byte aligned when the arrays are
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15) return cudaErrorMisalignedAddress;
    return launch_ex(pd::mlp::k_mlp_infer, dim3(n_work), dim3(pd::mlp::kInferThreads), kFwdSmem, s, pdl, refs, work,
                     x, y, err);
}

cudaError_t pd::mlp_init_attributes() {
    return cudaFuncSetAttribute(pd::mlp::k_mlp_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem);
}

int pd::mlp_forward_stream(pd_mlp *m, const float *x, float *y, int batch, cudaStream_t s) {
    if (!m || !m->bound) return pd::set_error(PD_ESTATE, "mlp not bound");
    return forward(m, x, y, batch, s);
}

extern "C" {

int pd_mlp_create(pd_mlp **out, int max_batch, void *cuda_stream) {
    if (!out || max_batch < 1 || max_batch > (1 << 22)) return pd::set_error(PD_EINVAL, "max_batch in [1, 4194304]");
    pd_mlp *m = new (std::nothrow) pd_mlp();
    if (!m) return pd::set_error(PD_ENOMEM, "out of host memory");
    m->stream = (cudaStream_t)cuda_stream;
    m->max_batch = max_batch;
    m->Bp = ((max_batch + TILE - 1) / TILE) * TILE;
    *out = m;
    return PD_OK;
}

int pd_mlp_destroy(pd_mlp *m) {
    if (m) {
        if (m->bound) cudaStreamSynchronize(m->stream);
        if (m->got) cudaFreeHost(m->got);
        delete m;
    }
    return PD_OK;
}

int pd_mlp_arena_bytes(pd_mlp *m, size_t *bytes) {
    if (!m || !bytes) return pd::set_error(PD_EINVAL, "null argument");
    *bytes = mlp_layout(m, nullptr);
    return PD_OK;
}

int pd_mlp_bind_arena(pd_mlp *m, void *dev, size_t bytes) {
    if (!m || !dev || ((uintptr_t)dev & 255)) return pd::set_error(PD_EINVAL, "arena null or not 256-byte aligned");
    if (bytes < mlp_layout(m, nullptr)) return pd::set_error(PD_EINVAL, "arena too small");
    mlp_layout(m, (char *)dev);
    MLP_CUDA(cudaFuncSetAttribute(pd::mlp::k_mlp_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem));
    MLP_CUDA(cudaFuncSetAttribute(pd::mlp::k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, kTrainSmem));
    if (!m->got) MLP_CUDA(cudaMallocHost(reinterpret_cast<void **>(&m->got), 2 * sizeof(float)));
    MLP_CUDA(cudaMemsetAsync(dev, 0, bytes, m->stream));
    m->bound = true;
    return PD_OK;
}

int pd_mlp_set_params(pd_mlp *m, const float *params) {
    if (!m || !m->bound || !params) return pd::set_error(PD_ESTATE, "mlp not bound or null params");
    MLP_CUDA(cudaMemcpyAsync(m->n.p, params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, m->stream));
    MLP_CUDA(cudaMemsetAsync(m->n.m, 0, sizeof(float) * NPARAM, m->stream));
    MLP_CUDA(cudaMemsetAsync(m->n.v, 0, sizeof(float) * NPARAM, m->stream));
    pd::mlp::k_to_bf16<<<(NPARAM + 255) / 256, 256, 0, m->stream>>>(m->n);
    MLP_CUDA(cudaGetLastError());
    MLP_CUDA(cudaStreamSynchronize(m->stream));
    m->adam_t = 0;
    return PD_OK;
}

int pd_mlp_get_params(pd_mlp *m, float *params) {
    if (!m || !m->bound || !params) return pd::set_error(PD_ESTATE, "mlp not bound or null params");
    MLP_CUDA(cudaMemcpyAsync(params, m->n.p, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, m->stream));
    MLP_CUDA(cudaStreamSynchronize(m->stream));
    return PD_OK;
}

int pd_mlp_forward(pd_mlp *m, const float *x, float *y, int batch) {
    if (!m || !m->bound) return pd::set_error(PD_ESTATE, "mlp not bound");
    if (batch > 0 && (!x || !y)) return pd::set_error(PD_EINVAL, "null input/output");
    return forward(m, x, y, batch, m->stream);
}

int pd_mlp_loss_grad(pd_mlp *m, const float *x, const float *t, int batch, float *loss, float *grad) {
    if (!m || !m->bound) return pd::set_error(PD_ESTATE, "mlp not bound");
    if (batch < 1 || batch > m->max_batch || !x || !t) return pd::set_error(PD_EINVAL, "bad batch or null input");
    if (int r = backward(m, x, t, batch, 0.f, 0)) return r;
    if (grad) MLP_CUDA(cudaMemcpyAsync(grad, m->n.g, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, m->stream));
    return finish(m, loss);
}

int pd_mlp_train_step(pd_mlp *m, const float *x, const float *t, int batch, float lr, float *loss) {
    if (!m || !m->bound) return pd::set_error(PD_ESTATE, "mlp not bound");
    if (batch < 1 || batch > m->max_batch || !x || !t) return pd::set_error(PD_EINVAL, "bad batch or null input");
    m->adam_t += 1;
    if (int r = backward(m, x, t, batch, lr, m->adam_t)) return r;
    return loss ? finish(m, loss) : PD_OK;
}

}  // extern "C"
