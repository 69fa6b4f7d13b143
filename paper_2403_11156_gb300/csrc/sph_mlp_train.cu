// sph_mlp_train.cu -- training of the warm-start network on the GPU: forward and backward
// of the mean-squared error on tcgen05 tensor cores (BF16 operands, FP32 accumulation in
// tensor memory), Adam updates of the FP32 master weights, and the feature / label
// standardisation statistics.  Per tile of 128 samples:
//   forward   D1 = F W1^T, a1 = gelu(z1);  D2 = a1 W2^T, a2 = gelu(z2);  y = a2 . W3 + b3
//   backward  dy = 2 (y - t) / B;  delta2 = dy W3 gelu'(z2);  D3 = delta2 W2 (-> delta1)
//             [delta2 | delta1]^T [a1 | F] as one MMA over the sample dimension: rows 0-63 x
//             columns 0-63 are dW2, rows 64-127 x columns 64-67 are dW1
// A CTA walks its tiles with the weight gradients accumulating in tensor memory and the
// vector gradients in registers, and adds them to the result once, with FP32 atomics
// (training does not need a bit-reproducible order); the loss sum in FP64.
#include <cuda_bf16.h>

#include <algorithm>

#include "sph.h"
#include "sph_gelu.cuh"
#include "sph_internal.cuh"
#include "sph_sweep.cuh"
#include "sph_tc.cuh"

namespace sph {

namespace {

constexpr int kH = 64;
constexpr int kF = 4;
constexpr int kOffW1 = 0;
constexpr int kOffB1 = kOffW1 + kH * kF;
constexpr int kOffW2 = kOffB1 + kH;
constexpr int kOffB2 = kOffW2 + kH * kH;
constexpr int kOffW3 = kOffB2 + kH;
constexpr int kOffB3 = kOffW3 + kH;
constexpr int kNW = kOffB3 + 1;
constexpr int kOffMuF = kNW;
constexpr int kOffSdF = kOffMuF + kF;
constexpr int kOffMuY = kOffSdF + kF;
constexpr int kOffSdY = kOffMuY + 1;
static_assert(kOffSdY + 1 == SPH_MLP_PARAMS, "parameter block layout");
static_assert(kNW == SPH_MLP_WEIGHTS, "weight count");

// shared-memory map (bytes) of one CTA.  Both operand tiles keep a sample's row of columns
// contiguous in core matrices of 8 samples x 8 columns, so the same bytes serve as a
// K-major operand (K = columns: the layers) and as an M/N-major one (K = samples: the weight
// gradients), without a transposed copy.
constexpr int kThreads = 256;          // two threads a row, 32 columns each
constexpr uint32_t kColsD = 128;       // delta tile: delta2 | delta1
constexpr uint32_t kColsA = 80;        // activation tile: a1 | F (4 features, 12 zeros)
constexpr uint32_t kSmD = 0;                               // 128 x 128
constexpr uint32_t kSmA = kSmD + 128 * kColsD * 2;         // 128 x 80
constexpr uint32_t kSmW1 = kSmA + 128 * kColsA * 2;        // 64 x 16  W1 (o x f)
constexpr uint32_t kSmW2 = kSmW1 + 64 * 16 * 2;            // 64 x 64  W2 (o x k)
constexpr uint32_t kSmVec = kSmW2 + 64 * 64 * 2;           // b1 / 2, b2 / 2, w3 (float[64] each)
constexpr uint32_t kSmY = kSmVec + 3 * 64 * 4;             // two partial outputs a row
constexpr uint32_t kSmRed = kSmY + 2 * 128 * 4;            // per warp: dW3, db2, db1 of its 32 columns
constexpr uint32_t kSmSum = kSmRed + 8 * 3 * 32 * 4;       // per warp: db3, and the loss (FP64)
constexpr uint32_t kSmBar = kSmSum + 8 * 16;
constexpr uint32_t kSmTmem = kSmBar + 8;
// requested: caps residency at two CTAs per SM, whose 256 tensor-memory columns each fill
// the SM's 512
constexpr uint32_t kSmem = 100 * 1024;
static_assert(kSmTmem + 4 <= kSmem, "shared-memory map");
constexpr int kCtasPerSm = 2;
constexpr uint32_t kCols = 256;        // tensor memory: z1 | z2, later delta2 W2 | gradients
constexpr uint32_t kColZ2 = 64, kColG = 128;
constexpr uint32_t kWaitLimit = 1u << 20;

__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ void store8(unsigned char *tile, uint32_t r, uint32_t k0, uint32_t K, const float *v)
{
    *reinterpret_cast<uint4 *>(tile + tc::tile_offset(r, k0, K)) =
        make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
}
__device__ __forceinline__ void sync_for_mma()
{
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
}

// Index of the sample in row r of batch position p: a bijection of [0, n) per epoch.
__device__ __forceinline__ int64_t permute(int64_t p, int64_t n, uint64_t a, uint64_t c)
{
    return (int64_t)(((uint64_t)p * a + c) % (uint64_t)n);
}

// Sums of 32 columns over the warp's 32 rows: v[k] is this lane's value of column k; lane l
// gets the sum of column l (recursive halving, 31 shuffles).
__device__ __forceinline__ float column_sums(float (&v)[32])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const float keep = up ? v[k + o] : v[k], give = up ? v[k] : v[k + o];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    return v[0];
}

// grad[0..3] += v (16-byte aligned, or element by element).
__device__ __forceinline__ void add4(float *g, const float *v, bool vec)
{
    if (vec) {
        asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(g), "f"(v[0]), "f"(v[1]),
                     "f"(v[2]), "f"(v[3])
                     : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) atomicAdd(g + k, v[k]);
    }
}

// gelu and its derivative of a pair z = 2 h by the library's erff.
__device__ __forceinline__ void gelu_grad_erff(float h0, float h1, gelu::f2 &g, gelu::f2 &d)
{
    float a[2], b[2];
    const float z[2] = {2.0f * h0, 2.0f * h1};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float e = erff(z[k] * 0.70710678118654752f);
        a[k] = 0.5f * z[k] * (1.0f + e);
        b[k] = 0.5f * (1.0f + e) + z[k] * 0.39894228040143268f * __expf(-0.5f * z[k] * z[k]);
    }
    g = gelu::pk(a[0], a[1]);
    d = gelu::pk(b[0], b[1]);
}

// Gradient of the batch's mean squared error (standardised features and labels).  A
// persistent grid of at most two CTAs per SM walks 128-sample tiles; warps w and w + 4 share
// the rows of tensor-memory lanes 32 (w mod 4) and take 32 of the 64 columns each.  Bound by
// the CUDA-core work of 64 x 4 GELU-like terms a sample; the column sums run as 31 shuffles
// per 32 columns.  200,000 samples: 56 us (86 TFLOP/s), 6,950 us before, when every row added
// its 192 terms to 192 shared words atomically, each tile added 4.5k weight gradients to
// memory and the transposed copies of the operands held a CTA at 146 KB.
// One gradient (ONCE) takes the polynomial GELU.  Training keeps erff and one summation order
// of the output: Adam divides by the gradient's own size, so that over hundreds of steps a
// last-bit change of an activation, where it moves a BF16 operand's rounding, grows a
// thousandfold (small batches are bound by latency, not by the formula).
//
// grad_tiles is the walk of one CTA over its tiles of one batch (every thread calls it); the
// kernels around it own the tensor memory and the mbarrier, whose phase and state a walk carries
// on.  next: the first tile's sample of this thread, loaded by the caller ahead of time.
struct Walk {
    uint32_t phase = 0;   // of the mbarrier
    bool good = true;     // no wait gave up
};
struct Sample {
    float4 f;
    float target;
    bool valid;
};
__device__ __forceinline__ Sample load_sample(const float4 *__restrict__ F, const float *__restrict__ T, int64_t n,
                                              int64_t batch_begin, int64_t batch_size, uint64_t pa, uint64_t pc,
                                              int64_t tile)
{
    const int64_t pos = tile * 128 + (threadIdx.x & 127);
    Sample s{make_float4(0.f, 0.f, 0.f, 0.f), 0.0f, pos < batch_size && batch_begin + pos < n};
    if (s.valid) {
        const int64_t i = permute(batch_begin + pos, n, pa, pc);
        if (threadIdx.x < 128) s.f = F[i];
        s.target = T[i];
    }
    return s;
}

template <bool ONCE>
__device__ __forceinline__ void grad_tiles(unsigned char *sm, Walk &walk, const float *w, const float4 *__restrict__ F,
                                           const float *__restrict__ T, int64_t n, int64_t batch_begin,
                                           int64_t batch_size, uint64_t pa, uint64_t pc, Sample next, float *grad,
                                           double *loss)
{
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int half = warp >> 2, row = t & 127, c0 = 32 * half;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + kSmBar);
    uint32_t *slot = reinterpret_cast<uint32_t *>(sm + kSmTmem);
    float *vb1 = reinterpret_cast<float *>(sm + kSmVec), *vb2 = vb1 + kH, *vw3 = vb2 + kH;
    float *ypart = reinterpret_cast<float *>(sm + kSmY);
    const int64_t ntiles = (batch_size + 127) / 128;
    if ((int64_t)blockIdx.x >= ntiles) return;   // uniform per block
    const float z8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (t < 128) store8(sm + kSmA, t, kH + 8, kColsA, z8);
    if (t < kH) {
        const float u[8] = {w[kOffW1 + 4 * t], w[kOffW1 + 4 * t + 1], w[kOffW1 + 4 * t + 2], w[kOffW1 + 4 * t + 3],
                            0.f, 0.f, 0.f, 0.f};
        store8(sm + kSmW1, t, 0, 16, u);
        store8(sm + kSmW1, t, 8, 16, z8);
        vb1[t] = 0.5f * w[kOffB1 + t];
        vb2[t] = 0.5f * w[kOffB2 + t];
        vw3[t] = w[kOffW3 + t];
    }
    for (int idx = t; idx < kH * 8; idx += kThreads) {
        const int r = idx >> 3, kc = (idx & 7) * 8;
        float u[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) u[q] = w[kOffW2 + r * kH + kc + q];
        store8(sm + kSmW2, r, kc, kH, u);
    }
    // the tensor-memory address is read after the first barrier of the walk below
    const uint32_t sb = tc::smem_addr(sm);
    constexpr uint32_t id_layer = tc::idesc_bf16_f32(128, 64);
    constexpr uint32_t id_layer_t = id_layer | tc::kIdescBMajorN;
    constexpr uint32_t id_grad = tc::idesc_bf16_f32(128, kColsA) | tc::kIdescAMajorM | tc::kIdescBMajorN;
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
    const float b3 = w[kOffB3], inv_b = 1.0f / (float)batch_size;
    uint32_t tmem = 0;
    auto wait_mma = [&]() {
        walk.good = tc::mbar_wait_bounded(bar, walk.phase & 1u, kWaitLimit) && walk.good;
        ++walk.phase;
        tc::fence_after_sync();
    };
    float s_w3 = 0.0f, s_b2 = 0.0f, s_b1 = 0.0f, s_b3 = 0.0f;   // of column c0 + lane; s_b3 of this row
    double s_loss = 0.0;
    bool first = true;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const bool valid = next.valid;
        const float f[8] = {next.f.x, next.f.y, next.f.z, next.f.w, 0.f, 0.f, 0.f, 0.f};
        const float target = next.target;
        if (tile + gridDim.x < ntiles) next = load_sample(F, T, n, batch_begin, batch_size, pa, pc, tile + gridDim.x);
        if (!first) wait_mma();   // the previous tile's gradient MMAs have read both tiles
        if (half == 0) store8(sm + kSmA, row, kH, kColsA, f);
        sync_for_mma();
        tmem = *slot;
        float g1[ONCE ? 1 : 32];   // gelu'(z1), kept to the backward pass (ONCE: taken again there)
        // layer 1: z1 -> columns [0, 64)
        if (t == 0) {
            tc::mma_bf16(tmem, tc::smem_desc(sb + kSmA + (kH / 8) * 128, 128, kColsA * 16),
                         tc::smem_desc(sb + kSmW1, 128, 256), id_layer, 0);
            tc::mma_commit(bar);
        }
        wait_mma();
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float v[16];
            tc::tmem_ld16(tmem + lanes + c0 + c * 16, v);
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const int o = c0 + c * 16 + k;
                const float h0 = fmaf(0.5f, v[k], vb1[o]), h1 = fmaf(0.5f, v[k + 1], vb1[o + 1]);
                if (ONCE) {
                    gelu::upk(gelu::gelu_pair(h0, h1), v[k], v[k + 1]);
                } else {
                    gelu::f2 a, d;
                    gelu_grad_erff(h0, h1, a, d);
                    gelu::upk(a, v[k], v[k + 1]);
                    gelu::upk(d, g1[c * 16 + k], g1[c * 16 + k + 1]);
                }
            }
            store8(sm + kSmA, row, c0 + c * 16, kColsA, v);
            store8(sm + kSmA, row, c0 + c * 16 + 8, kColsA, v + 8);
        }
        sync_for_mma();
        // layer 2: z2 -> columns [64, 128)
        if (t == 0) {
            for (int k = 0; k < 4; ++k)
                tc::mma_bf16(tmem + kColZ2, tc::smem_desc(sb + kSmA + k * 256, 128, kColsA * 16),
                             tc::smem_desc(sb + kSmW2 + k * 256, 128, 1024), id_layer, k > 0);
            tc::mma_commit(bar);
        }
        wait_mma();
        float a2[32], g2[32];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float v[16];
            tc::tmem_ld16(tmem + lanes + kColZ2 + c0 + c * 16, v);
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const int o = c0 + c * 16 + k, q = c * 16 + k;
                gelu::f2 a, d;
                const float h0 = fmaf(0.5f, v[k], vb2[o]), h1 = fmaf(0.5f, v[k + 1], vb2[o + 1]);
                if (ONCE) gelu::gelu_grad_pair(h0, h1, a, d);
                else gelu_grad_erff(h0, h1, a, d);
                gelu::upk(a, a2[q], a2[q + 1]);
                gelu::upk(d, g2[q], g2[q + 1]);
            }
        }
        // y = b3 + w3 . a2, in column order: the second half goes on from the first's sum
        auto dot = [&](float y) {
#pragma unroll
            for (int k = 0; k < 32; ++k) y = fmaf(vw3[c0 + k], a2[k], y);
            return y;
        };
        if (half == 0) ypart[row] = dot(b3);
        else if (ONCE) ypart[128 + row] = dot(0.0f);
        __syncthreads();
        float y;
        if (ONCE) {
            y = ypart[row] + ypart[128 + row];
        } else {
            if (half == 1) ypart[128 + row] = dot(ypart[row]);
            __syncthreads();
            y = ypart[128 + row];
        }
        const float e = valid ? (y - target) : 0.0f;
        const float dy = 2.0f * e * inv_b;
        if (half == 0) {
            s_loss += (double)e * (double)e;
            s_b3 += dy;
        }
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            g2[k] *= dy * vw3[c0 + k];
            a2[k] *= dy;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) store8(sm + kSmD, row, c0 + c * 8, kColsD, g2 + c * 8);
        s_w3 += column_sums(a2);
        s_b2 += column_sums(g2);
        sync_for_mma();
        // delta2 W2 -> columns [64, 128) (z2 has been read)
        if (t == 0) {
            for (int k = 0; k < 4; ++k)
                tc::mma_bf16(tmem + kColZ2, tc::smem_desc(sb + kSmD + k * 256, 128, kColsD * 16),
                             tc::smem_desc(sb + kSmW2 + k * 2048, 1024, 128), id_layer_t, k > 0);
            tc::mma_commit(bar);
        }
        wait_mma();
        float d1[32];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float g[16], z[16];
            tc::tmem_ld16(tmem + lanes + kColZ2 + c0 + c * 16, g);
            if (ONCE) tc::tmem_ld16(tmem + lanes + c0 + c * 16, z);
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const int o = c0 + c * 16 + k, q = c * 16 + k;
                if constexpr (ONCE) {
                    gelu::f2 a, d;
                    gelu::gelu_grad_pair(fmaf(0.5f, z[k], vb1[o]), fmaf(0.5f, z[k + 1], vb1[o + 1]), a, d);
                    gelu::upk(gelu::mul2(d, gelu::pk(g[k], g[k + 1])), d1[q], d1[q + 1]);
                } else {
                    d1[q] = g[k] * g1[q];
                    d1[q + 1] = g[k + 1] * g1[q + 1];
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) store8(sm + kSmD, row, kH + c0 + c * 8, kColsD, d1 + c * 8);
        s_b1 += column_sums(d1);
        sync_for_mma();
        // [delta2 | delta1]^T [a1 | F], accumulated over the CTA's tiles -> columns [128, 208)
        if (t == 0) {
            for (int k = 0; k < 8; ++k)
                tc::mma_bf16(tmem + kColG, tc::smem_desc(sb + kSmD + k * 4096, 2048, 128),
                             tc::smem_desc(sb + kSmA + k * 2560, 1280, 128), id_grad, (!first || k > 0) ? 1u : 0u);
            tc::mma_commit(bar);
        }
        first = false;
    }
    wait_mma();
    const bool vec = (reinterpret_cast<uintptr_t>(grad) & 15u) == 0;
    {
        const int lrow = (warp & 3) * 32 + lane;      // gradient row of this thread
        if (lrow < kH) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float v[16];
                tc::tmem_ld16(tmem + lanes + kColG + c0 + c * 16, v);
#pragma unroll
                for (int k = 0; k < 16; k += 4) add4(grad + kOffW2 + lrow * kH + c0 + c * 16 + k, v + k, vec);
            }
        } else if (half == 0) {
            float v[16];
            tc::tmem_ld16(tmem + lanes + kColG + kH, v);
            add4(grad + kOffW1 + (lrow - kH) * kF, v, vec);
        }
    }
    float *red = reinterpret_cast<float *>(sm + kSmRed);
    red[warp * 96 + lane] = s_w3;
    red[warp * 96 + 32 + lane] = s_b2;
    red[warp * 96 + 64 + lane] = s_b1;
    if (half == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s_b3 += __shfl_xor_sync(0xffffffffu, s_b3, o);
            s_loss += __shfl_xor_sync(0xffffffffu, s_loss, o);
        }
        if (lane == 0) {
            *reinterpret_cast<double *>(sm + kSmSum + warp * 16) = s_loss;
            *reinterpret_cast<float *>(sm + kSmSum + warp * 16 + 8) = s_b3;
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (t < 192) {
        // quantity t / 64 (dW3, db2, db1), column t % 64: the four warps of its half
        const int q = t >> 6, c = t & 63;
        float v = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) v += red[((c >> 5) * 4 + k) * 96 + q * 32 + (c & 31)];
        atomicAdd(&grad[(q == 0 ? kOffW3 : (q == 1 ? kOffB2 : kOffB1)) + c], v);
    }
    if (t == 192) {
        float v = 0.0f;
        double l = 0.0;
        for (int k = 0; k < 4; ++k) {
            l += *reinterpret_cast<double *>(sm + kSmSum + k * 16);
            v += *reinterpret_cast<float *>(sm + kSmSum + k * 16 + 8);
        }
        atomicAdd(&grad[kOffB3], v);
        atomicAdd(loss, l);
    }
    __syncthreads();   // the sums above have been read: the next walk may write
}

// Tensor memory and mbarrier of a CTA, around its walks.
__device__ __forceinline__ void walk_begin(unsigned char *sm)
{
    if (threadIdx.x < 32) tc::tmem_alloc(reinterpret_cast<uint32_t *>(sm + kSmTmem), kCols);
    if (threadIdx.x == 0) tc::mbar_init(reinterpret_cast<uint64_t *>(sm + kSmBar), 1);
    __syncthreads();
}
__device__ __forceinline__ void walk_end(unsigned char *sm, const Walk &walk, int *err)
{
    if (!walk.good && threadIdx.x == 0) {
        // an MMA did not report completion: one more bounded wait before the memory is released
        tc::mbar_wait_bounded(reinterpret_cast<uint64_t *>(sm + kSmBar), (walk.phase - 1) & 1u, kWaitLimit);
        atomicExch(err, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (threadIdx.x < 32) tc::tmem_dealloc(*reinterpret_cast<uint32_t *>(sm + kSmTmem), kCols);
}

__global__ void __launch_bounds__(kThreads, kCtasPerSm)
    k_mlp_grad(const float *__restrict__ w, const float4 *__restrict__ F, const float *__restrict__ T, int64_t n,
               float *grad, double *loss, int *err)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    Walk walk;
    walk_begin(sm);
    grad_tiles<true>(sm, walk, w, F, T, n, 0, n, 1, 0, load_sample(F, T, n, 0, n, 1, 0, blockIdx.x), grad, loss);
    walk_end(sm, walk, err);
}

// One epoch of training in one cooperative launch: per mini-batch the gradient, a barrier, Adam
// (Kingma & Ba) on the FP32 master weights by all CTAs, which also clears the gradient, and a
// barrier; the next batch's samples are loaded across the barriers.  As a gradient and an Adam launch a
// batch, 4,096 samples took 21 us, 12 of them in the gradient; 17 us here with two CTAs an SM,
// 15 with one that keeps gelu'(z1) in registers from the forward to the backward pass.
struct AdamArgs {
    float lr, b1, b2, eps;
};
// Zero before the first epoch; failed: a barrier's wait gave up, and the epochs that follow return
// at once instead of waiting in vain on the barrier that it left half full (the caller's error
// word may hold anything before the call).
struct EpochSync {
    GridBar bar;
    int32_t failed, pad;
};
constexpr int kAccDoubles = 12;   // of the moments, and of the loss
__global__ void __launch_bounds__(kThreads, 1)
    k_mlp_epoch(float *w, float *m, float *v, float *grad, const float4 *__restrict__ F, const float *__restrict__ T,
                int64_t n, int64_t batch, uint64_t pa, uint64_t pc, int64_t step, AdamArgs h, double *acc,
                float *history, EpochSync *sync, int *err)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    GridBar *gbar = &sync->bar;
    bool came = *reinterpret_cast<volatile int32_t *>(&sync->failed) == 0;   // (every block alike)
    Walk walk;
    uint32_t gen = *reinterpret_cast<volatile uint32_t *>(&gbar->gen);
    walk_begin(sm);
    Sample next = load_sample(F, T, n, 0, min(batch, n), pa, pc, blockIdx.x);
    for (int64_t b0 = 0; came && b0 < n; b0 += batch) {
        grad_tiles<false>(sm, walk, w, F, T, n, b0, min(batch, n - b0), pa, pc, next, grad, acc);
        const int64_t b1 = b0 + batch;
        if (b1 < n) next = load_sample(F, T, n, b1, min(batch, n - b1), pa, pc, blockIdx.x);
        if (!(came = grid_barrier(gbar, &sync->failed, gen))) break;
        ++step;
        const float c1 = 1.0f - powf(h.b1, (float)step), c2 = 1.0f - powf(h.b2, (float)step);
        for (int k = blockIdx.x * kThreads + threadIdx.x; k < kNW; k += gridDim.x * kThreads) {
            const float g = __ldcg(grad + k);
            grad[k] = 0.0f;
            const float mk = h.b1 * m[k] + (1.0f - h.b1) * g;
            const float vk = h.b2 * v[k] + (1.0f - h.b2) * g * g;
            m[k] = mk;
            v[k] = vk;
            w[k] -= h.lr * (mk / c1) / (sqrtf(vk / c2) + h.eps);
        }
        if (b1 >= n && blockIdx.x == 0 && threadIdx.x == 0) {   // the epoch's mean loss
            if (history) *history = (float)(__ldcg(acc) / (double)n);
            *acc = 0.0;
        }
        came = grid_barrier(gbar, &sync->failed, gen);
    }
    if (!came && threadIdx.x == 0) atomicExch(err, 5);
    walk_end(sm, walk, err);
}

// Mean and standard deviation of the raw features and labels (FP64 sums).
__global__ void k_mlp_moments(const float4 *__restrict__ F, const float *__restrict__ T, int64_t n, double *acc)
{
    double s[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 q = F[i];
        const double x[5] = {q.x, q.y, q.z, q.w, T[i]};
        for (int a = 0; a < 5; ++a) {
            s[a] += x[a];
            s[5 + a] += x[a] * x[a];
        }
    }
    // one atomic a block and sum (one a warp, 24,000 on ten words, took 32 us)
    __shared__ double sh[8][10];
#pragma unroll
    for (int a = 0; a < 10; ++a) {
        double r = s[a];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][a] = r;
    }
    __syncthreads();
    if (threadIdx.x < 10) {
        double r = 0.0;
        for (int k = 0; k < 8; ++k) r += sh[k][threadIdx.x];
        atomicAdd(&acc[threadIdx.x], r);
    }
}

__global__ void k_mlp_standardise(const float4 *__restrict__ F, const float *__restrict__ T, int64_t n,
                                  const double *acc, float *params, float4 *Fs, float *Ts)
{
    __shared__ float mu[5], sd[5];
    if (threadIdx.x < 5) {
        const double m = acc[threadIdx.x] / (double)n;
        double var = acc[5 + threadIdx.x] / (double)n - m * m;
        double s = var > 0.0 ? sqrt(var) : 0.0;
        if (!(s > 1e-12 * (fabs(m) + 1.0))) s = 1.0;   // a constant column is left unscaled
        mu[threadIdx.x] = (float)m;
        sd[threadIdx.x] = (float)s;
        if (blockIdx.x == 0) {
            if (threadIdx.x < 4) {
                params[kOffMuF + threadIdx.x] = (float)m;
                params[kOffSdF + threadIdx.x] = (float)s;
            } else {
                params[kOffMuY] = (float)m;
                params[kOffSdY] = (float)s;
            }
        }
    }
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 q = F[i];
        Fs[i] = make_float4((q.x - mu[0]) / sd[0], (q.y - mu[1]) / sd[1], (q.z - mu[2]) / sd[2], (q.w - mu[3]) / sd[3]);
        Ts[i] = (T[i] - mu[4]) / sd[4];
    }
}

uint64_t mix64(uint64_t x)
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}
uint64_t gcd64(uint64_t a, uint64_t b)
{
    while (b) {
        uint64_t r = a % b;
        a = b;
        b = r;
    }
    return a;
}

cudaError_t set_attr()
{
    const cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_mlp_epoch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
}

// CTAs over a batch: one per tile, at most two per SM (training, which keeps more in registers:
// one).
unsigned grad_grid(int64_t batch, int per_sm = kCtasPerSm)
{
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm <= 0)
        nsm = 1;
    return (unsigned)std::min<int64_t>((batch + 127) / 128, (int64_t)nsm * per_sm);
}

}  // namespace

}  // namespace sph

using namespace sph;

extern "C" sph_status sph_mlp_grad(const float *params, const float *features, const float *labels, int64_t n,
                                   float *grad, double *loss, int32_t *error, void *stream)
{
    if (n <= 0 || !params || !features || !labels || !grad || !loss || !error) return SPH_EINVAL;
    if ((n + 127) / 128 > 0x7fffffff) return SPH_EINVAL;
    if (set_attr() != cudaSuccess) return SPH_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemsetAsync(grad, 0, sizeof(float) * kNW, s) != cudaSuccess) return SPH_ECUDA;
    if (cudaMemsetAsync(loss, 0, sizeof(double), s) != cudaSuccess) return SPH_ECUDA;
    k_mlp_grad<<<grad_grid(n), kThreads, kSmem, s>>>(params, reinterpret_cast<const float4 *>(features), labels, n, grad,
                                                     loss, reinterpret_cast<int *>(error));
    return cudaGetLastError() == cudaSuccess ? SPH_OK : SPH_ECUDA;
}

extern "C" sph_status sph_mlp_train(const float *features, const float *labels, int64_t n, float *params,
                                    float *adam_state, int32_t epochs, int32_t batch, float lr, uint64_t seed,
                                    float *loss_history, int32_t *error, void *stream)
{
    if (n < 2 || !features || !labels || !params || !adam_state || !error || epochs < 0 || batch < 1 ||
        !(lr > 0.0f))
        return SPH_EINVAL;
    if (set_attr() != cudaSuccess) return SPH_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    float4 *Fs = nullptr;
    float *Ts = nullptr, *grad = nullptr;
    double *acc = nullptr;
    constexpr size_t kAccBytes = sizeof(double) * kAccDoubles + sizeof(EpochSync);
    auto cleanup = [&]() {
        if (Fs) cudaFreeAsync(Fs, s);
        if (Ts) cudaFreeAsync(Ts, s);
        if (grad) cudaFreeAsync(grad, s);
        if (acc) cudaFreeAsync(acc, s);
    };
    if (cudaMallocAsync(&Fs, sizeof(float4) * n, s) != cudaSuccess || cudaMallocAsync(&Ts, sizeof(float) * n, s) != cudaSuccess ||
        cudaMallocAsync(&grad, sizeof(float) * kNW, s) != cudaSuccess ||
        cudaMallocAsync(&acc, kAccBytes, s) != cudaSuccess) {
        cleanup();
        return SPH_ENOMEM;
    }
    bool ok = cudaMemsetAsync(acc, 0, kAccBytes, s) == cudaSuccess &&
              cudaMemsetAsync(grad, 0, sizeof(float) * kNW, s) == cudaSuccess;
    const float4 *F = reinterpret_cast<const float4 *>(features);
    k_mlp_moments<<<304, 256, 0, s>>>(F, labels, n, acc);
    k_mlp_standardise<<<304, 256, 0, s>>>(F, labels, n, acc, params, Fs, Ts);
    cudaMemsetAsync(acc, 0, kAccBytes, s);
    float *m = adam_state, *v = adam_state + kNW;
    EpochSync *sync = reinterpret_cast<EpochSync *>(acc + kAccDoubles);
    int64_t step = 0;
    const int64_t B = batch;
    for (int32_t e = 0; e < epochs && ok; ++e) {
        // a fresh bijection of the samples for this epoch
        uint64_t a = mix64(seed * 0x100000001B3ull + (uint64_t)e) % (uint64_t)(n - 1) + 1;
        while (gcd64(a, (uint64_t)n) != 1) a = a % (uint64_t)(n - 1) + 1;
        const uint64_t c = mix64(seed ^ (0xA5A5A5A5ull + (uint64_t)e)) % (uint64_t)n;
        float *hist = loss_history ? loss_history + e : nullptr;
        int *err = reinterpret_cast<int *>(error);
        AdamArgs h{lr, 0.9f, 0.999f, 1e-8f};
        const float4 *Fe = Fs;
        const float *Te = Ts;
        void *args[] = {&params, &m, &v, &grad, &Fe, &Te, (void *)&n, (void *)&B, (void *)&a, (void *)&c, &step, &h, &acc,
                        &hist, &sync, &err};
        ok = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(&k_mlp_epoch), dim3(grad_grid(std::min(B, n), 1)),
                                         dim3(kThreads), args, kSmem, s) == cudaSuccess;
        step += (n + B - 1) / B;
    }
    ok = ok && cudaGetLastError() == cudaSuccess;
    cleanup();
    return ok && cudaGetLastError() == cudaSuccess ? SPH_OK : SPH_ECUDA;
}
