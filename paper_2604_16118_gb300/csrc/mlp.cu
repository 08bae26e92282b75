// Small multilayer perceptron for the learned preconditioner controller:
// ReLU hidden layers, linear output, BF16 weights (rounded from FP32 master
// weights after every update), mean-squared-error loss and Adam updates of the
// masters.  Every product of the forward and backward passes runs on the
// 5th-generation tensor cores (tcgen05.mma kind::tf32, FP32 accumulation in
// tensor memory): the BF16 weights are exact in TF32, and the activations and
// back-propagated errors enter the products rounded to TF32 (nearest, ties
// away from zero).  Every result is stored once in the layouts in which the next
// products read it (operand images), so that the products move their operands
// with bulk copies only.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <functional>
#include <vector>

#include "ops.h"
#include "tc_common.cuh"

struct bsmps_mlp_s {
    bsm::Context* ctx;
    std::vector<int> widths;          // n_layers + 1
    std::vector<int64_t> w_off, b_off; // offsets into the flat parameter vector
    int64_t n_params = 0;
    float* master = nullptr;          // FP32 parameters (device)
    __nv_bfloat16* wbf = nullptr;     // BF16 copy of the parameters (device)
    float* img = nullptr;             // the BF16 weights as FP32 operand images (device), zero padded
    std::vector<int64_t> w1_off, w2_off;   // per layer: W (rows = outputs) and W^T (rows = inputs), in floats
    float* m1 = nullptr;              // Adam first moment
    float* m2 = nullptr;              // Adam second moment
    float* grad = nullptr;
    int64_t step = 0;
};

namespace bsm {
namespace {

constexpr int kT = 256;

// Operand image of a matrix of n rows x K values (FP32, already rounded to TF32):
// blocks of 128 rows x 32 values (16 KB, K-major with 128-byte swizzle), the blocks
// of a row range contiguous along K, so that a chunk of a tile is one bulk copy.  The
// blocks of the last row range end with row n - 1: a layer of 2 outputs and a batch of
// 10^6 takes 8 MB and not 512.  Values of k >= K are zero (the products run over whole
// chunks); the rows that a block lacks are whatever stands in shared memory behind its
// copy (they reach only entries that are not stored).
constexpr int kImgRows = 128, kImgK = 32;
constexpr int64_t kImgBlock = kImgRows * kImgK;   // floats
__host__ __device__ __forceinline__ int img_chunks(int K) { return (K + kImgK - 1) / kImgK; }
inline int64_t img_size(int n, int K) { return (int64_t)n * img_chunks(K) * kImgK; }
// Rows of the block that holds row r of n.
__host__ __device__ __forceinline__ int img_rows(int r, int n) {
    const int left = n - r / kImgRows * kImgRows;
    return left < kImgRows ? left : kImgRows;
}
// Row r < n, value k, over nkc chunks.
__host__ __device__ __forceinline__ int64_t img_at(int r, int k, int n, int nkc) {
    return (int64_t)(r / kImgRows) * nkc * kImgBlock + (int64_t)(k / kImgK) * img_rows(r, n) * kImgK +
           (r % kImgRows) * kImgK + ((((k >> 2) & 7) ^ (r & 7)) << 2) + (k & 3);
}
__device__ __forceinline__ float tf32_round(float f) { return __uint_as_float(tc::tf32_bits(f)); }

// One product of the network on the tensor cores, C(m, n) = epi( sum_k a(m, k) b(n, k) ),
// both factors given as operand images over nkc chunks of 32 values of k.  Outputs:
//  - part: raw sums of a k range to part[z] (row-major), summed by k_mlp_reduce or k_mlp_finish;
//  - y: row-major FP32 (the network's output);
//  - i1, i2: the operand images of the result (rows = m; rows = n), rounded to TF32
//    as the next products read them.
// epi adds bias[n] (BF16) and applies ReLU, or keeps the entry only where the image
// mask (rows = m) is positive (the derivative of the ReLU that produced it).
struct MlpGemm {
    const float* A;
    const float* B;
    int M, N, K, nkc;   // nkc: chunks of K
    int n_acc, acc_len; // accumulators of a CTA (at most), chunks per accumulator
    const __nv_bfloat16* bias;
    int relu;
    const float* mask;
    float* y;
    float *i1, *i2;
    float* part;
};

constexpr int kMlpM = 128;         // rows of a tile (the M of one tcgen05.mma)
constexpr int kMlpN = 128;         // columns of a tile (its N, and the tensor-memory columns of an accumulator)
constexpr int kMlpAcc = 4;         // accumulators at most (512 tensor-memory columns)
constexpr int kMlpStages = 4;
constexpr uint32_t kMlpOperand = kImgBlock * 4;       // bytes of one operand block
constexpr uint32_t kMlpStage = 2 * kMlpOperand;
constexpr int kMlpThreads = 128;   // warp w reads tensor-memory lanes 32 w .. 32 w + 31
constexpr uint32_t kMlpIdesc = tc::idesc_tf32(kMlpM, kMlpN);

// One CTA per 128 x 128 output tile and range of chunks (blockIdx.z): one thread
// streams the blocks through four stages by bulk copies, another issues four MMAs
// per chunk; no thread touches an operand (staging them through registers, strided
// and rounded on the way, took 0.86 ms for the products of a batch of 8192).  All
// four warps run the epilogue, which adds a tile's accumulators in order.  What is left is latency: at 8 chunks a tile's copies
// and its epilogue (two images) are longer than its 32 MMAs.  Waits are bounded; a CTA that
// gives up sets *err and frees its tensor memory after its MMAs and copies.
__global__ void __launch_bounds__(kMlpThreads) k_mlp_gemm_tc(const MlpGemm g, int chunks, int* err) {
    extern __shared__ __align__(1024) unsigned char mlp_smem[];
    __shared__ __align__(8) uint64_t bars[2 * kMlpStages + 1];
    __shared__ uint32_t tmem_slot;
    const uint32_t base = (tc::smem_addr(mlp_smem) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * kMlpM, n0 = blockIdx.y * kMlpN;
    const int c0 = blockIdx.z * chunks, nc = min(chunks, g.nkc - c0);   // >= 1
    const int rows_a = img_rows(m0, g.M), rows_b = img_rows(n0, g.N);
    auto full = [&](int s) { return tc::smem_addr(&bars[s]); };
    auto empty = [&](int s) { return tc::smem_addr(&bars[kMlpStages + s]); };
    const uint32_t done = tc::smem_addr(&bars[2 * kMlpStages]);
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * kMlpStages + 1; ++i) tc::mbar_init(tc::smem_addr(&bars[i]), 1);
        tc::mbar_init_fence();
    }
    const int cols = kMlpN * (g.n_acc > 2 ? 4 : g.n_acc);   // a power of two
    if (warp == 1) tc::tmem_alloc(&tmem_slot, cols);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_slot;
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            const int64_t step_a = rows_a * kImgK, step_b = rows_b * kImgK;   // floats of a chunk
            const float* a = g.A + (int64_t)blockIdx.x * g.nkc * kImgBlock + c0 * step_a;
            const float* b = g.B + (int64_t)blockIdx.y * g.nkc * kImgBlock + c0 * step_b;
            int c = 0;
            for (; c < nc; ++c) {
                const int s = c % kMlpStages;
                if (c >= kMlpStages && !tc::mbar_wait(empty(s), (c / kMlpStages - 1) & 1)) {
                    ok = false;
                    break;
                }
                const uint32_t dst = base + s * kMlpStage;
                tc::mbar_expect(full(s), (uint32_t)(step_a + step_b) * 4);
                tc::bulk_load(dst, a + c * step_a, (uint32_t)step_a * 4, full(s));
                tc::bulk_load(dst + kMlpOperand, b + c * step_b, (uint32_t)step_b * 4, full(s));
            }
            // copies in flight land before the CTA may end
            for (int i = c > kMlpStages ? c - kMlpStages : 0; i < c; ++i)
                tc::mbar_wait(full(i % kMlpStages), (i / kMlpStages) & 1);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            for (int c = 0; c < nc; ++c) {
                const int s = c % kMlpStages;
                if (!tc::mbar_wait(full(s), (c / kMlpStages) & 1)) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                const uint64_t a = tc::desc_sw128(base + s * kMlpStage), b = a + (kMlpOperand >> 4);
#pragma unroll
                for (int kk = 0; kk < kImgK / 8; ++kk)   // 32 bytes along k per MMA
                    tc::mma_tf32(tmem + (uint32_t)(c / g.acc_len * kMlpN), a + 2 * kk, b + 2 * kk, kMlpIdesc,
                                 c % g.acc_len == 0 && kk == 0 ? 0u : 1u);
                tc::commit(empty(s));
            }
            tc::commit(done);   // covers every MMA and every earlier commit
            ok = tc::mbar_wait(done, 0) && ok;
        }
        __syncwarp();
    }
    ok = __all_sync(0xffffffffu, tc::mbar_wait(done, 0) && ok);
    tc::fence_after();
    const int row = m0 + warp * 32 + lane;
    const int n_acc = (nc + g.acc_len - 1) / g.acc_len;   // (the last range of k may be shorter)
    const int nk1 = img_chunks(g.N), nk2 = img_chunks(g.M);   // chunks of the result's images
    for (int cc = 0; ok && cc < kMlpN; cc += 16) {
        uint32_t v[16];
        tc::ld_32x32b_x16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)cc, v);
        for (int a = 1; a < n_acc; ++a) {
            uint32_t u[16];
            tc::ld_32x32b_x16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(a * kMlpN + cc), u);
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(u[j]));
        }
        const int col = n0 + cc;
        if (g.part) {
            if (row < g.M) {
                float* o = g.part + ((int64_t)blockIdx.z * g.M + row) * g.N + col;
                if ((g.N & 3) == 0 && ((uintptr_t)g.part & 15) == 0) {
#pragma unroll
                    for (int j = 0; j < 16; j += 4)
                        if (col + j < g.N) *(uint4*)(o + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (col + j < g.N) o[j] = __uint_as_float(v[j]);
                }
            }
            continue;
        }
        float w[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            float acc = __uint_as_float(v[j]);
            if (g.bias && col + j < g.N) acc += __bfloat162float(g.bias[col + j]);
            if (g.relu) acc = fmaxf(acc, 0.0f);
            w[j] = acc;
        }
        if (g.mask && row < g.M && col < nk1 * kImgK) {
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
                const float4 h = *(const float4*)(g.mask + img_at(row, col + j, g.M, nk1));
                if (!(h.x > 0.0f)) w[j] = 0.0f;
                if (!(h.y > 0.0f)) w[j + 1] = 0.0f;
                if (!(h.z > 0.0f)) w[j + 2] = 0.0f;
                if (!(h.w > 0.0f)) w[j + 3] = 0.0f;
            }
        }
        if (g.y) {
            if (row < g.M)
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (col + j < g.N) g.y[(int64_t)row * g.N + col + j] = w[j];
            continue;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) w[j] = row < g.M && col + j < g.N ? tf32_round(w[j]) : 0.0f;
        if (row < g.M && col < nk1 * kImgK)
#pragma unroll
            for (int j = 0; j < 16; j += 4)
                *(float4*)(g.i1 + img_at(row, col + j, g.M, nk1)) = make_float4(w[j], w[j + 1], w[j + 2], w[j + 3]);
        if (g.i2 && row < nk2 * kImgK)
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (col + j < g.N) g.i2[img_at(col + j, row, g.N, nk2)] = w[j];
    }
    if (!ok) atomicExch(err, 1);
    tc::fence_before();
    __syncthreads();
    if (warp == 1) tc::tmem_free(tmem, cols);
}

// C = sum_z part[z], the k ranges summed in order.
__global__ void k_mlp_reduce(const float* __restrict__ part, float* __restrict__ C, int64_t n, int n_parts) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    float acc = 0.0f;
#pragma unroll 8
    for (int z = 0; z < n_parts; ++z) acc += part[(int64_t)z * n + e];
    C[e] = acc;
}

// The result of a product whose k ranges were summed by different CTAs: the ranges in order, then
// what the epilogue of k_mlp_gemm_tc does (bias, ReLU or mask; y, or the images i1 and i2).
// 32 x 32 tiles through shared memory, so that both images are written along their rows.
__global__ void __launch_bounds__(256) k_mlp_finish(const MlpGemm g, int n_parts) {
    __shared__ float t[32][33];
    const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32, x = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int nk1 = img_chunks(g.N), nk2 = img_chunks(g.M);
    for (int i = y; i < 32; i += 8) {
        const int r = r0 + i, c = c0 + x;
        const bool in = r < g.M && c < g.N;
        float v = 0.0f;
        if (in) {
#pragma unroll 8
            for (int z = 0; z < n_parts; ++z) v += g.part[((int64_t)z * g.M + r) * g.N + c];
            if (g.bias) v += __bfloat162float(g.bias[c]);
            if (g.relu) v = fmaxf(v, 0.0f);
            if (g.mask && !(g.mask[img_at(r, c, g.M, nk1)] > 0.0f)) v = 0.0f;
        }
        if (g.y) {
            if (in) g.y[(int64_t)r * g.N + c] = v;
            continue;
        }
        v = tf32_round(v);
        t[i][x] = v;
        if (r < g.M) g.i1[img_at(r, c, g.M, nk1)] = v;
    }
    if (g.y || !g.i2) return;
    __syncthreads();
    for (int i = y; i < 32; i += 8)
        if (c0 + i < g.N) g.i2[img_at(c0 + i, r0 + x, g.N, nk2)] = t[x][i];
}

// The operand images of a row-major matrix X (n x K): rows of X, and (i2 not
// null) rows of X^T over n.  32 x 32 tiles through shared memory.
__global__ void __launch_bounds__(256) k_mlp_pack(const float* __restrict__ X, int n, int K, float* __restrict__ i1,
                                                  float* __restrict__ i2) {
    __shared__ float t[32][33];
    const int r0 = blockIdx.x * 32, k0 = blockIdx.y * 32, x = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int nk1 = img_chunks(K), nk2 = img_chunks(n);
    for (int i = y; i < 32; i += 8) {
        const int r = r0 + i, k = k0 + x;
        const float v = r < n && k < K ? tf32_round(X[(int64_t)r * K + k]) : 0.0f;
        t[i][x] = v;
        if (r < n) i1[img_at(r, k, n, nk1)] = v;
    }
    if (!i2) return;
    __syncthreads();
    for (int i = y; i < 32; i += 8)
        if (k0 + i < K) i2[img_at(k0 + i, r0 + x, K, nk2)] = t[x][i];
}

// dY of the loss 1/(B out) sum (Y - T)^2 as operand images (rows = batch, rows =
// outputs; rounded to TF32), and the per-element squared error.
__global__ void k_mse(const float* __restrict__ Y, const float* __restrict__ T, float* __restrict__ d1,
                      float* __restrict__ d2, float* __restrict__ sq, int B, int out, float scale) {
    const int nk1 = img_chunks(out), nk2 = img_chunks(B);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int b = (int)(e / (nk1 * kImgK)), o = (int)(e % (nk1 * kImgK));
    if (b >= nk2 * kImgK) return;
    float v = 0.0f;
    if (b < B && o < out) {
        const float d = Y[(int64_t)b * out + o] - T[(int64_t)b * out + o];
        v = tf32_round(2.0f * scale * d);
        sq[(int64_t)b * out + o] = d * d;
    }
    if (b < B) d1[img_at(b, o, B, nk1)] = v;
    if (o < out) d2[img_at(o, b, out, nk2)] = v;
}

// db[o] = sum_b dY[b, o] (rounded as the weight-gradient product reads it), eight o
// per CTA: their rows are a contiguous 1 KB of every block of the image (rows = o, k
// = b, zeros beyond B; fewer in the last CTA), a warp's eight lanes per row, the blocks
// dealt to the warps.
constexpr int kBiasThreads = 512;
__global__ void __launch_bounds__(kBiasThreads) k_mlp_bgrad(const float* __restrict__ d2, float* __restrict__ db, int B,
                                                            int out) {
    __shared__ float red[kBiasThreads / 32][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, o0 = 8 * blockIdx.x, nk2 = img_chunks(B);
    const int64_t step = (int64_t)(kBiasThreads / 32) * img_rows(o0, out) * (kImgK / 4);   // float4
    const float4* p = (const float4*)(d2 + img_at(o0, 0, out, nk2)) + (int64_t)warp * img_rows(o0, out) * (kImgK / 4);
    // rows lane / 8 and 4 + lane / 8; lanes of rows that the image lacks read its last one
    const float4* p0 = p + min(lane >> 3, out - 1 - o0) * 8 + (lane & 7);
    const float4* p1 = p + min(4 + (lane >> 3), out - 1 - o0) * 8 + (lane & 7);
    float s0 = 0.0f, s1 = 0.0f;
#pragma unroll 4
    for (int c = warp; c < nk2; c += kBiasThreads / 32, p0 += step, p1 += step) {
        const float4 x = *p0, y = *p1;
        s0 += (x.x + x.y) + (x.z + x.w);
        s1 += (y.x + y.y) + (y.z + y.w);
    }
    for (int d = 4; d > 0; d >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, d);
        s1 += __shfl_xor_sync(0xffffffffu, s1, d);
    }
    if ((lane & 7) == 0) {
        red[warp][lane >> 3] = s0;
        red[warp][4 + (lane >> 3)] = s1;
    }
    __syncthreads();
    if (threadIdx.x < 8 && o0 + (int)threadIdx.x < out) {
        float acc = 0.0f;
        for (int w = 0; w < kBiasThreads / 32; ++w) acc += red[w][threadIdx.x];
        db[o0 + threadIdx.x] = acc;
    }
}

// Where parameter e lies: the weight images of its layer.
constexpr int kMaxLayers = 16;
struct MlpLayers {
    int n;
    int64_t w_off[kMaxLayers], w1[kMaxLayers], w2[kMaxLayers];
    int in[kMaxLayers], out[kMaxLayers];
};
__device__ __forceinline__ void store_bf16(const MlpLayers& L, float* img, __nv_bfloat16* pb, int64_t e, float q) {
    const __nv_bfloat16 h = __float2bfloat16_rn(q);
    pb[e] = h;
    for (int l = 0; l < L.n; ++l) {
        const int64_t d = e - L.w_off[l];
        if (d < 0 || d >= (int64_t)L.in[l] * L.out[l]) continue;
        const int o = (int)(d / L.in[l]), i = (int)(d % L.in[l]);
        const float w = __bfloat162float(h);
        img[L.w1[l] + img_at(o, i, L.out[l], img_chunks(L.in[l]))] = w;
        img[L.w2[l] + img_at(i, o, L.in[l], img_chunks(L.out[l]))] = w;
    }
}

// Adam (beta1 = 0.9, beta2 = 0.999, eps = 1e-8) on the FP32 masters, then the BF16 copy and its images.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, __nv_bfloat16* __restrict__ pb, float* __restrict__ img,
                       const MlpLayers L, int64_t n, float lr, float c1, float c2) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const float gg = g[e];
    const float a = 0.9f * m1[e] + 0.1f * gg;
    const float v = 0.999f * m2[e] + 0.001f * gg * gg;
    m1[e] = a;
    m2[e] = v;
    const float q = p[e] - lr * (a / c1) / (sqrtf(v / c2) + 1e-8f);
    p[e] = q;
    store_bf16(L, img, pb, e, q);
}

__global__ void k_to_bf16(const float* __restrict__ p, __nv_bfloat16* __restrict__ pb, float* __restrict__ img,
                          const MlpLayers L, int64_t n) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) store_bf16(L, img, pb, e, p[e]);
}

unsigned grid(int64_t n) { return (unsigned)((n + kT - 1) / kT); }

void done(Context* ctx) {
    ctx->launches++;
    BSM_CUDA(cudaGetLastError());
}

MlpLayers layers_of(const bsmps_mlp_s* net) {
    MlpLayers L{};
    L.n = (int)net->widths.size() - 1;
    for (int l = 0; l < L.n; ++l) {
        L.w_off[l] = net->w_off[l];
        L.w1[l] = net->w1_off[l];
        L.w2[l] = net->w2_off[l];
        L.in[l] = net->widths[l];
        L.out[l] = net->widths[l + 1];
    }
    return L;
}

float* floats(Scratch& s, int64_t n) { return (float*)s.dbl((size_t)(n + 1) / 2); }

// A product's sum over k is taken in ranges, each from zero in an FP32 accumulator of its own
// (the tensor cores truncate every addition to an accumulator: a sum of positive terms over
// 4096 values of k loses 68 units of 2^-24 in 4 ranges and 3.6 in 32).  As many ranges as bring
// the 128 x 64 tiles to kMlpRangeTiles, four chunks at least in each.  The rule is part of the
// result: activations and errors enter the next product rounded to TF32, so the order of their
// sums shows in the gradient (3e-5 of it).
constexpr int kMlpRangeTiles = 296;

// One product.  Up to four ranges are the accumulators of one CTA; more go to a CTA each
// (there are few tiles then; 4096 x 4096 at a batch of 16: 57 -> 30 us), summed in order by
// k_mlp_finish.  grad != null: one wave of CTAs over tiles and k, each with accumulators no
// longer than a range, the CTAs' sums added in order into grad.
void launch_mlp_gemm(Context* ctx, MlpGemm g, Scratch& s, float* grad = nullptr) {
    const int smem = kMlpStages * (int)kMlpStage + 1024;
    static bool attr = false;
    if (!attr) {
        BSM_CUDA(cudaFuncSetAttribute(k_mlp_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        attr = true;
    }
    const int tm = (g.M + kMlpM - 1) / kMlpM, tn = (g.N + kMlpN - 1) / kMlpN;
    const int64_t tiles = (int64_t)tm * ((g.N + 63) / 64);
    int ranges = 1;
    while (tiles * ranges < kMlpRangeTiles && g.nkc / (2 * ranges) >= 4) ranges *= 2;
    const int len = (g.nkc + ranges - 1) / ranges;
    int chunks = g.nkc;   // of one CTA
    g.acc_len = len;
    g.n_acc = (g.nkc + len - 1) / len;
    if (grad) {
        // one CTA per SM (128 KB of stages), at least four chunks each
        int nsm = 0;
        BSM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
        const int splits = std::max(1, std::min(nsm / std::max(1, tm * tn), g.nkc / 4));
        chunks = (g.nkc + splits - 1) / splits;
        g.n_acc = std::min(kMlpAcc, (chunks + len - 1) / len);   // (at most four by the rule of the ranges)
        g.acc_len = (chunks + g.n_acc - 1) / g.n_acc;
    } else if (g.n_acc > kMlpAcc) {
        chunks = len;
        g.n_acc = 1;
    }
    const int parts = (g.nkc + chunks - 1) / chunks;
    if (parts > 1) g.part = floats(s, (int64_t)parts * g.M * g.N);
    else if (grad) g.part = grad;
    const double fl = 2.0 * g.M * (double)g.N * g.K;
    const double by = 4.0 * ((double)(g.M + g.N) * g.K + (double)g.M * g.N);
    ProfScope ps(ctx, KK_MLP, fl, by);
    k_mlp_gemm_tc<<<dim3((unsigned)tm, (unsigned)tn, (unsigned)parts), kMlpThreads, smem, ctx->stream>>>(
        g, chunks, ctx->err_word());
    done(ctx);
    if (parts > 1 && !grad) {
        k_mlp_finish<<<dim3((unsigned)img_chunks(g.M), (unsigned)img_chunks(g.N)), 256, 0, ctx->stream>>>(g, parts);
        done(ctx);
    } else if (parts > 1) {
        const int64_t n = (int64_t)g.M * g.N;
        k_mlp_reduce<<<grid(n), kT, 0, ctx->stream>>>(g.part, grad, n, parts);
        done(ctx);
    }
    ps.done();
}

// A host array on the device by one copy from the caller's memory (staging a 4 MB
// batch through the pinned ring took 0.25 ms, the copy takes 0.04 ms).
float* upload_batch(Context* ctx, const float* host, int64_t n, Scratch& s) {
    float* d = floats(s, n);
    BSM_CUDA(cudaMemcpyAsync(d, host, sizeof(float) * (size_t)n, cudaMemcpyHostToDevice, ctx->stream));
    return d;
}

// Forward pass of a batch: y (B x out, row-major, device); with `keep`, the images
// of every layer's input (rows = batch, rows = features) for the backward pass.
struct Acts {
    std::vector<float*> h1, h2;
    float* y = nullptr;
};
Acts forward(Context* ctx, bsmps_mlp_s* net, const float* x_host, int B, Scratch& s, bool keep) {
    const int nl = (int)net->widths.size() - 1;
    Acts a;
    const int in0 = net->widths[0];
    const float* x = upload_batch(ctx, x_host, (int64_t)B * in0, s);
    a.h1.push_back(floats(s, img_size(B, in0)));
    a.h2.push_back(keep ? floats(s, img_size(in0, B)) : nullptr);
    k_mlp_pack<<<dim3((unsigned)img_chunks(B), (unsigned)img_chunks(in0)), 256, 0, ctx->stream>>>(x, B, in0, a.h1[0],
                                                                                                  a.h2[0]);
    done(ctx);
    for (int l = 0; l < nl; ++l) {
        const int in = net->widths[l], out = net->widths[l + 1];
        // Y[b, o] = sum_i X[b, i] W[o, i] + bias[o]
        MlpGemm g{};
        g.A = a.h1[l];
        g.B = net->img + net->w1_off[l];
        g.M = B;
        g.N = out;
        g.K = in;
        g.nkc = img_chunks(in);
        g.bias = net->wbf + net->b_off[l];
        if (l + 1 < nl) {
            g.relu = 1;
            a.h1.push_back(floats(s, img_size(B, out)));
            a.h2.push_back(keep ? floats(s, img_size(out, B)) : nullptr);
            g.i1 = a.h1.back();
            g.i2 = a.h2.back();
        } else {
            g.y = a.y = floats(s, (int64_t)B * out);
        }
        launch_mlp_gemm(ctx, g, s);
    }
    return a;
}

// loss and gradient into net->grad (device)
float loss_grad(Context* ctx, bsmps_mlp_s* net, const float* x_host, const float* t_host, int B) {
    const int nl = (int)net->widths.size() - 1;
    const int outL = net->widths[nl];
    Scratch s(ctx);
    const float* td = upload_batch(ctx, t_host, (int64_t)B * outL, s);
    Acts a = forward(ctx, net, x_host, B, s, true);
    const int n = B * outL;
    float* d1 = floats(s, img_size(B, outL));
    float* d2 = floats(s, img_size(outL, B));
    float* sq = floats(s, n);
    k_mse<<<grid((int64_t)img_chunks(B) * kImgK * img_chunks(outL) * kImgK), kT, 0, ctx->stream>>>(
        a.y, td, d1, d2, sq, B, outL, 1.0f / (float)n);
    done(ctx);
    for (int l = nl - 1; l >= 0; --l) {
        const int in = net->widths[l], out = net->widths[l + 1];
        // dW[o, i] = sum_b dY[b, o] X[b, i]
        MlpGemm gw{};
        gw.A = d2;
        gw.B = a.h2[l];
        gw.M = out;
        gw.N = in;
        gw.K = B;
        gw.nkc = img_chunks(B);
        launch_mlp_gemm(ctx, gw, s, net->grad + net->w_off[l]);
        k_mlp_bgrad<<<(unsigned)((out + 7) / 8), kBiasThreads, 0, ctx->stream>>>(d2, net->grad + net->b_off[l], B, out);
        done(ctx);
        if (l > 0) {
            // dX[b, i] = (sum_o dY[b, o] W[o, i]) [X[b, i] > 0]
            MlpGemm gx{};
            gx.A = d1;
            gx.B = net->img + net->w2_off[l];
            gx.M = B;
            gx.N = in;
            gx.K = out;
            gx.nkc = img_chunks(out);
            gx.mask = a.h1[l];
            gx.i1 = floats(s, img_size(B, in));
            gx.i2 = floats(s, img_size(in, B));
            launch_mlp_gemm(ctx, gx, s);
            d1 = gx.i1;
            d2 = gx.i2;
        }
    }
    std::vector<float> sh((size_t)n);
    BSM_CUDA(cudaMemcpyAsync(sh.data(), sq, sizeof(float) * n, cudaMemcpyDeviceToHost, ctx->stream));
    ctx->sync();
    double acc = 0.0;
    for (float v : sh) acc += v;
    return (float)(acc / n);
}

}  // namespace
}  // namespace bsm

namespace {
bsmps_status mlp_guard(bsm::Context* ctx, const std::function<void()>& f) {
    try {
        f();
        return BSMPS_OK;
    } catch (const bsm::Error& e) {
        if (ctx) ctx->last_error = e.what();
        return e.code;
    } catch (const std::exception& e) {
        if (ctx) ctx->last_error = e.what();
        return BSMPS_ERR_INVALID_ARG;
    }
}

bsm::Context* ctx_of(bsmps_mlp m) {
    if (!m || !m->ctx) throw bsm::Error(BSMPS_ERR_INVALID_ARG, "null MLP handle");
    BSM_CUDA(cudaSetDevice(m->ctx->device));
    (void)cudaGetLastError();   // a stale error left by another caller is not this call's
    return m->ctx;
}
}  // namespace

namespace bsm {
Context* context_of(bsmps_ctx ctx);
}

extern "C" {

bsmps_status bsmps_mlp_create(bsmps_ctx c, int n_layers, const int* widths, const float* params, int64_t n_params,
                              bsmps_mlp* out) {
    bsm::Context* ctx = nullptr;
    bsmps_status st = mlp_guard(nullptr, [&] { ctx = bsm::context_of(c); });
    if (st != BSMPS_OK) return st;
    bsmps_mlp_s* net = nullptr;
    st = mlp_guard(ctx, [&] {
        BSM_REQUIRE(n_layers >= 1 && n_layers <= 16 && widths && params && out, BSMPS_ERR_INVALID_ARG,
                    "mlp_create: 1..16 layers, widths, params and out required");
        net = new bsmps_mlp_s;
        net->ctx = ctx;
        int64_t off = 0;
        for (int l = 0; l <= n_layers; ++l) {
            BSM_REQUIRE(widths[l] > 0 && widths[l] <= 4096, BSMPS_ERR_INVALID_ARG, "mlp_create: width out of range");
            net->widths.push_back(widths[l]);
        }
        for (int l = 0; l < n_layers; ++l) {
            net->w_off.push_back(off);
            off += (int64_t)widths[l] * widths[l + 1];
            net->b_off.push_back(off);
            off += widths[l + 1];
        }
        net->n_params = off;
        BSM_REQUIRE(n_params == off, BSMPS_ERR_INVALID_ARG, "mlp_create: params must hold every weight and bias");
        BSM_CUDA(cudaMalloc(&net->master, sizeof(float) * off));
        BSM_CUDA(cudaMalloc(&net->wbf, sizeof(__nv_bfloat16) * off));
        int64_t images = 0;
        for (int l = 0; l < n_layers; ++l) {
            net->w1_off.push_back(images);
            images += bsm::img_size(widths[l + 1], widths[l]);
            net->w2_off.push_back(images);
            images += bsm::img_size(widths[l], widths[l + 1]);
        }
        BSM_CUDA(cudaMalloc(&net->img, sizeof(float) * images));
        BSM_CUDA(cudaMemsetAsync(net->img, 0, sizeof(float) * images, ctx->stream));
        BSM_CUDA(cudaMalloc(&net->m1, sizeof(float) * off));
        BSM_CUDA(cudaMalloc(&net->m2, sizeof(float) * off));
        BSM_CUDA(cudaMalloc(&net->grad, sizeof(float) * off));
        BSM_CUDA(cudaMemcpy(net->master, params, sizeof(float) * off, cudaMemcpyHostToDevice));
        BSM_CUDA(cudaMemset(net->m1, 0, sizeof(float) * off));
        BSM_CUDA(cudaMemset(net->m2, 0, sizeof(float) * off));
        bsm::k_to_bf16<<<bsm::grid(off), bsm::kT, 0, ctx->stream>>>(net->master, net->wbf, net->img,
                                                                        bsm::layers_of(net), off);
        bsm::done(ctx);
        ctx->sync();
        *out = net;
        net = nullptr;
    });
    if (net) {
        cudaFree(net->master);
        cudaFree(net->wbf);
        cudaFree(net->img);
        cudaFree(net->m1);
        cudaFree(net->m2);
        cudaFree(net->grad);
        delete net;
    }
    return st;
}

bsmps_status bsmps_mlp_num_params(bsmps_mlp m, int64_t* n) {
    if (!m || !n) return BSMPS_ERR_INVALID_ARG;
    *n = m->n_params;
    return BSMPS_OK;
}

bsmps_status bsmps_mlp_get_params(bsmps_mlp m, float* params) {
    return mlp_guard(m ? m->ctx : nullptr, [&] {
        bsm::Context* ctx = ctx_of(m);
        BSM_REQUIRE(params, BSMPS_ERR_INVALID_ARG, "null out");
        BSM_CUDA(cudaMemcpyAsync(params, m->master, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost, ctx->stream));
        ctx->sync();
    });
}

bsmps_status bsmps_mlp_forward(bsmps_mlp m, const float* x, int B, float* y) {
    return mlp_guard(m ? m->ctx : nullptr, [&] {
        bsm::Context* ctx = ctx_of(m);
        BSM_REQUIRE(x && y && B > 0, BSMPS_ERR_INVALID_ARG, "mlp_forward: x, y and B > 0 required");
        bsm::Scratch s(ctx);
        bsm::Acts a = bsm::forward(ctx, m, x, B, s, false);
        const int out = m->widths.back();
        BSM_CUDA(cudaMemcpyAsync(y, a.y, sizeof(float) * B * out, cudaMemcpyDeviceToHost, ctx->stream));
        ctx->sync();
    });
}

bsmps_status bsmps_mlp_loss_grad(bsmps_mlp m, const float* x, const float* t, int B, float* loss, float* grad) {
    return mlp_guard(m ? m->ctx : nullptr, [&] {
        bsm::Context* ctx = ctx_of(m);
        BSM_REQUIRE(x && t && B > 0, BSMPS_ERR_INVALID_ARG, "mlp_loss_grad: x, t and B > 0 required");
        const float l = bsm::loss_grad(ctx, m, x, t, B);
        if (loss) *loss = l;
        if (grad) {
            BSM_CUDA(cudaMemcpyAsync(grad, m->grad, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost, ctx->stream));
            ctx->sync();
        }
    });
}

bsmps_status bsmps_mlp_train_step(bsmps_mlp m, const float* x, const float* t, int B, float lr, float* loss) {
    return mlp_guard(m ? m->ctx : nullptr, [&] {
        bsm::Context* ctx = ctx_of(m);
        BSM_REQUIRE(x && t && B > 0 && lr > 0.0f, BSMPS_ERR_INVALID_ARG, "mlp_train_step: bad argument");
        const float l = bsm::loss_grad(ctx, m, x, t, B);
        m->step += 1;
        const float c1 = 1.0f - std::pow(0.9f, (float)m->step);
        const float c2 = 1.0f - std::pow(0.999f, (float)m->step);
        bsm::k_adam<<<bsm::grid(m->n_params), bsm::kT, 0, ctx->stream>>>(m->master, m->grad, m->m1, m->m2, m->wbf,
                                                                          m->img, bsm::layers_of(m), m->n_params, lr,
                                                                          c1, c2);
        bsm::done(ctx);
        if (loss) *loss = l;
    });
}

bsmps_status bsmps_mlp_destroy(bsmps_mlp m) {
    if (!m) return BSMPS_ERR_INVALID_ARG;
    cudaSetDevice(m->ctx->device);
    cudaFree(m->master);
    cudaFree(m->wbf);
    cudaFree(m->img);
    cudaFree(m->m1);
    cudaFree(m->m2);
    cudaFree(m->grad);
    delete m;
    return BSMPS_OK;
}

}  // extern "C"
