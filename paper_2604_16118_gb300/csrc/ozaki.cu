// FP64 matrix product emulated on bf16 tensor cores by exact integer slice
// products (the Ozaki scheme: Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 59
// (2012); integer slices as in Uchino, Ozaki, Imamura 2024).  Not part of the
// paper: an FP64 path for the large contractions of the solver.
//
// Row i of A is scaled by 2^-(e_i + 1) (e_i the smallest integer with
// max_j |a_ij| < 2^e_i), column j of B by 2^-(f_j + 1); the scaled values, below
// 1/2 in magnitude, are cut into S balanced digits of b bits (integers in
// [-2^(b-1), 2^(b-1)], exact in bf16; what lies below the last digit is rounded, so
// that the remainder is at most 2^(e_i - b S)).  C = sum over slice pairs (p, q) with
// p + q = d <= S + 1 of 2^{e_i + f_j + 2 - b d} A_p B_q.  The slice products of one d
// over 128 values of k are integers below 2^24, so the FP32 accumulator of the
// tensor-core product (tcgen05.mma kind::f16, BF16 operands, accumulators in
// tensor memory) is exact, the diagonals are combined exactly in 64-bit integers,
// and the result is rounded once.  b = 7, except that the full 56 bits (8 slices asked
// for) are cut into 7 digits of 8 bits: the same remainders and the same size of
// the first dropped pairs, with 28 products instead of 36.
#include <algorithm>

#include "kernels.h"
#include "row_scan.cuh"
#include "tc_common.cuh"

namespace bsm {
namespace {

void launched(Context* ctx) {
    ctx->launches++;
    BSM_CUDA(cudaGetLastError());
}

constexpr int kOzKStep = 32;       // k values of one staged chunk; Kp is a multiple of it (zeros from K on)
constexpr int kOzMaxS = 8;
constexpr int kOzM = 128;          // tile rows: the M of one tcgen05.mma (cta_group::1)
constexpr int kOzN = 64;           // tile columns: its N, and the tensor-memory columns of one diagonal
constexpr int kOzSbo = 8 * kOzKStep * 2;              // bytes between 8-row groups of a slice tile
constexpr int kOzSliceA = kOzM * kOzKStep * 2;        // bytes of one A slice tile (128 x 32 bf16)
constexpr int kOzSliceB = kOzN * kOzKStep * 2;        // bytes of one B slice tile (64 x 32 bf16)
constexpr int kOzGroup = 128 / kOzKStep;              // chunks whose FP32 sums of slice products stay exact
constexpr int kOzWays = 4;                            // diagonals whose products alternate
constexpr int kOzEpiWarps = 8;
constexpr int kOzThreads = 32 * (2 + kOzEpiWarps);    // producer warp, MMA warp, epilogue warps
constexpr uint32_t kOzIdesc = tc::idesc_bf16(kOzM, kOzN);

// One factor of a product, read as n rows of K values (rows of op(A), columns of
// B: row r, value k at src[r rs + k ks], one of the strides 1), and its slices:
// blocks of `blk` rows x 32 k values, all S slices of a block one after the
// other, each in the K-major operand layout with 64-byte swizzle (rows of 32
// values, 8-row groups kOzSbo apart), so that a chunk of a tile is one contiguous
// copy.  The slices of the last row range end with its last row (padded to 128 rows, one
// row over 2^22 values of k took 7.5 GB); they are copied one by one.
constexpr int kOzRow = kOzKStep * 2;   // bytes of a row of a slice
struct OzSide : ScanSide {
    int nkc, blk;
    int64_t dst;         // bytes from the slice buffer to block (0, 0)
    int cut0;            // first CTA of this factor in k_oz_slice
};

// Exponents and slices.  e = the smallest integer with max |x| < 2^e; x 2^-(e+1)
// is a 56-bit signed fraction X (rounded to nearest where the 53 bits of x reach
// below it), rounded to b S bits, whose balanced digits are the slices: integer
// operations only (an FP64 digit costs four FP64 instructions, 0.4 ms at n = 2048
// on this GPU).  A warp writes 8 rows x 32 k values: lane
// (kg, r) the eight values k = 8 kg .. 8 kg + 7 of row r as one 16-byte store per
// slice, 512 contiguous bytes per warp.  Eight warps of a CTA cover eight chunks of
// k (rows contiguous in k) or eight row groups (rows contiguous across).
__global__ void __launch_bounds__(256) k_oz_slice(const OzSide* __restrict__ sides, int n_sides, int S, int bits,
                                                  const unsigned long long* __restrict__ mx, int* __restrict__ exps,
                                                  unsigned char* __restrict__ buf) {
    int f = 0;   // the last factor whose CTAs start at or before this one
    for (int hi = n_sides - 1; f < hi;) {
        const int mid = (f + hi + 1) >> 1;
        if (sides[mid].cut0 <= (int)blockIdx.x) f = mid;
        else hi = mid - 1;
    }
    const OzSide sd = sides[f];
    const int u = (int)blockIdx.x - sd.cut0, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int rg, kc;
    if (sd.ks == 1) {
        const int nk8 = (sd.nkc + 7) / 8;
        rg = u / nk8;
        kc = 8 * (u % nk8) + warp;
    } else {
        const int ng = ((sd.n + 7) / 8 + 7) / 8;
        rg = 8 * (u % ng) + warp;
        kc = u / ng;
    }
    if (kc >= sd.nkc || 8 * rg >= sd.n) return;
    const int r = 8 * rg + (lane & 7), kg = lane >> 3;
    const bool on = r < sd.n;
    const unsigned long long top = on ? mx[sd.row0 + r] : 0ull;
    int e = 0;
    if (top != 0ull) frexp(__longlong_as_double((long long)top), &e);   // max = m 2^e, 0.5 <= m < 1
    if (on && kc == 0 && kg == 0) exps[sd.row0 + r] = e;
    long long X[8];
    const int drop = 56 - bits * S, half = 1 << (bits - 1);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int k = kOzKStep * kc + 8 * kg + t;
        X[t] = 0;
        if (on && k < sd.K) {
            const unsigned long long b = ((const unsigned long long*)sd.src)[r * sd.rs + k * sd.ks];
            const int ef = (int)((b >> 52) & 0x7ff);
            const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (ef ? 1ull << 52 : 0ull);
            const int sh = (ef ? ef : 1) - 1023 - e + 3;   // |x| = m 2^(ef - 1075), |X| = |x| 2^(55 - e)
            unsigned long long f = 0ull;
            if (sh >= 0) f = m << min(sh, 63);   // (beyond 2 for subnormal x only)
            else if (sh > -55) f = (m + (1ull << (-sh - 1))) >> -sh;
            if (drop > 0) f = (f + (1ull << (drop - 1))) >> drop;
            X[t] = (b >> 63) ? -(long long)f : (long long)f;
        }
    }
    if (!on) return;
    const int row0 = r / sd.blk * sd.blk;   // of the block
    const int64_t slice = (int64_t)min(sd.blk, sd.n - row0) * kOzRow;
    unsigned char* dst = buf + sd.dst + (int64_t)row0 * sd.nkc * S * kOzRow + (int64_t)kc * S * slice +
                         (r - row0) * kOzRow + (kg ^ ((lane >> 1) & 3)) * 16;
    for (int p = S - 1; p >= 0; --p) {
        uint32_t w[4];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            // the lowest digit, in [-half, half) (the first one takes what is left, at most half)
            const int d = p ? (((int)X[t] + half) & (2 * half - 1)) - half : (int)X[t];
            X[t] = (X[t] - d) >> bits;
            // d as a float (1.5 2^23 + d - 1.5 2^23), whose upper half is the BF16 value
            const uint32_t h =
                __float_as_uint(__uint_as_float(0x4B400000u + (uint32_t)d) - 12582912.0f) >> 16;
            if (t & 1) w[t >> 1] |= h << 16;
            else w[t >> 1] = h;
        }
        *(uint4*)(dst + p * slice) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// One product of a group, C = alpha op(A) B, with its slices and exponents.
struct OzProd {
    double* C;
    int M, N, nkc, ldc;
    double alpha;
    int64_t a_off, b_off;   // bytes from the slice buffer to the blocks of op(A) (128 rows) and of B (64 columns)
    int e_off, f_off;       // row exponents of op(A), column exponents of B
};

struct OzTile {
    int prod, m0, n0;
};

// (hi 2^64 + lo) 2^sc rounded to nearest even, by integer operations.
__device__ __forceinline__ double oz_round(long long hi, unsigned long long lo, int sc) {
    const bool neg = hi < 0;
    unsigned long long h = (unsigned long long)hi;
    if (neg) {
        h = ~h;
        lo = ~lo + 1ull;
        h += lo == 0ull;
    }
    if ((h | lo) == 0ull) return 0.0;
    const int lz = h ? __clzll((long long)h) : 64 + __clzll((long long)lo);
    unsigned long long top, rest;
    if (lz >= 64) {
        top = lo << (lz - 64);
        rest = 0ull;
    } else {
        top = lz ? (h << lz) | (lo >> (64 - lz)) : h;
        rest = lo << lz;
    }
    unsigned long long m = top >> 11;
    const unsigned r = (unsigned)top & 0x7ffu;
    if (r > 0x400u || (r == 0x400u && (rest != 0ull || (m & 1ull)))) ++m;
    const int E = 127 - lz + sc;   // exponent of the leading bit
    if (E < -1022 || E > 1022) return ldexp(neg ? -(double)m : (double)m, E - 52);
    // m = 2^53 after a carry raises the exponent by one: the addition does it
    const unsigned long long b = ((unsigned long long)(E + 1022) << 52) + m;
    return __longlong_as_double((long long)(b | (neg ? 1ull << 63 : 0ull)));
}

// C (M x N, row-major, ldc) = alpha sum_d 2^{e_i + f_j + 2 - b(d + 2)} sum_{p + q = d + 2} A_p B_q
// (slices numbered from 1).  A persistent CTA per SM takes 128 x 64 output tiles:
//  - one thread copies chunks of 32 k values of every slice (84 KB at S = 7: two
//    contiguous pieces, cp.async.bulk) into a ring of stages;
//  - one thread issues a tcgen05.mma.kind::f16 (BF16 operands, FP32 accumulation)
//    per slice pair (p, q), p + q <= S + 1, and 16 values of k, into the
//    tensor-memory accumulator of its diagonal d = p + q - 2 (64 columns each),
//    diagonals in descending order;
//  - every 128 values of k (where the FP32 sums of integer slice products are
//    still exact) eight warps read a diagonal as soon as its last product is done
//    and add it, shifted to its weight, to two exact 64-bit integers per entry in
//    registers (below 2^46 per 128 values of k), and the next
//    products of that diagonal may restart it: the tensor cores wait only for the
//    first of the eight reads;
//  - at the end of a tile the two integers are combined and rounded once.
// What bounds it is the spacing of the MMAs: at n = 2048 the busiest SMs issue 14336 of 64 columns
// in 654 us, one per 91 cycles, where the multiplication takes 32 and the operand reads 48 (128 x 16 +
// 64 x 16 BF16 at 128 bytes per cycle; shared memory 54 % busy, tensor pipe 30 %).  A wider tile has no
// room in tensor memory beside seven or eight diagonals.
// Every mbarrier wait is bounded; whoever gives up sets *err and leaves, the
// others run out of their own waits, and the tensor memory is freed after a
// bounded wait for the MMAs and copies in flight.
template <int S>
constexpr int oz_stages() {
    return S * (kOzSliceA + kOzSliceB) * 4 <= 200 * 1024 ? 4 : 2;
}

// An integer below 2^24 in a float (b = 7: within 2^22) as an int: by FP32 additions, whose
// sums with 1.5 2^23 hold it in their last bits (a conversion instruction takes 32 cycles per
// warp and scheduler here).
template <int B>
__device__ __forceinline__ int oz_int(float v) {
    constexpr float kMagic = 12582912.0f;
    if (B == 7) return (int)__float_as_uint(v + kMagic) - 0x4B400000;
    const float h = fmaf(v, 0.25f, kMagic);                   // v / 4, rounded
    const float l = fmaf(h - kMagic, -4.0f, v) + kMagic;      // the rest, within 2
    return ((int)__float_as_uint(h) - 0x4B400000) * 4 + ((int)__float_as_uint(l) - 0x4B400000);
}

// The S slices of a chunk, `bytes` each, to `stride` bytes apart in shared memory.
template <int S>
__device__ __forceinline__ void load_slices(uint32_t dst, const unsigned char* src, uint32_t bytes, uint32_t stride,
                                            uint32_t bar) {
    if (bytes == stride) {
        tc::bulk_load(dst, src, S * stride, bar);
        return;
    }
    for (int p = 0; p < S; ++p) tc::bulk_load(dst + p * stride, src + (int64_t)p * bytes, bytes, bar);
}

template <int S, int B>
__global__ void __launch_bounds__(kOzThreads, 1) k_oz_gemm(const OzProd* __restrict__ prods,
                                                           const OzTile* __restrict__ tiles, int n_tiles,
                                                           const unsigned char* __restrict__ slices,
                                                           const int* __restrict__ exps, int* err) {
    constexpr uint32_t kCols = S * kOzN <= 64 ? 64 : S * kOzN <= 128 ? 128 : S * kOzN <= 256 ? 256 : 512;
    constexpr int kStages = oz_stages<S>();
    constexpr int kTop = B == 7 ? 7 : 6;   // last diagonal of the second integer
    constexpr uint32_t kBytesA = S * kOzSliceA, kBytesB = S * kOzSliceB, kStage = kBytesA + kBytesB;
    extern __shared__ __align__(1024) unsigned char oz_smem[];
    __shared__ __align__(8) uint64_t bars[2 * kStages + 2 * S + 1];
    __shared__ uint32_t tmem_slot;
    const uint32_t base = (tc::smem_addr(oz_smem) + 1023u) & ~1023u;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto full = [&](int s) { return tc::smem_addr(&bars[s]); };                          // a stage's copies landed
    auto empty = [&](int s) { return tc::smem_addr(&bars[kStages + s]); };               // its MMAs are done
    auto dfull = [&](int d) { return tc::smem_addr(&bars[2 * kStages + d]); };           // a diagonal's sums are done
    auto dempty = [&](int d) { return tc::smem_addr(&bars[2 * kStages + S + d]); };      // they have been read
    const uint32_t drain = tc::smem_addr(&bars[2 * kStages + 2 * S]);
    if (tid == 0) {
        for (int i = 0; i < 2 * kStages + 2 * S + 1; ++i) {
            const uint32_t count = i >= 2 * kStages + S && i < 2 * kStages + 2 * S ? kOzEpiWarps : 1;
            tc::mbar_init(tc::smem_addr(&bars[i]), count);
        }
        tc::mbar_init_fence();
    }
    if (warp == 1) tc::tmem_alloc(&tmem_slot, kCols);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_slot;
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            uint32_t it = 0;   // chunks issued: stage it % kStages, use it / kStages of its barriers
            for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
                const OzTile tl = tiles[t];
                const OzProd& pd = prods[tl.prod];
                const int nkc = pd.nkc;
                const unsigned char* a = slices + pd.a_off + (int64_t)tl.m0 * nkc * (S * kOzRow);
                const unsigned char* b = slices + pd.b_off + (int64_t)tl.n0 * nkc * (S * kOzRow);
                // bytes of a slice; the rows that the last blocks lack are whatever stands in shared
                // memory there (they reach only entries that are not stored)
                const uint32_t sa = (uint32_t)min(kOzM, pd.M - tl.m0) * kOzRow;
                const uint32_t sb = (uint32_t)min(kOzN, pd.N - tl.n0) * kOzRow;
                for (int c = 0; c < nkc; ++c, ++it) {
                    const int s = it % kStages;
                    if (it >= kStages && !tc::mbar_wait(empty(s), (it / kStages - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    const uint32_t dst = base + s * kStage;
                    tc::mbar_expect(full(s), S * (sa + sb));
                    load_slices<S>(dst, a + (int64_t)c * (S * sa), sa, kOzSliceA, full(s));
                    load_slices<S>(dst + kBytesA, b + (int64_t)c * (S * sb), sb, kOzSliceB, full(s));
                }
            }
            // copies in flight land before the CTA may end
            for (uint32_t i = it > kStages ? it - kStages : 0; i < it; ++i)
                tc::mbar_wait(full(i % kStages), (i / kStages) & 1);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            uint32_t it = 0, g = 0;   // g: groups of 128 values of k (uses of every diagonal)
            for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
                const int nkc = prods[tiles[t].prod].nkc;
                for (int c = 0; c < nkc && ok; ++c, ++it) {
                    const int s = it % kStages;
                    const bool first = c % kOzGroup == 0, last = c % kOzGroup == kOzGroup - 1 || c + 1 == nkc;
                    if (!tc::mbar_wait(full(s), (it / kStages) & 1)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after();
                    const uint64_t da = tc::desc_sw64(base + s * kStage);
                    const uint64_t db = tc::desc_sw64(base + s * kStage + kBytesA);
                    // consecutive MMAs go to kOzWays accumulators in turn (4 % faster than one after the
                    // other: one accumulator takes a new product of 64 columns every 75 cycles)
#pragma unroll
                    for (int d1 = S - 1; d1 >= 0; d1 -= kOzWays) {
                        const int d0 = d1 - kOzWays + 1 > 0 ? d1 - kOzWays + 1 : 0;
                        if (first && g > 0) {
#pragma unroll
                            for (int d = d1; d >= d0; --d) ok = ok && tc::mbar_wait(dempty(d), (g - 1) & 1);
                            if (!ok) break;
                            tc::fence_after();
                        }
#pragma unroll
                        for (int p = 0; p <= d1; ++p)
#pragma unroll
                            for (int kk = 0; kk < kOzKStep / 16; ++kk)
#pragma unroll
                                for (int d = d1; d >= d0; --d)
                                    if (p <= d)
                                        tc::mma_bf16(tmem + (uint32_t)(d * kOzN),
                                                     da + ((p * kOzSliceA + kk * 32) >> 4),
                                                     db + (((d - p) * kOzSliceB + kk * 32) >> 4), kOzIdesc,
                                                     first && p == 0 && kk == 0 ? 0u : 1u);
                        if (last)
#pragma unroll
                            for (int d = d1; d >= d0; --d) tc::commit(dfull(d));
                    }
                    tc::commit(empty(s));
                    if (last) ++g;
                }
            }
            // every MMA and every earlier commit has happened before the CTA ends
            tc::commit(drain);
            ok = tc::mbar_wait(drain, 0) && ok;
        }
        __syncwarp();
    } else {
        const int quad = warp & 3, half = (warp - 2) >> 2;   // tensor-memory lanes 32 quad .., columns 32 half ..
        uint32_t g = 0;
        for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
            const OzTile tl = tiles[t];
            const OzProd pd = prods[tl.prod];
            const int n_groups = (pd.nkc + kOzGroup - 1) / kOzGroup;
            long long i0[32], i1[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) i0[j] = i1[j] = 0;
            for (int q = 0; q < n_groups && ok; ++q, ++g) {
#pragma unroll
                for (int d = S - 1; d >= 0; --d) {
                    if (!__all_sync(0xffffffffu, tc::mbar_wait(dfull(d), g & 1))) {
                        ok = false;
                        break;
                    }
                    tc::fence_after();
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint32_t v[16];
                        tc::ld_32x32b_x16(
                            tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(d * kOzN + half * 32 + 16 * h), v);
                        if (h == 1) {
                            tc::fence_before();
                            __syncwarp();
                            if (lane == 0)
                                tc::mbar_arrive(dempty(d));
                        }
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const long long x = oz_int<B>(__uint_as_float(v[j]));
                            if (d < 4)
                                i0[16 * h + j] += x * (1 << (B * (3 - d)));
                            else
                                i1[16 * h + j] += x * (1 << (B * (kTop - d)));
                        }
                    }
                }
            }
            if (!ok) break;
            // diagonal d carries 2^(2 - B(d + 2)): C = (i0 2^(B (kTop - 3)) + i1) 2^(e + f + 2 - B (kTop + 2))
            constexpr int kUp = B * (kTop - 3);
            const int row = tl.m0 + quad * 32 + lane, c0 = tl.n0 + half * 32;
            if (row < pd.M) {
                const int e = exps[pd.e_off + row] + 2 - B * (kTop + 2);
                const int* f = exps + pd.f_off;
                double* out = pd.C + (int64_t)row * pd.ldc;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    if (c0 + j < pd.N) {
                        const unsigned long long l0 = (unsigned long long)i0[j] << kUp;
                        const unsigned long long lo = l0 + (unsigned long long)i1[j];
                        const long long hi = (i0[j] >> (64 - kUp)) + (i1[j] >> 63) + (lo < l0 ? 1 : 0);
                        const double v = oz_round(hi, lo, e + f[c0 + j]);
                        out[c0 + j] = pd.alpha == 1.0 ? v : pd.alpha * v;
                    }
                }
            }
        }
    }
    if (!ok) atomicExch(err, 1);
    tc::fence_before();
    __syncthreads();
    if (warp == 1) tc::tmem_free(tmem, kCols);
}

template <int S, int B = 7>
void launch_oz_gemm(Context* ctx, int n_tiles, const OzProd* prods, const OzTile* tiles, const unsigned char* slices,
                    const int* exps) {
    const size_t smem = (size_t)oz_stages<S>() * S * (kOzSliceA + kOzSliceB) + 1024;
    static bool attr = false;
    if (!attr) {
        BSM_CUDA(cudaFuncSetAttribute(k_oz_gemm<S, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        attr = true;
    }
    int nsm = 0;
    BSM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
    k_oz_gemm<S, B><<<std::min(n_tiles, nsm), kOzThreads, smem, ctx->stream>>>(prods, tiles, n_tiles, slices, exps,
                                                                            ctx->err_word());
}

}  // namespace

void launch_gemm_ozaki_group(Context* ctx, const std::vector<OzGemm>& gs, int slices_asked) {
    BSM_REQUIRE(slices_asked >= 1 && slices_asked <= kOzMaxS, BSMPS_ERR_INVALID_ARG, "emulated GEMM: 1 <= slices <= 8");
    const int bits = slices_asked == kOzMaxS ? 8 : 7, S = slices_asked == kOzMaxS ? 7 : slices_asked;
    std::vector<OzProd> prods;
    std::vector<OzSide> sides;
    std::vector<OzTile> tiles;
    int64_t bytes = 0;
    int rows = 0, max_ctas = 0, cut_ctas = 0;
    double fl = 0.0;
    auto side = [&](const double* src, int64_t rs, int64_t ks, int n, int K, int nkc, int blk) {
        const OzSide sd{{src, rs, ks, n, K, rows, max_ctas}, nkc, blk, bytes, cut_ctas};
        bytes += (int64_t)n * nkc * S * kOzRow;
        rows += n;
        const int groups = (n + 7) / 8;
        max_ctas += scan_ctas(ks, n, K);
        cut_ctas += ks == 1 ? groups * ((nkc + 7) / 8) : ((groups + 7) / 8) * nkc;
        sides.push_back(sd);
        return sd;
    };
    for (const OzGemm& g : gs) {
        BSM_REQUIRE(g.M >= 0 && g.N >= 0 && g.K >= 0, BSMPS_ERR_INVALID_ARG, "emulated GEMM: sizes >= 0");
        // the exact 64-bit sums of the diagonals (below 2^46 per 128 values of k) stay below 2^63
        BSM_REQUIRE(g.K < (1 << 24), BSMPS_ERR_INVALID_ARG, "emulated GEMM: K < 2^24");
        if (g.M == 0 || g.N == 0) continue;
        const int nkc = (g.K + kOzKStep - 1) / kOzKStep;
        // (a stride-1 row of one value each counts as contiguous in k)
        const OzSide a = side(g.A, g.lda, 1, g.M, g.K, nkc, kOzM);
        const OzSide b = side(g.B, 1, g.ldb, g.N, g.K, nkc, kOzN);
        for (int m0 = 0; m0 < g.M; m0 += kOzM)
            for (int n0 = 0; n0 < g.N; n0 += kOzN) tiles.push_back({(int)prods.size(), m0, n0});
        prods.push_back({g.C, g.M, g.N, nkc, g.ldc, g.alpha, a.dst, b.dst, a.row0, b.row0});
        fl += 2.0 * g.M * (double)g.N * g.K;
    }
    if (prods.empty()) return;
    Scratch s(ctx);
    unsigned char* slices = (unsigned char*)ctx->alloc((size_t)bytes + 128);
    s.ptrs.push_back(slices);
    unsigned long long* mx = (unsigned long long*)ctx->alloc(sizeof(unsigned long long) * (size_t)rows);
    s.ptrs.push_back(mx);
    int* exps = (int*)ctx->alloc(sizeof(int) * (size_t)rows);
    s.ptrs.push_back(exps);
    const OzSide* d_sides = s.up(sides);
    const OzProd* d_prods = s.up(prods);
    const OzTile* d_tiles = s.up(tiles);
    BSM_CUDA(cudaMemsetAsync(mx, 0, sizeof(unsigned long long) * (size_t)rows, ctx->stream));
    k_row_max<OzSide><<<max_ctas, 256, 0, ctx->stream>>>(d_sides, (int)sides.size(), mx);
    launched(ctx);
    if (cut_ctas > 0) {
        k_oz_slice<<<cut_ctas, 256, 0, ctx->stream>>>(d_sides, (int)sides.size(), S, bits, mx, exps, slices);
        launched(ctx);
    } else {
        BSM_CUDA(cudaMemsetAsync(exps, 0, sizeof(int) * (size_t)rows, ctx->stream));   // K = 0: C = 0
    }
    const int nt = (int)tiles.size();
    switch (slices_asked) {
        case 1: launch_oz_gemm<1>(ctx, nt, d_prods, d_tiles, slices, exps); break;
        case 2: launch_oz_gemm<2>(ctx, nt, d_prods, d_tiles, slices, exps); break;
        case 3: launch_oz_gemm<3>(ctx, nt, d_prods, d_tiles, slices, exps); break;
        case 4: launch_oz_gemm<4>(ctx, nt, d_prods, d_tiles, slices, exps); break;
        case 5: launch_oz_gemm<5>(ctx, nt, d_prods, d_tiles, slices, exps); break;
        case 6: launch_oz_gemm<6>(ctx, nt, d_prods, d_tiles, slices, exps); break;
        case 7: launch_oz_gemm<7>(ctx, nt, d_prods, d_tiles, slices, exps); break;
        default: launch_oz_gemm<7, 8>(ctx, nt, d_prods, d_tiles, slices, exps); break;
    }
    launched(ctx);
    ctx->flops += fl;
}

void launch_gemm_ozaki(Context* ctx, int M, int N, int K, const double* A, int lda, const double* B, int ldb,
                       double* C, int ldc, int S, double alpha) {
    launch_gemm_ozaki_group(ctx, {OzGemm{A, B, C, M, N, K, lda, ldb, ldc, alpha}}, S);
}

}  // namespace bsm
