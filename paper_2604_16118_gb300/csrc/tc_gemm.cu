// Grouped FP64-in / FP64-out GEMM on the 5th-generation tensor cores in split
// precision (3xTF32): every operand value v (scaled by its contribution's alpha)
// is split into v_hi (its leading 11 significant bits) and v_lo = tf32(v - v_hi),
// by integer operations on the FP64 bit pattern, and a tile accumulates
// A_hi B_hi + A_hi B_lo + A_lo B_hi in FP32 in tensor memory (the A_lo B_lo term,
// below 2^-21 relative, is dropped).  The relative error of an entry is a few
// units of 2^-21 times sum_k |a_ik| |b_kj| plus the FP32 accumulation error.
//
// Every row i of a tile is scaled by 2^-e_i and every column j by 2^-f_j before
// the split, with e_i (f_j) the exponent of the largest |alpha a_ik| (|b_kj|)
// over all contributions of the output: the scaling is exact, keeps every
// operand in TF32's range whatever the magnitudes of the FP64 data (MPS blocks
// can carry factors far outside the FP32 range), and is undone in FP64 when the
// tile is stored (C_ij = acc_ij 2^(e_i + f_j)).
//
// One CTA computes one 128 x 64 output tile of one grouped-GEMM output: 4 warps
// stage 32-wide k chunks of every contribution in shared memory (FP64 loads,
// split, canonical K-major layout without swizzle), one thread issues the
// tcgen05.mma instructions and commits them to an mbarrier, and at the end the
// four warps read their 32 accumulator lanes with tcgen05.ld.  Every wait on the
// mbarrier is bounded by the global timer; a CTA that gives up sets the device
// error word, waits (bounded) for its own MMAs, frees its tensor memory and
// returns.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "kernels.h"
#include "row_scan.cuh"
#include "tc_common.cuh"

namespace bsm {
namespace {

constexpr int kTcM = 128;         // rows of a tile: the M of one tcgen05.mma (cta_group::1)
constexpr int kTcN = 64;          // columns of a tile: the N of one tcgen05.mma, also the TMEM columns
constexpr int kTcK = 32;          // k values per staged chunk (4 MMAs of K = 8 for tf32)
constexpr int kTcThreads = 128;   // warp w reads TMEM lanes 32 w .. 32 w + 31
constexpr int kTcOperandBytes = (2 * kTcM + 2 * kTcN) * kTcK * 4;   // A_hi, A_lo, B_hi, B_lo

struct TcTile {
    int out, m0, n0;
};

constexpr uint32_t kTcIdesc = tc::idesc_tf32(kTcM, kTcN);
using tc::global_ns;
using tc::mbar_wait;
using tc::smem_addr;
using tc::tf32_bits;

__device__ __forceinline__ uint32_t tc_off(int r, int k) { return tc::off(r, k); }
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) { return tc::desc(saddr); }

// v 2^-sc for the FP64 value with bit pattern `bits`, split into TF32 parts
// (FP32 bit patterns) by integer operations only (this GPU's FP64 pipe retires
// one warp instruction per 16 cycles per SM): hi = the leading 11 significant
// bits (truncated), lo = the rest rounded to TF32, so |v 2^-sc - hi - lo| <=
// 2^-22 |v 2^-sc|.  The scaling is an exponent subtraction (exact); a scaled
// value below FP32's normal range (2^-126 of a row or column maximum brought
// to [1, 2)) becomes 0, as do FP64 zeros and subnormals.
__device__ __forceinline__ void split_scaled(unsigned long long bits, int sc, uint32_t* hi, uint32_t* lo) {
    const uint32_t sign = (uint32_t)(bits >> 32) & 0x80000000u;
    const int e = (int)((bits >> 52) & 0x7ff);
    const int E = e - 1023 - sc;
    if (e == 0 || E < -126) {
        *hi = *lo = 0u;
        return;
    }
    const unsigned long long m = bits & 0xFFFFFFFFFFFFFull;   // 52 fraction bits
    *hi = sign | ((uint32_t)(E + 127) << 23) | ((uint32_t)(m >> 42) << 13);
    const unsigned long long r = m & ((1ull << 42) - 1);      // value r 2^(E - 52)
    if (r == 0ull) {
        *lo = 0u;
        return;
    }
    const int lz = __clzll((long long)r);                      // leading one at bit 63 - lz
    const int El = E - 52 + (63 - lz);
    if (El < -126) {
        *lo = 0u;
        return;
    }
    const uint32_t frac = (uint32_t)((r << (lz + 1)) >> 41);   // the 23 bits after the leading one
    *lo = (((sign | ((uint32_t)(El + 127) << 23) | frac) + 0x1000u) & 0xFFFFE000u);
}

// acc 2^sh in FP64 from the FP32 accumulator bits by exponent arithmetic, with
// ldexp only for FP32 subnormals and results outside the FP64 normal range.
__device__ __forceinline__ double scale_out(uint32_t a, int sh) {
    const int e = (int)((a >> 23) & 0xff);
    if (e == 0 || e == 255) return ldexp((double)__uint_as_float(a), sh);
    const int E = e - 127 + sh + 1023;
    if (E <= 0 || E >= 2047) return ldexp((double)__uint_as_float(a), sh);
    const unsigned long long b = ((unsigned long long)(a & 0x80000000u) << 32) | ((unsigned long long)E << 52) |
                                 ((unsigned long long)(a & 0x7FFFFFu) << 29);
    return __longlong_as_double((long long)b);
}

// Exponent e with 2^-e x in [1, 2) for the largest magnitude x given by its bit
// pattern (0 for x = 0: such rows and columns hold zeros only).
__device__ __forceinline__ int pow2_exponent(unsigned long long bits) {
    if (bits == 0ull) return 0;
    return (int)((bits >> 52) & 0x7ff) - 1023;
}

__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    tc::mma_tf32(tmem, adesc, bdesc, kTcIdesc, accumulate);
}

__global__ void __launch_bounds__(kTcThreads) k_gemm_tf32x3(const GemmOut* __restrict__ outs,
                                                           const GemmIn* __restrict__ ins,
                                                           const TcTile* __restrict__ tiles, int* err) {
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int gave_up;
    __shared__ unsigned long long row_max[kTcM], col_max[kTcN];
    __shared__ int row_sc[kTcM], col_sc[kTcN];
    unsigned char* base = (unsigned char*)(((uintptr_t)tc_smem + 1023) & ~(uintptr_t)1023);
    unsigned char* a_hi = base;
    unsigned char* a_lo = a_hi + kTcM * kTcK * 4;
    unsigned char* b_hi = a_lo + kTcM * kTcK * 4;
    unsigned char* b_lo = b_hi + kTcN * kTcK * 4;
    const TcTile tl = tiles[blockIdx.x];
    const GemmOut o = outs[tl.out];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar_a = smem_addr(&bar);

    if (threadIdx.x == 0) {
        gave_up = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    // row and column scales: largest magnitudes (as ordered bit patterns of
    // non-negative doubles) over every contribution, then powers of two
    for (int r = threadIdx.x; r < kTcM; r += kTcThreads) row_max[r] = 0ull;
    for (int c = threadIdx.x; c < kTcN; c += kTcThreads) col_max[c] = 0ull;
    __syncthreads();
    // magnitudes compared as integers (the bit patterns of non-negative doubles
    // are ordered like their values)
    constexpr unsigned long long kAbs = 0x7FFFFFFFFFFFFFFFull;
    for (int c = o.beg; c < o.end; ++c) {
        const GemmIn in = ins[c];
        const double aa = fabs(in.alpha);
        const unsigned long long* Ab = (const unsigned long long*)in.A;
        const unsigned long long* Bb = (const unsigned long long*)in.B;
        for (int r = warp; r < kTcM; r += kTcThreads / 32) {
            const int gm = tl.m0 + r;
            if (gm >= o.M) break;
            unsigned long long mx = 0ull;
            for (int k = lane; k < in.K; k += 32) mx = max(mx, Ab[(int64_t)gm * in.lda + k] & kAbs);
            for (int d = 16; d > 0; d >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, d));
            const double mxa = __longlong_as_double((long long)mx) * aa;
            if (lane == 0 && mxa > 0.0) atomicMax(&row_max[r], (unsigned long long)__double_as_longlong(mxa));
        }
        for (int n = threadIdx.x; n < kTcN; n += kTcThreads) {
            const int gn = tl.n0 + n;
            if (gn >= o.N) continue;
            unsigned long long mx = 0ull;
            for (int k = 0; k < in.K; ++k) mx = max(mx, Bb[(int64_t)k * in.ldb + gn] & kAbs);
            if (mx > 0ull) atomicMax(&col_max[n], mx);
        }
    }
    __syncthreads();
    for (int r = threadIdx.x; r < kTcM; r += kTcThreads) row_sc[r] = pow2_exponent(row_max[r]);
    for (int c = threadIdx.x; c < kTcN; c += kTcThreads) col_sc[c] = pow2_exponent(col_max[c]);
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                     "r"(kTcN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_slot;

    uint32_t n_commits = 0;
    for (int c = o.beg; c < o.end; ++c) {
        const GemmIn in = ins[c];
        for (int k0 = 0; k0 < in.K; k0 += kTcK) {
            // the chunk before this one must have been consumed by the tensor cores
            if (n_commits > 0) {
                if (!mbar_wait(bar_a, (n_commits - 1) & 1)) {
                    if (threadIdx.x == 0) atomicExch(&gave_up, 1);
                }
                __syncthreads();
                if (gave_up) goto finish;
            }
            // A: rows m0 .. m0 + 127, k0 .. k0 + 31 (alpha folded in), split into hi / lo
            for (int idx = threadIdx.x; idx < kTcM * kTcK; idx += kTcThreads) {
                const int r = idx / kTcK, k = idx % kTcK;
                const int gm = tl.m0 + r, gk = k0 + k;
                uint32_t hi = 0u, lo = 0u;
                if (gm < o.M && gk < in.K)
                    split_scaled((unsigned long long)__double_as_longlong(in.alpha * in.A[(int64_t)gm * in.lda + gk]),
                                 row_sc[r], &hi, &lo);
                const uint32_t off = tc_off(r, k);
                *(uint32_t*)(a_hi + off) = hi;
                *(uint32_t*)(a_lo + off) = lo;
            }
            // B: k0 .. k0 + 31 x columns n0 .. n0 + 63, stored K-major (row = column n)
            for (int idx = threadIdx.x; idx < kTcN * kTcK; idx += kTcThreads) {
                const int k = idx / kTcN, n = idx % kTcN;
                const int gk = k0 + k, gn = tl.n0 + n;
                uint32_t hi = 0u, lo = 0u;
                if (gk < in.K && gn < o.N)
                    split_scaled(((const unsigned long long*)in.B)[(int64_t)gk * in.ldb + gn], col_sc[n], &hi, &lo);
                const uint32_t off = tc_off(n, k);
                *(uint32_t*)(b_hi + off) = hi;
                *(uint32_t*)(b_lo + off) = lo;
            }
            // generic-proxy writes become visible to the tensor cores' (async) proxy
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (threadIdx.x == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t sa_hi = smem_addr(a_hi), sa_lo = smem_addr(a_lo);
                const uint32_t sb_hi = smem_addr(b_hi), sb_lo = smem_addr(b_lo);
                for (int kk = 0; kk < kTcK / 8; ++kk) {
                    const uint32_t step = (uint32_t)kk * 256u;   // two core matrices along k per MMA
                    const uint32_t first = (n_commits == 0 && kk == 0) ? 0u : 1u;
                    tc_mma(tmem, tc_desc(sa_lo + step), tc_desc(sb_hi + step), first);
                    tc_mma(tmem, tc_desc(sa_hi + step), tc_desc(sb_lo + step), 1u);
                    tc_mma(tmem, tc_desc(sa_hi + step), tc_desc(sb_hi + step), 1u);
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 bar_a)
                             : "memory");
            }
            ++n_commits;
        }
    }
    if (n_commits > 0) {
        if (!mbar_wait(bar_a, (n_commits - 1) & 1)) {
            if (threadIdx.x == 0) atomicExch(&gave_up, 1);
        }
        __syncthreads();
        if (gave_up) goto finish;
        asm volatile("tcgen05.fence::after_thread_sync;");
    }
    {
        // warp w holds rows m0 + 32 w + lane of the tile
        const int row = tl.m0 + warp * 32 + lane;
        for (int c0 = 0; c0 < kTcN; c0 += 16) {
            uint32_t v[16];
            if (n_commits > 0) {
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
                    "%12, %13, %14, %15}, [%16];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                      "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
                      "=r"(v[14]), "=r"(v[15])
                    : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = 0u;
            }
            if (row < o.M) {
                double* cr = o.C + (int64_t)row * o.ldc;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int col = tl.n0 + c0 + j;
                    const double acc = scale_out(v[j], row_sc[warp * 32 + lane] + col_sc[c0 + j]);
                    if (col < o.N) cr[col] = o.beta == 0.0 ? acc : o.beta * cr[col] + acc;
                }
            }
        }
    }
finish:
    if (gave_up) {
        if (threadIdx.x == 0) atomicExch(err, 1);
        // MMAs of this CTA may still be in flight: give them a bounded wait before
        // the tensor memory they write is released
        if (n_commits > 0) mbar_wait(bar_a, (n_commits - 1) & 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcN));
}

// ---- one large product: operands split once, then a pipelined GEMM ----
//
// The grouped kernel above splits the operands of every tile again (each value of
// A once per 64 columns of C) and scans them for the scales first; for one product
// of 3000 x 1100 x 700 that took 800 us.  Here k_row_max finds the scales, k_tc_split
// writes the TF32 parts once, in operand layout (128 rows x 32 k values per block,
// 128-byte swizzle: the high parts, then the low parts; the blocks of the last row range
// end with its last row), and k_gemm_split streams blocks by bulk copies through a ring of
// stages: the same products in the same order per entry.  Workspace: 8 bytes per value of
// the factors, K rounded up to 32; where the device has no room for it the grouped
// kernel, which needs none, takes the product.

// One factor with its split blocks and power-of-two exponents (alpha folded into A).
struct SplitSide : ScanSide {
    int nkc;
    double alpha;
    int is_b;
    int64_t dst;   // bytes from the buffer to block (0, 0)
    int cut0;      // first CTA in k_tc_split
};

constexpr int kSpTile = 128;                          // rows and columns of a tile
constexpr int kSpRow = kTcK * 4;                      // bytes of a row of a part
constexpr uint32_t kSpPart = kSpTile * kSpRow;        // bytes of the high (or low) parts of a full block
constexpr uint32_t kSpStage = 4 * kSpPart;            // A and B blocks of one chunk
constexpr int kSpStages = 3;
constexpr int kSpThreads = 192;                       // producer warp, MMA warp, four epilogue warps
constexpr uint32_t kSpIdesc = tc::idesc_tf32(kSpTile, kSpTile);

// One warp writes 8 rows x 32 k values: a lane four values of k (16 bytes of each part) twice.
__global__ void __launch_bounds__(256) k_tc_split(const SplitSide* __restrict__ sides,
                                                  const unsigned long long* __restrict__ mx, int* __restrict__ exps,
                                                  unsigned char* __restrict__ buf) {
    const SplitSide sd = sides[(int)blockIdx.x >= sides[1].cut0 ? 1 : 0];
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
    const int row0 = 8 * rg / kSpTile * kSpTile;   // of the block
    const int64_t part = (int64_t)min(kSpTile, sd.n - row0) * kSpRow;
    unsigned char* dst =
        buf + sd.dst + (int64_t)row0 * sd.nkc * (2 * kSpRow) + kc * 2 * part + (8 * rg - row0) * kSpRow;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        // rows contiguous in k: eight lanes along k; rows contiguous across: eight lanes along the rows
        const int rr = sd.ks == 1 ? (lane >> 3) + 4 * h : lane & 7;
        const int kg = sd.ks == 1 ? lane & 7 : (lane >> 3) + 4 * h;
        const int r = 8 * rg + rr;
        const unsigned long long top = r < sd.n ? mx[sd.row0 + r] : 0ull;
        // (the columns of B have no factor; their largest bit pattern decides as it is)
        const double mxa = __longlong_as_double((long long)top) * fabs(sd.alpha);
        const int sc = sd.is_b ? pow2_exponent(top)
                                             : mxa > 0.0 ? pow2_exponent((unsigned long long)__double_as_longlong(mxa)) : 0;
        if (r < sd.n && kc == 0 && kg == 0) exps[sd.row0 + r] = sc;
        if (r >= sd.n) continue;
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int k = kTcK * kc + 4 * kg + t;
            hi[t] = lo[t] = 0u;
            if (k < sd.K)
                split_scaled(
                    (unsigned long long)__double_as_longlong(sd.alpha * sd.src[(int64_t)r * sd.rs + k * sd.ks]), sc,
                    &hi[t], &lo[t]);
        }
        unsigned char* o = dst + rr * kSpRow + (kg ^ rr) * 16;
        *(uint4*)o = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *(uint4*)(o + part) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
}

// High and low parts of one block (`part` bytes each) to kSpPart apart in shared memory; the
// rows that a last block lacks are whatever stands there (they reach only entries that are not stored).
__device__ __forceinline__ void load_parts(uint32_t dst, const unsigned char* src, uint32_t part, uint32_t bar) {
    if (part == kSpPart) {
        tc::bulk_load(dst, src, 2 * kSpPart, bar);
        return;
    }
    tc::bulk_load(dst, src, part, bar);
    tc::bulk_load(dst + kSpPart, src + part, part, bar);
}

// C tile (128 x 128 per CTA): one thread streams the chunks (64 KB each) into three
// stages, one issues 12 MMAs per chunk (A_lo B_hi, A_hi B_lo, A_hi B_hi per 8 values of k),
// four warps read the accumulators and store FP64.  Waits bounded as above; the wait for the
// last product covers all of K (0.4 us a chunk) and has another second for every 65536 chunks.
// Tiles in one grid dimension, rows first (the others end at 65535).
__global__ void __launch_bounds__(kSpThreads, 1) k_gemm_split(const GemmOut o, int nkc, int e_a, int e_b,
                                                              const unsigned char* __restrict__ A,
                                                              const unsigned char* __restrict__ B,
                                                              const int* __restrict__ exps, int* err) {
    extern __shared__ __align__(1024) unsigned char sp_smem[];
    __shared__ __align__(8) uint64_t bars[2 * kSpStages + 1];
    __shared__ uint32_t tmem_slot;
    const uint32_t base = (smem_addr(sp_smem) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tm = (o.M + kSpTile - 1) / kSpTile;
    const int m0 = (int)(blockIdx.x % tm) * kSpTile, n0 = (int)(blockIdx.x / tm) * kSpTile;
    auto full = [&](int s) { return smem_addr(&bars[s]); };
    auto empty = [&](int s) { return smem_addr(&bars[kSpStages + s]); };
    const uint32_t done = smem_addr(&bars[2 * kSpStages]);
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * kSpStages + 1; ++i) tc::mbar_init(smem_addr(&bars[i]), 1);
        tc::mbar_init_fence();
    }
    if (warp == 1) tc::tmem_alloc(&tmem_slot, kSpTile);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_slot;
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            const unsigned char* a = A + (int64_t)m0 * nkc * (2 * kSpRow);
            const unsigned char* b = B + (int64_t)n0 * nkc * (2 * kSpRow);
            const uint32_t pa = min(kSpTile, o.M - m0) * kSpRow, pb = min(kSpTile, o.N - n0) * kSpRow;
            int c = 0;
            for (; c < nkc; ++c) {
                const int s = c % kSpStages;
                if (c >= kSpStages && !mbar_wait(empty(s), (c / kSpStages - 1) & 1)) {
                    ok = false;
                    break;
                }
                const uint32_t dst = base + s * kSpStage;
                tc::mbar_expect(full(s), 2 * (pa + pb));
                load_parts(dst, a + (int64_t)c * (2 * pa), pa, full(s));
                load_parts(dst + 2 * kSpPart, b + (int64_t)c * (2 * pb), pb, full(s));
            }
            // copies in flight land before the CTA may end
            for (int i = c > kSpStages ? c - kSpStages : 0; i < c; ++i)
                mbar_wait(full(i % kSpStages), (i / kSpStages) & 1);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            for (int c = 0; c < nkc; ++c) {
                const int s = c % kSpStages;
                if (!mbar_wait(full(s), (c / kSpStages) & 1)) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                const uint64_t a_hi = tc::desc_sw128(base + s * kSpStage), a_lo = a_hi + (kSpPart >> 4);
                const uint64_t b_hi = a_hi + (2 * kSpPart >> 4), b_lo = a_hi + (3 * kSpPart >> 4);
#pragma unroll
                for (int kk = 0; kk < kTcK / 8; ++kk) {
                    const uint64_t step = (uint64_t)kk * 2;   // 32 bytes along k
                    tc::mma_tf32(tmem, a_lo + step, b_hi + step, kSpIdesc, c == 0 && kk == 0 ? 0u : 1u);
                    tc::mma_tf32(tmem, a_hi + step, b_lo + step, kSpIdesc, 1u);
                    tc::mma_tf32(tmem, a_hi + step, b_hi + step, kSpIdesc, 1u);
                }
                tc::commit(empty(s));
            }
            tc::commit(done);   // covers every MMA and every earlier commit
            ok = mbar_wait(done, 0) && ok;
        }
        __syncwarp();
    } else {
        ok = false;
        for (int i = 0; i <= nkc >> 16 && !ok; ++i) ok = __all_sync(0xffffffffu, mbar_wait(done, 0));
        tc::fence_after();
        const int quad = warp & 3, row = m0 + quad * 32 + lane;
        const int e = row < o.M ? exps[e_a + row] : 0;
        for (int c0 = 0; ok && c0 < kSpTile; c0 += 16) {
            uint32_t v[16];
            tc::ld_32x32b_x16(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0, v);
            if (row < o.M) {
                double* cr = o.C + (int64_t)row * o.ldc;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int col = n0 + c0 + j;
                    if (col < o.N) {
                        const double acc = scale_out(v[j], e + exps[e_b + col]);
                        cr[col] = o.beta == 0.0 ? acc : o.beta * cr[col] + acc;
                    }
                }
            }
        }
    }
    if (!ok) atomicExch(err, 1);
    tc::fence_before();
    __syncthreads();
    if (warp == 1) tc::tmem_free(tmem, kSpTile);
}

// false, with nothing launched: no room for the parts on the device.
bool launch_gemm_split(Context* ctx, const GemmOut& o, const GemmIn& in, int kind) {
    const int nkc = (in.K + kTcK - 1) / kTcK;
    std::vector<SplitSide> sides;
    int64_t bytes = 0;
    int rows = 0, max_ctas = 0, cut_ctas = 0;
    auto side = [&](const double* src, int64_t rs, int64_t ks, int n, double alpha, int is_b) {
        sides.push_back({{src, rs, ks, n, in.K, rows, max_ctas}, nkc, alpha, is_b, bytes, cut_ctas});
        bytes += (int64_t)n * nkc * (2 * kSpRow);
        rows += n;
        const int groups = (n + 7) / 8;
        max_ctas += scan_ctas(ks, n, in.K);
        cut_ctas += ks == 1 ? groups * ((nkc + 7) / 8) : ((groups + 7) / 8) * nkc;
    };
    side(in.A, in.lda, 1, o.M, in.alpha, 0);
    side(in.B, 1, in.ldb, o.N, 1.0, 1);
    Scratch s(ctx);
    unsigned char* buf = nullptr;
    try {
        buf = (unsigned char*)ctx->alloc((size_t)bytes);
    } catch (const Error& e) {
        if (e.code != BSMPS_ERR_OOM) throw;
        (void)cudaGetLastError();
        return false;
    }
    s.ptrs.push_back(buf);
    const double fl = 2.0 * o.M * (double)o.N * in.K;
    const double by = 8.0 * ((double)o.M * in.K + (double)in.K * o.N + o.M * (double)o.N * (o.beta == 0.0 ? 1.0 : 2.0));
    ctx->flops += fl;
    unsigned long long* mx = (unsigned long long*)ctx->alloc(sizeof(unsigned long long) * (size_t)rows);
    s.ptrs.push_back(mx);
    int* exps = (int*)ctx->alloc(sizeof(int) * (size_t)rows);
    s.ptrs.push_back(exps);
    const SplitSide* d_sides = s.up(sides);
    const int smem = kSpStages * (int)kSpStage + 1024;
    static bool attr = false;
    if (!attr) {
        BSM_CUDA(cudaFuncSetAttribute(k_gemm_split, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        attr = true;
    }
    BSM_CUDA(cudaMemsetAsync(mx, 0, sizeof(unsigned long long) * (size_t)rows, ctx->stream));
    ProfScope ps(ctx, kind, fl, by);
    k_row_max<SplitSide><<<max_ctas, 256, 0, ctx->stream>>>(d_sides, 2, mx);
    check_launch(ctx);
    k_tc_split<<<cut_ctas, 256, 0, ctx->stream>>>(d_sides, mx, exps, buf);
    check_launch(ctx);
    const unsigned tiles = (unsigned)((o.M + kSpTile - 1) / kSpTile) * (unsigned)((o.N + kSpTile - 1) / kSpTile);
    k_gemm_split<<<tiles, kSpThreads, smem, ctx->stream>>>(o, nkc, sides[0].row0, sides[1].row0, buf + sides[0].dst,
                                                          buf + sides[1].dst, exps, ctx->err_word());
    check_launch(ctx);
    ps.done();
    return true;
}

}  // namespace

bool gemm_tf32x3_eligible(const std::vector<GemmOut>& outs, const std::vector<GemmIn>& ins) {
    for (const GemmOut& g : outs)
        for (int c = g.beg; c < g.end; ++c)
            if (ins[c].transA) return false;
    return true;
}

void launch_gemm_tf32x3(Context* ctx, const std::vector<GemmOut>& outs, const std::vector<GemmIn>& ins, int kind) {
    if (outs.empty()) return;
    // One product with one contribution (bsmps_gemm_tf32x3, a contraction with a single block): split
    // once.  Below 2^17 multiplications its three launches cost more than the grouped kernel's repeated splits
    // save, and so they do where few rows meet short sums (the columns are split once either way,
    // and their parts padded to 32 values of k and written to memory): rows x columns x k, grouped
    // against split, 1 x 131072 x 1 76 and 146 us, 1 x 20000 x 64 51 and 63, x 128 76 and 65; 16 x 20000 x
    // 32 44 and 61, x 80 66 and 63; 32 x 20000 x 32 52 and 66, x 64 72 and 71; 64 x 20000 x 32 72 and 71.
    // The grouped launches of the zip-up stay on the grouped kernel (the scales there span several
    // contributions).
    if (outs.size() == 1 && outs[0].end == outs[0].beg + 1 && !ins[outs[0].beg].transA && outs[0].M > 0 &&
        outs[0].N > 0 && ins[outs[0].beg].K > 0) {
        const GemmIn& in = ins[outs[0].beg];
        const int nkc = (in.K + kTcK - 1) / kTcK;
        if ((double)outs[0].M * outs[0].N * in.K >= (double)(1 << 17) && (nkc >= 4 || outs[0].M >= (128 >> nkc)) &&
            launch_gemm_split(ctx, outs[0], in, kind))
            return;
    }
    std::vector<TcTile> tiles;
    double fl = 0.0, by = 0.0;
    for (int o = 0; o < (int)outs.size(); ++o) {
        const GemmOut& g = outs[o];
        if (g.M <= 0 || g.N <= 0) continue;
        for (int m0 = 0; m0 < g.M; m0 += kTcM)
            for (int n0 = 0; n0 < g.N; n0 += kTcN) tiles.push_back({o, m0, n0});
        for (int c = g.beg; c < g.end; ++c) {
            BSM_REQUIRE(!ins[c].transA, BSMPS_ERR_INVALID_ARG, "split-precision GEMM: untransposed operands only");
            fl += 2.0 * g.M * g.N * (double)ins[c].K;
            by += 8.0 * ((double)g.M * ins[c].K + (double)ins[c].K * g.N);
        }
        by += 8.0 * g.M * (double)g.N * (g.beta == 0.0 ? 1.0 : 2.0);
    }
    if (tiles.empty()) return;
    ctx->flops += fl;
    Scratch s(ctx);
    const GemmOut* d_outs = s.up(outs);
    const GemmIn* d_ins = ins.empty() ? nullptr : s.up(ins);
    const TcTile* d_tiles = s.up(tiles);
    const int smem = kTcOperandBytes + 1024;   // room to align the operand tiles to 1024 bytes
    static bool attr_set = false;
    if (!attr_set) {
        BSM_CUDA(cudaFuncSetAttribute(k_gemm_tf32x3, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        attr_set = true;
    }
    ProfScope ps(ctx, kind, fl, by);
    k_gemm_tf32x3<<<(unsigned)tiles.size(), kTcThreads, smem, ctx->stream>>>(d_outs, d_ins, d_tiles,
                                                                             ctx->err_word());
    check_launch(ctx);
    ps.done();
}

}  // namespace bsm
