// Largest magnitudes of the rows (or columns) of FP64 factors, the first pass of
// the products that scale their operands by powers of two before they cut or
// split them.
#pragma once

#include <algorithm>
#include <cstdint>

namespace bsm {

// n rows of K values: row r, value k at src[r rs + k ks], one of the strides 1.
struct ScanSide {
    const double* src;
    int64_t rs, ks;
    int n, K;
    int row0;   // first row in the maxima
    int max0;   // first CTA of this factor
};

constexpr int kScanK = 128;
inline int scan_ctas(int64_t ks, int n, int K) {
    return ks == 1 ? (n + 7) / 8 : ((n + 31) / 32) * std::max(1, (K + kScanK - 1) / kScanK);
}

// mx[row0 + r] = the largest |x| of row r as a bit pattern (those of non-negative
// doubles are ordered like their values; mx zeroed before).  Rows contiguous in
// k: one warp per row, eight rows per CTA.  Rows contiguous across: 32 rows x 128
// values per CTA, whole 256-byte lines per load.  Side: ScanSide or derived from it.
template <class Side>
__global__ void __launch_bounds__(256) k_row_max(const Side* __restrict__ sides, int n_sides,
                                                 unsigned long long* __restrict__ mx) {
    int f = 0;
    for (int hi = n_sides - 1; f < hi;) {
        const int mid = (f + hi + 1) >> 1;
        if (sides[mid].max0 <= (int)blockIdx.x) f = mid;
        else hi = mid - 1;
    }
    const ScanSide sd = sides[f];
    const int u = (int)blockIdx.x - sd.max0, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr unsigned long long kAbs = 0x7FFFFFFFFFFFFFFFull;
    const unsigned long long* src = (const unsigned long long*)sd.src;
    unsigned long long m = 0ull;
    if (sd.ks == 1) {
        const int r = 8 * u + warp;
        if (r >= sd.n) return;
#pragma unroll 8
        for (int k = lane; k < sd.K; k += 32) m = max(m, src[(int64_t)r * sd.rs + k] & kAbs);
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) mx[sd.row0 + r] = m;
        return;
    }
    __shared__ unsigned long long part[8][32];
    const int nb = (sd.n + 31) / 32;
    const int r = 32 * (u % nb) + lane, k0 = (u / nb) * kScanK;
    if (r < sd.n)
#pragma unroll 8
        for (int k = k0 + warp; k < min(sd.K, k0 + kScanK); k += 8) m = max(m, src[r * sd.rs + k * sd.ks] & kAbs);
    part[warp][lane] = m;
    __syncthreads();
    if (warp == 0 && r < sd.n) {
        for (int w = 1; w < 8; ++w) m = max(m, part[w][lane]);
        atomicMax(&mx[sd.row0 + r], m);
    }
}

}  // namespace bsm
