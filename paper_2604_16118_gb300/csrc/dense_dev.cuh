// Block-cooperative dense FP64 routines (one CTA of kThreads threads works on
// one small matrix): reductions, Householder QR, one-sided Jacobi and the SVD
// assembly used by the truncation kernels.
#pragma once

#include <cfloat>
#include <cstdint>

namespace bsm {
namespace dev {

constexpr int kThreads = 256;            // default block size of the batched kernels
constexpr int kWarps = kThreads / 32;
constexpr int kMaxSweeps = 40;

// The routines below work with any block size that is a multiple of 32
// (callers size small problems down to fewer warps).
__device__ __forceinline__ int nthreads() { return (int)blockDim.x; }
__device__ __forceinline__ int nwarps() { return (int)(blockDim.x >> 5); }

// One 32 x 32 output tile of a grouped FP64 GEMM, accumulated over one
// contribution alpha op(A) B (op(A): M x K, transA selects A^T stored K x M):
// the thread (ty, tx) of a 256-thread CTA owns rows m0 + ty + 8 r (r < 4) and
// column n0 + tx.  The K loop stages 32 x 32 chunks of op(A) and B in shared
// memory (As[k][m], Bs[k][n]); only the valid part of a chunk and the rows
// below M issue FP64 instructions.  In: any struct with A, B, K, lda, ldb,
// transA and alpha.
constexpr int kGemmTile = 32;
template <class In>
__device__ __forceinline__ void gemm_tile_accumulate(const In& in, int M, int N, int m0, int n0,
                                                     double (*As)[kGemmTile + 1], double (*Bs)[kGemmTile + 1],
                                                     double acc[4]) {
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int k0 = 0; k0 < in.K; k0 += kGemmTile) {
        for (int idx = threadIdx.x; idx < kGemmTile * kGemmTile; idx += kThreads) {
            int mm, kk;
            if (in.transA) {
                kk = idx / kGemmTile;
                mm = idx % kGemmTile;
            } else {
                mm = idx / kGemmTile;
                kk = idx % kGemmTile;
            }
            const int gm = m0 + mm, gk = k0 + kk;
            double v = 0.0;
            if (gm < M && gk < in.K)
                v = in.transA ? in.A[(int64_t)gk * in.lda + gm] : in.A[(int64_t)gm * in.lda + gk];
            As[kk][mm] = in.alpha * v;
        }
        for (int idx = threadIdx.x; idx < kGemmTile * kGemmTile; idx += kThreads) {
            const int kk = idx / kGemmTile, nn = idx % kGemmTile;
            const int gk = k0 + kk, gn = n0 + nn;
            Bs[kk][nn] = (gk < in.K && gn < N) ? in.B[(int64_t)gk * in.ldb + gn] : 0.0;
        }
        __syncthreads();
        const int kk_end = min(kGemmTile, in.K - k0);
        for (int kk = 0; kk < kk_end; ++kk) {
            const double b = Bs[kk][tx];
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (m0 + ty + 8 * r < M) acc[r] = fma(As[kk][ty + 8 * r], b, acc[r]);
        }
        __syncthreads();
    }
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// sum over the block; every thread gets the result (red: 33 shared doubles)
__device__ __forceinline__ double block_sum(double v, double* red) {
    v = warp_sum(v);
    if (blockDim.x == 32) return v;   // one warp: no shared-memory stage
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        t = warp_sum(t);
        if (threadIdx.x == 0) red[32] = t;
    }
    __syncthreads();
    return red[32];
}

// Sum within aligned segments of S lanes (S a power of two, S <= 32); every
// lane of a segment receives its segment's sum.
__device__ __forceinline__ double seg_sum(double v, int S) {
    for (int o = S >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// acc + sum_{k < n} a[k sa] b[k sb] with the global loads issued eight terms
// at a time, so that a dot product of length n waits for about n/8 memory
// round trips instead of n.  CGA / CGB: loads of a / b through L2 (global
// data written by other CTAs of the same launch); otherwise plain loads (which
// also serve shared-memory operands).
template <bool CGA, bool CGB>
__device__ __forceinline__ double dot_global(const double* a, int64_t sa, const double* b, int64_t sb, int n,
                                             double acc) {
    for (int k0 = 0; k0 < n; k0 += 8) {
        double x[8], y[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k = k0 + u;
            if (k < n) {
                if constexpr (CGA) x[u] = __ldcg(a + (int64_t)k * sa);
                else x[u] = a[(int64_t)k * sa];
                if constexpr (CGB) y[u] = __ldcg(b + (int64_t)k * sb);
                else y[u] = b[(int64_t)k * sb];
            } else {
                x[u] = 0.0;
                y[u] = 0.0;
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (k0 + u < n) acc = fma(x[u], y[u], acc);
    }
    return acc;
}

__device__ __forceinline__ int pow2_at_least(int n) {
    int s = 1;
    while (s < n) s <<= 1;
    return s;
}

// Householder reflector of the column (alpha, x) with ||x||^2 = s > 0:
// beta = -sign(alpha) n with n = ||(alpha, x)||, tau = (beta - alpha)/beta =
// 1 + |alpha|/n and scale = 1/(alpha - beta) = sign(alpha)/(|alpha| + n).
// On this GPU an FP64 square root or division costs about ten dependent FP64
// instructions; both quotients come from reciprocal square roots instead
// (1/n = rsqrt(n^2), 1/q = rsqrt(q)^2).
__device__ __forceinline__ void reflector(double alpha, double s, double* beta, double* tau, double* scale) {
    const double w = fma(alpha, alpha, s);
    const double rn = rsqrt(w);
    const double n = w * rn;
    const double aa = fabs(alpha);
    const double rq = rsqrt(aa + n);
    *beta = alpha >= 0.0 ? -n : n;
    *tau = fma(aa, rn, 1.0);
    *scale = (alpha >= 0.0 ? rq : -rq) * rq;
}

// householder() for few rows (at most 32, used up to 16): lanes are rows within aligned segments of
// S = pow2_at_least(M) lanes, so one warp instruction serves 32/S columns of
// the trailing update; every warp forms the reflector itself (no broadcast
// through shared memory), and the column's scaled v is stored after the
// barrier that ends the column.
__device__ __forceinline__ void householder_small(double* A, double* tau, int M, int N) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = nwarps();
    const int k = M < N ? M : N;
    const int S = pow2_at_least(M), G = 32 / S;
    const int i = lane % S, sg = lane / S;
    for (int j = 0; j < k; ++j) {
        const double xi = i < M ? A[(int64_t)j * M + i] : 0.0;
        const double s = seg_sum((i > j && i < M) ? xi * xi : 0.0, S);
        const double alpha = A[(int64_t)j * M + j];
        double tj = 0.0, scale = 0.0, beta = alpha;
        if (s != 0.0) reflector(alpha, s, &beta, &tj, &scale);
        if (tj != 0.0) {
            const double vi = (i > j && i < M) ? xi * scale : (i == j ? 1.0 : 0.0);
            for (int c0 = j + 1 + warp * G; c0 < N; c0 += nw * G) {
                const int c = c0 + sg;
                const bool own = c < N && i < M && i >= j;
                const double aic = own ? A[(int64_t)c * M + i] : 0.0;
                const double w = seg_sum(own ? vi * aic : 0.0, S);
                if (own) A[(int64_t)c * M + i] = fma(-(tj * w), vi, aic);
            }
        }
        __syncthreads();
        if (warp == 0 && sg == 0) {
            if (tj != 0.0) {
                if (i > j && i < M) A[(int64_t)j * M + i] = xi * scale;
                if (i == j) A[(int64_t)j * M + j] = beta;
            }
            if (i == 0) tau[j] = tj;
        }
    }
    __syncthreads();
}

// form_q() for few rows (segment layout as in householder_small).
__device__ __forceinline__ void form_q_small(const double* A, const double* tau, double* Q, int M, int k) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = nwarps();
    const int S = pow2_at_least(M), G = 32 / S;
    const int i = lane % S, sg = lane / S;
    for (int64_t e = threadIdx.x; e < (int64_t)M * k; e += nthreads()) {
        const int r = (int)(e % M), c = (int)(e / M);
        Q[e] = r == c ? 1.0 : 0.0;
    }
    __syncthreads();
    for (int j = k - 1; j >= 0; --j) {
        const double tj = tau[j];
        if (tj == 0.0) continue;
        const double vi = (i > j && i < M) ? A[(int64_t)j * M + i] : (i == j ? 1.0 : 0.0);
        for (int c0 = j + warp * G; c0 < k; c0 += nw * G) {
            const int c = c0 + sg;
            const bool own = c < k && i < M && i >= j;
            const double qic = own ? Q[(int64_t)c * M + i] : 0.0;
            const double w = seg_sum(own ? vi * qic : 0.0, S);
            if (own) Q[(int64_t)c * M + i] = fma(-(tj * w), vi, qic);
        }
        __syncthreads();
    }
}

// Segments of 8 lanes: a warp works on four columns (or column pairs) at once,
// lane sl of a segment on the rows i = sl mod 8.  On this GPU an SMSP issues one
// FP64 warp instruction per 64 cycles however many lanes it serves, so what a
// routine costs is its FP64 warp instructions: a 32-lane dot product of n rows
// takes n/32 + 5 of them per column, four 8-lane ones n/8 + 3 together.
__device__ __forceinline__ double seg8_sum(double v) {
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}

// x 2^sh as a float (truncated; 0 below 2^-126, saturated above, NaN for a
// non-finite x), by integer operations: FP64 conversions would occupy the FP64 pipe.
__device__ __forceinline__ float to_float_scaled(double x, int sh) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int ex = (int)((hi >> 20) & 0x7ff), e = ex - 1023 + 127 + sh;
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const unsigned u = ex == 0x7ff ? 0x7fc00000u : e <= 0 ? 0u : (e >= 255 ? 0x7f7fffffu : ((unsigned)e << 23) | m);
    return __uint_as_float(u | (hi & 0x80000000u));
}
// A finite float as a double, by integer operations (FP32 subnormals become 0).
__device__ __forceinline__ double to_double(float f) {
    const unsigned u = __float_as_uint(f), e = (u >> 23) & 0xff;
    const unsigned hi = e ? ((e + 896u) << 20) | ((u & 0x7fffffu) >> 3) : 0u;
    return __hiloint2double((int)(hi | (u & 0x80000000u)), e ? (int)(u << 29) : 0);
}
// Sum over the warp by integer arithmetic: the 32 values as 58-bit fixed-point numbers
// of a common exponent, added in three limbs by warp reductions (redux), their exact
// sum rounded once.  275 cycles against 605 for five shuffle and FP64 addition
// steps (about 45 + 75 cycles each here), and no FP64 instruction.  Values outside
// the middle of the exponent range (and non-finite ones) take the shuffles.  A term is cut below 2^-57 of
// the largest one's leading bit, which 32 of them keep within 2^-52 of it: the rounding of the shuffles' additions.
__device__ __forceinline__ double warp_sum_fixed(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned e = (hi >> 20) & 0x7ff;
    const unsigned em = __reduce_max_sync(0xffffffffu, e);
    if (em < 64 || em > 2036) return warp_sum(v);
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32) | lo;
    const int d = (int)(em - (e ? e : 1u));
    const long long f = d < 58 ? (long long)((m << 5) >> d) : 0;
    const long long x = (int)hi < 0 ? -f : f;
    const unsigned r0 = __reduce_add_sync(0xffffffffu, (unsigned)x & 0xffffffu);
    const unsigned r1 = __reduce_add_sync(0xffffffffu, (unsigned)(x >> 24) & 0xffffffu);
    const int r2 = __reduce_add_sync(0xffffffffu, (int)(x >> 48));
    const long long t = (long long)r0 + ((long long)r1 << 24) + (long long)((unsigned long long)(long long)r2 << 48);
    if (t == 0) return 0.0;
    const unsigned long long a = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;   // below 2^63
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << lz;
    unsigned long long q = n >> 11;
    const unsigned r = (unsigned)n & 0x7ffu;
    q += (r > 0x400u || (r == 0x400u && (q & 1ull))) ? 1ull : 0ull;
    // a = 2^57 for a value of exponent field em
    const unsigned long long bits = ((unsigned long long)(em + 5 - lz) << 52) + q;
    return __longlong_as_double((long long)(bits | (t < 0 ? 1ull << 63 : 0ull)));
}

// x 2^-h by exponent arithmetic (0 when the result leaves the normal range downwards).
__device__ __forceinline__ double scale_down(double x, int h) {
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    return e == 0 || e - h < 1 ? 0.0 : __hiloint2double(hi - (int)((unsigned)h << 20), __double2loint(x));
}

// Householder vector of the column (alpha, x) with ||x||^2 = s != 0: H = I - tau v v^T
// with v = (vd, x 2^-shift), vd = sign(alpha) (|alpha| + n) 2^-shift, n = ||(alpha, x)||,
// tau = 2^(2 shift) / (n (n + |alpha|)); beta = -sign(alpha) n.  shift = 0 unless the
// norm is so large or small that tau would leave the range.  1/n by Halley's
// iteration from an FP32 reciprocal square root, 1/(n + |alpha|) by one step of
// order three from an FP32 reciprocal that is formed while the FP64 chain of 1/n
// runs (the errors of both are of order 2^-63): about 900 cycles against 1500 for
// the two in turn.
__device__ __forceinline__ void reflector_vector(double alpha, double s, double* tau, double* vd, double* beta,
                                                 int* shift) {
    const double w = fma(alpha, alpha, s);
    const int e = (__double2hiint(w) >> 20) & 0x7ff;
    *shift = 0;
    if (__double2hiint(w) < 0 || e < 64 || e > 1980) {   // tiny, huge, subnormal or non-finite
        const double rn = rsqrt(w), n = w * rn;
        int h = 0;
        if (n > 0.0 && n < 1.7976931348623157e308) frexp(n, &h);
        const double nu = ldexp(n, -h), qu = nu + ldexp(fabs(alpha), -h);
        *shift = h;
        *tau = 1.0 / (nu * qu);
        *vd = alpha >= 0.0 ? qu : -qu;
        *beta = alpha >= 0.0 ? -n : n;
        return;
    }
    const int h = (e - 1023) >> 1;   // w = 4^h u, u in [1, 4)
    const double u = __hiloint2double(__double2hiint(w) - (h << 21), __double2loint(w));
    const double au = scale_down(fabs(alpha), h);
    const float uf = to_float_scaled(u, 0);
    float yf, zf;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(uf));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(zf) : "f"(fmaf(uf, yf, to_float_scaled(au, 0))));
    const double y0 = to_double(yf), z0 = to_double(zf);
    const double r = fma(-(u * y0), y0, 1.0);
    const double y = fma(y0 * r, fma(0.375, r, 0.5), y0);   // 1/sqrt(u)
    const double nu = u * y, qu = nu + au;
    const double p = fma(-qu, z0, 1.0);
    const double z = fma(z0, fma(p, p, p), z0);             // 1/qu
    const double t = y * z;                                 // in (0.1, 1]: times 4^-h
    *tau = __hiloint2double(__double2hiint(t) - (h << 21), __double2loint(t));
    const double q = __hiloint2double(__double2hiint(qu) + (h << 20), __double2loint(qu));
    const double n = __hiloint2double(__double2hiint(nu) + (h << 20), __double2loint(nu));
    *vd = alpha >= 0.0 ? q : -q;
    *beta = alpha >= 0.0 ? -n : n;
}

// One warp: H_{j-1} (v the column j - 1 and vj, tw_scale = tau_{j-1}; none when tau = 0)
// applied to column j, then the reflector of column j (rows j .. M-1, v below row j left
// in place): tau[j], vd[j] = v_j, R(j, j) in the diagonal entry (tau[j] = 0: nothing to
// eliminate).
__device__ __forceinline__ void reflect_column(double* A, double* tau, double* vd, int M, int j, double tj, double vj,
                                               int lane) {
    double* x = A + (int64_t)j * M;
    const double* v = x - M;
    double tw = 0.0;
    if (tj != 0.0) {
        double d = lane == 0 ? vj * x[j - 1] : 0.0;
        for (int i = j + lane; i < M; i += 32) d = fma(v[i], x[i], d);
        tw = tj * warp_sum_fixed(d);
    }
    double s = 0.0, alpha = 0.0;
    for (int i = j + lane; i < M; i += 32) {
        double y = x[i];
        if (tj != 0.0) {
            y = fma(-tw, v[i], y);
            x[i] = y;
        }
        if (i == j) alpha = y;
        else s = fma(y, y, s);
    }
    if (tj != 0.0 && lane == 0) x[j - 1] = fma(-tw, vj, x[j - 1]);
    s = warp_sum_fixed(s);
    alpha = __shfl_sync(0xffffffffu, alpha, 0);
    double t = 0.0, d = 0.0, beta = 0.0;
    if (s != 0.0) {
        int shift;
        reflector_vector(alpha, s, &t, &d, &beta, &shift);
        if (shift)
            for (int i = j + lane; i < M; i += 32)   // the rows this lane wrote
                if (i != j) x[i] = ldexp(x[i], -shift);
    }
    if (lane == 0) {
        if (s != 0.0) x[j] = beta;
        vd[j] = d;
        tau[j] = t;
    }
    __syncwarp();
}

// The columns c0 + 4 w + segment, stepping 4 nw, of A: a_c -= tau_j (v_j^T a_c) v_j.
__device__ __forceinline__ void reflect_segments(double* A, double tj, double vj, int M, int N, int j, int c0, int w,
                                                 int nw, int lane) {
    const int sl = lane & 7;
    const double* v = A + (int64_t)j * M;
    for (int cb = c0 + 4 * w; cb < N; cb += 4 * nw) {
        const int c = cb + (lane >> 3);
        const bool on = c < N;   // (a segment without a column reads none: another one may be writing it)
        double* a = A + (int64_t)(on ? c : cb) * M;
        const double a_j = on ? a[j] : 0.0;
        double d = sl == 0 ? vj * a_j : 0.0;
        if (on)
            for (int i = j + 1 + sl; i < M; i += 8) d = fma(v[i], a[i], d);
        const double tw = tj * seg8_sum(d);
        if (on) {
            if (sl == 0) a[j] = fma(-tw, vj, a_j);
            for (int i = j + 1 + sl; i < M; i += 8) a[i] = fma(-tw, v[i], a[i]);
        }
    }
}

// Householder factorisation of A (M x N, column-major, ld M) in place: R in the
// upper trapezoid, the reflectors' vectors below the diagonal and in vd (their
// diagonal entries), tau[j]; form_q() reads them.
//
// One barrier per column: while the other warps apply H_j to the columns beyond
// j + 1, warp 0 applies it to column j + 1 and forms H_{j+1} at once (its chain,
// about 2300 cycles, is what bounds a small QR).  Warps that
// share warp 0's scheduler (4, 8, ...) stay out of the updates while these are
// shorter than that chain, which they would lengthen.
__device__ __forceinline__ void householder(double* A, double* tau, double* vd, int M, int N) {
    if (M <= 16) {
        householder_small(A, tau, M, N);
        return;
    }
    const int k = M < N ? M : N;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = nwarps();
    const int w_all = nw == 1 ? 0 : warp - 1, n_all = nw == 1 ? 1 : nw - 1;
    const int w_off = (warp & 3) ? (warp >> 2) * 3 + (warp & 3) - 1 : -1;
    const int n_off = (nw >> 2) * 3 + ((nw & 3) ? (nw & 3) - 1 : 0);
    if (warp == 0) reflect_column(A, tau, vd, M, 0, 0.0, 0.0, lane);
    __syncthreads();
    for (int j = 0; j < k; ++j) {
        const double tj = tau[j], vj = vd[j];
        if (warp == 0 && j + 1 < k) reflect_column(A, tau, vd, M, j + 1, tj, vj, lane);
        // FP64 instructions of the other columns' updates against the chain's
        const bool off = nw >= 6 && (N - j) * ((M - j) / 4 + 4) <= 4 * 75;
        const int w = off ? w_off : w_all;
        if (w >= 0 && tj != 0.0) reflect_segments(A, tj, vj, M, N, j, j + 1 < k ? j + 2 : j + 1, w, off ? n_off : n_all, lane);
        __syncthreads();
    }
}

// Q (M x k, column-major) = H_0 ... H_{k-1} applied to the first k columns of I.
// Column c needs H_c ... H_0 only and no other column of Q: every 8-lane segment
// takes a column through all its reflectors without a barrier (each lane keeps
// to the rows i = sl mod 8), longest columns first.
__device__ __forceinline__ void form_q(const double* A, const double* tau, const double* vd, double* Q, int M, int k) {
    if (M <= 16) {
        form_q_small(A, tau, Q, M, k);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sl = lane & 7;
    for (int cb = 4 * warp; cb < k; cb += 4 * nwarps()) {
        const int c = k - 1 - (cb + (lane >> 3));
        const bool own = c >= 0;
        double* q = Q + (int64_t)(own ? c : 0) * M;
        if (own)
            for (int i = sl; i < M; i += 8) q[i] = i == c ? 1.0 : 0.0;
        for (int j = k - 1 - cb; j >= 0; --j) {
            const double tj = tau[j];
            if (tj == 0.0) continue;
            const double vj = vd[j];
            const double* v = A + (int64_t)j * M;
            const int i0 = j + ((sl - j) & 7);
            double d = 0.0;
            if (own && c >= j)
                for (int i = i0; i < M; i += 8) d = fma(i == j ? vj : v[i], q[i], d);
            const double tw = tj * seg8_sum(d);
            if (own && c >= j)
                for (int i = i0; i < M; i += 8) q[i] = fma(-tw, i == j ? vj : v[i], q[i]);
        }
    }
    __syncthreads();
}

// householder() and form_q() for a matrix in global memory (one that neither a CTA's nor a cluster's
// shared memory holds): every column is read by a whole warp (256 contiguous bytes a load) and the
// reflector's column by the whole CTA, since the loads from L2 bound it; the 8-lane segments and the one-warp
// chain of householder() lose there (truncation at rank 2000 over one charge 2.05 -> 1.64 s, zip-up of a
// chain of 16 at rank 100 184 -> 150 ms).
// v_j = 1 is implicit, v below the diagonal scaled to it.  red: 33 shared doubles.
__device__ __forceinline__ void householder_global(double* A, double* tau, int M, int N, double* red) {
    const int k = M < N ? M : N;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int j = 0; j < k; ++j) {
        double* x = A + (int64_t)j * M;
        double s = 0.0;
        for (int i = j + 1 + threadIdx.x; i < M; i += nthreads()) s = fma(x[i], x[i], s);
        s = block_sum(s, red);
        const double alpha = x[j];
        double tj = 0.0, scale = 0.0, beta = alpha;
        if (s != 0.0) {
            beta = alpha >= 0.0 ? -sqrt(fma(alpha, alpha, s)) : sqrt(fma(alpha, alpha, s));
            tj = (beta - alpha) / beta;
            scale = 1.0 / (alpha - beta);
        }
        __syncthreads();   // every thread has read alpha
        if (threadIdx.x == 0) {
            x[j] = beta;
            tau[j] = tj;
        }
        if (tj != 0.0) {
            for (int i = j + 1 + threadIdx.x; i < M; i += nthreads()) x[i] *= scale;
            __syncthreads();
            for (int c = j + 1 + warp; c < N; c += nwarps()) {
                double* a = A + (int64_t)c * M;
                const double a_j = a[j];
                double w = 0.0;
                for (int i = j + 1 + lane; i < M; i += 32) w = fma(x[i], a[i], w);
                const double tw = tj * (warp_sum(w) + a_j);
                if (lane == 0) a[j] = a_j - tw;
                for (int i = j + 1 + lane; i < M; i += 32) a[i] = fma(-tw, x[i], a[i]);
            }
        }
        __syncthreads();
    }
}
__device__ __forceinline__ void form_q_global(const double* A, const double* tau, double* Q, int M, int k) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // column c needs H_c ... H_0 only: one warp takes it through all of them, longest columns first
    for (int cb = warp; cb < k; cb += nwarps()) {
        const int c = k - 1 - cb;
        double* q = Q + (int64_t)c * M;
        for (int i = lane; i < M; i += 32) q[i] = i == c ? 1.0 : 0.0;
        for (int j = c; j >= 0; --j) {
            const double tj = tau[j];
            if (tj == 0.0) continue;
            const double* v = A + (int64_t)j * M;
            const int i0 = j + ((lane - j) & 31);   // every lane keeps to the rows i = lane mod 32
            double w = 0.0;
            for (int i = i0; i < M; i += 32) w = fma(i == j ? 1.0 : v[i], q[i], w);
            const double tw = tj * warp_sum(w);
            for (int i = i0; i < M; i += 32) q[i] = fma(-tw, i == j ? 1.0 : v[i], q[i]);
        }
    }
    __syncthreads();
}

// X (M x k, column-major) <- H_0 ... H_{k-1} X with householder()'s reflectors (M > 16),
// whose diagonal entries stand in A: every 8-lane segment takes a column through
// all of them without a barrier, as in form_q().  Q V this way takes 2 k (M k - k^2 / 2)
// FMAs; forming Q and multiplying takes 2 k (M k - k^2 / 2) - k^3 / 3 and M k^2 more.
__device__ __forceinline__ void apply_q(const double* A, const double* tau, double* X, int M, int k) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sl = lane & 7;
    for (int cb = 4 * warp; cb < k; cb += 4 * nwarps()) {
        const bool own = cb + (lane >> 3) < k;
        double* x = X + (int64_t)(own ? cb + (lane >> 3) : cb) * M;
        for (int j = k - 1; j >= 0; --j) {
            const double tj = tau[j];
            if (tj == 0.0) continue;
            const double* v = A + (int64_t)j * M;
            const int i0 = j + ((sl - j) & 7);
            double d = 0.0;
            if (own)
                for (int i = i0; i < M; i += 8) d = fma(v[i], x[i], d);
            const double tw = tj * seg8_sum(d);
            if (own)
                for (int i = i0; i < M; i += 8) x[i] = fma(-tw, v[i], x[i]);
        }
    }
    __syncthreads();
}

__device__ __forceinline__ int rr_player(int pos, int round, int n2) {
    if (pos == 0) return 0;
    int v = pos - 1 + round;   // < 2 (n2 - 1) for round < n2 - 1
    if (v >= n2 - 1) v -= n2 - 1;
    return v + 1;
}

// Order of non-negative doubles through their bit patterns (integer compares
// instead of FP64 ones).
__device__ __forceinline__ long long nonneg_key(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ long long abs_key(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }

// sqrt(x) for x >= 0 from one reciprocal square root (about 2/3 of the cost of
// an FP64 square root here); 1 ulp-level accuracy.
__device__ __forceinline__ double sqrt_via_rsqrt(double x) { return x > 0.0 ? x * rsqrt(x) : 0.0; }

// Rotation (c, s) that makes the columns with squared norms a, b and inner
// product g orthogonal: with d = b - a, t = sign(zeta) 2|g| / (|d| + sqrt(d^2
// + 4 g^2)) equals sign(zeta) / (|zeta| + sqrt(1 + zeta^2)) for zeta = d/(2g)
// (sign(zeta) = +1 at d = 0), c = 1/sqrt(1 + t^2), s = c t.
__device__ __forceinline__ void jacobi_rotation(double a, double b, double g, double* c, double* s) {
    const double d = b - a;
    const double r = sqrt(fma(d, d, 4.0 * g * g));
    const double sz = (d == 0.0 || (d > 0.0) == (g > 0.0)) ? 1.0 : -1.0;
    const double t = sz * (2.0 * fabs(g)) / (fabs(d) + r);
    *c = rsqrt(fma(t, t, 1.0));
    *s = *c * t;
}

// jacobi_rotation() with the angle taken in FP32: d = b - a and 2g are
// brought into FP32 range (scaled by a power of two when needed), t is formed
// in FP32, and c = rsqrt(1 + t^2), s = c t in FP64, so that c^2 + s^2 = 1
// within FP64 rounding.  The rotation is orthogonal in FP64 and only its angle
// carries the FP32 error, which leaves |g'| ~ 1e-7 |g| for the next sweep.
__device__ __forceinline__ void jacobi_rotation_fast(double a, double b, double g, double* c, double* s) {
    const double d = b - a, g2 = g + g;
    const int ed = (__double2hiint(d) >> 20) & 0x7ff, eg = (__double2hiint(g2) >> 20) & 0x7ff;
    const int e = ed > eg ? ed : eg;
    if (e < 2 || e > 2045) {   // zero, subnormal or non-finite scale: exact formula
        jacobi_rotation(a, b, g, c, s);
        return;
    }
    float df, gf;
    if (e >= 1023 - 60 && e <= 1023 + 60) {   // squares stay normal in FP32
        df = __double2float_rn(d);
        gf = __double2float_rn(g2);
    } else {
        const double sc = __hiloint2double((2046 - e) << 20, 0);   // 2^(1023 - e)
        df = __double2float_rn(d * sc);
        gf = __double2float_rn(g2 * sc);
    }
    // the angle only needs FP32 accuracy: hardware reciprocal square root and
    // fast division (the larger of |df|, |gf| is at least 2^-60, so both are in range)
    const float w = fmaf(df, df, gf * gf);
    const float r = w * rsqrtf(w);
    const float sz = (df == 0.0f || ((df > 0.0f) == (gf > 0.0f))) ? 1.0f : -1.0f;
    const double t = (double)(sz * __fdividef(fabsf(gf), fabsf(df) + r));
    const double cd = rsqrt(fma(t, t, 1.0));
    *c = cd;
    *s = cd * t;
}

// jacobi() for k <= 16: one round-robin pair per warp; the pair's three inner
// products are formed in aligned lane segments of S = pow2_at_least(k) lanes
// (S <= 8: a, b, g in three segments of one register; S = 16: a | b in one
// register, g in another), and the rotation of the G and V columns runs with
// lanes [0, S) on G and [S, 2S) on V.
__device__ __forceinline__ void jacobi_small(double* G, double* V, double* Sraw, int k, double* red, int* s_rot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double f = 0.0;
    for (int64_t e = threadIdx.x; e < (int64_t)k * k; e += nthreads()) {
        const double v = G[e];
        f += v * v;
        V[e] = (e % k) == (e / k) ? 1.0 : 0.0;
    }
    f = block_sum(f, red);
    const double tol = (double)k * DBL_EPSILON;
    const double tol2 = tol * tol, tiny2 = tol2 * f;
    const int n2 = k + (k & 1);
    const int S = pow2_at_least(k);
    const int i = lane % S, sg = lane / S;
    for (int sweep = 0; sweep < kMaxSweeps && k > 1; ++sweep) {
        if (threadIdx.x == 0) *s_rot = 0;
        __syncthreads();
        for (int round = 0; round < n2 - 1; ++round) {
            for (int pi = warp; pi < n2 / 2; pi += nwarps()) {
                int p = rr_player(pi, round, n2), q = rr_player(n2 - 1 - pi, round, n2);
                if (p >= k || q >= k) continue;
                if (p > q) {
                    const int tmp = p;
                    p = q;
                    q = tmp;
                }
                const double xp = i < k ? G[(int64_t)p * k + i] : 0.0;
                const double xq = i < k ? G[(int64_t)q * k + i] : 0.0;
                double a, b, g;
                if (S <= 8) {
                    // segment 0: xp xp, 1: xq xq, 2: xp xq (segment 3 idle)
                    const double u = sg == 1 ? xq : xp, w = sg == 0 ? xp : xq;
                    const double prod = seg_sum(sg < 3 ? u * w : 0.0, S);
                    a = __shfl_sync(0xffffffffu, prod, 0);
                    b = __shfl_sync(0xffffffffu, prod, S);
                    g = __shfl_sync(0xffffffffu, prod, 2 * S);
                } else {
                    const double u = sg == 0 ? xp : xq;
                    const double ab = seg_sum(u * u, 16);
                    const double pg = seg_sum(xp * xq, 16);
                    a = __shfl_sync(0xffffffffu, ab, 0);
                    b = __shfl_sync(0xffffffffu, ab, 16);
                    g = __shfl_sync(0xffffffffu, pg, 0);
                }
                if (g * g > tol2 * (a * b) && nonneg_key(a) > nonneg_key(tiny2) &&
                    nonneg_key(b) > nonneg_key(tiny2)) {
                    double c, s;
                    jacobi_rotation_fast(a, b, g, &c, &s);
                    if (lane < 2 * S && i < k) {
                        double* X = lane < S ? G : V;
                        const double vp = X[(int64_t)p * k + i], vq = X[(int64_t)q * k + i];
                        X[(int64_t)p * k + i] = c * vp - s * vq;
                        X[(int64_t)q * k + i] = s * vp + c * vq;
                    }
                    if (lane == 0) *s_rot = 1;
                }
            }
            __syncthreads();
        }
        const int rot = *s_rot;
        __syncthreads();
        if (!rot) break;
    }
    // column norms: 32/S columns per warp instruction
    const int Gc = 32 / S;
    for (int j0 = warp * Gc; j0 < k; j0 += nwarps() * Gc) {
        const int j = j0 + sg;
        const double x = (j < k && i < k) ? G[(int64_t)j * k + i] : 0.0;
        const double a = seg_sum(x * x, S);
        if (j < k && i == 0) Sraw[j] = sqrt_via_rsqrt(a);
    }
    __syncthreads();
}

// FP64 one-sided Jacobi of B (rows x k, column-major, rows <= 32) with the rotations accumulated in V:
// one pair per warp, its inner products in aligned segments of S = pow2_at_least(rows)
// lanes.  For the smallest sectors, where a handful of rotations is all there is to do and the stages
// of jacobi_pre() (an FP32 iteration, the orthogonalisation of its rotations, a Gram test) cost more than
// they save.  Angles in FP64: two columns are done after one rotation (with FP32 angles after two, 0 to
// 3 % slower).  Threshold |g| > rows eps sqrt(a b), columns below the numerical-zero level
// (rows eps)^2 ||B||_F^2 are left alone.  Sraw: column norms of the result.
__device__ __forceinline__ void jacobi_tiny(double* B, double* V, double* Sraw, int rows, int k, int ldb, int ldv,
                                            double* red, int* s_rot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double f = 0.0;
    for (int e = threadIdx.x; e < k * ldb; e += nthreads()) f = fma(B[e], B[e], f);   // (padding zero)
    for (int e = threadIdx.x; e < k * ldv; e += nthreads()) V[e] = e % ldv == e / ldv ? 1.0 : 0.0;
    f = block_sum(f, red);
    // exact scaling to ||B||_F in [1, 2): squares and products of the norms stay in range
    const int fe = (__double2hiint(f) >> 20) & 0x7ff, h = fe == 0 || fe == 0x7ff ? 0 : (fe - 1023) >> 1;
    const double sc = __hiloint2double((1023 - h) << 20, 0), up = __hiloint2double((1023 + h) << 20, 0);
    for (int e = threadIdx.x; e < k * ldb; e += nthreads()) B[e] *= sc;
    const double tol = (double)rows * DBL_EPSILON;
    const double tol2 = tol * tol, tiny2 = tol2 * (f * sc * sc);
    const int n2 = k + (k & 1);
    const int S = pow2_at_least(rows);
    const int i = lane % S, sg = lane / S;
    for (int sweep = 0; sweep < kMaxSweeps && k > 1; ++sweep) {
        if (threadIdx.x == 0) *s_rot = 0;
        __syncthreads();
        for (int round = 0; round < n2 - 1; ++round) {
            for (int pi = warp; pi < n2 / 2; pi += nwarps()) {
                const int u = rr_player(pi, round, n2), v = rr_player(n2 - 1 - pi, round, n2);
                if (u >= k || v >= k) continue;
                double* Bp = B + min(u, v) * ldb;
                double* Bq = B + max(u, v) * ldb;
                const double xp = i < rows ? Bp[i] : 0.0, xq = i < rows ? Bq[i] : 0.0;
                double a, b, g;
                if (S <= 8) {   // segment 0: xp xp, 1: xq xq, 2: xp xq
                    const double prod =
                        seg_sum(sg < 3 ? (sg == 1 ? xq : xp) * (sg == 0 ? xp : xq) : 0.0, S);
                    a = __shfl_sync(0xffffffffu, prod, 0);
                    b = __shfl_sync(0xffffffffu, prod, S);
                    g = __shfl_sync(0xffffffffu, prod, 2 * S);
                } else if (S == 16) {
                    const double x = sg == 0 ? xp : xq;
                    const double ab = seg_sum(x * x, 16);
                    g = seg_sum(xp * xq, 16);
                    a = __shfl_sync(0xffffffffu, ab, 0);
                    b = __shfl_sync(0xffffffffu, ab, 16);
                } else {
                    a = warp_sum(xp * xp);
                    b = warp_sum(xq * xq);
                    g = warp_sum(xp * xq);
                }
                if (g * g > tol2 * (a * b) && nonneg_key(a) > nonneg_key(tiny2) && nonneg_key(b) > nonneg_key(tiny2)) {
                    double c, s;
                    jacobi_rotation(a, b, g, &c, &s);
                    double* Vp = V + min(u, v) * ldv;
                    double* Vq = V + max(u, v) * ldv;
                    if (lane < S && i < rows) {
                        Bp[i] = c * xp - s * xq;
                        Bq[i] = s * xp + c * xq;
                    }
                    // V on the second segment, or after B where the rows take the warp
                    if ((S <= 16 ? sg == 1 : true) && i < k) {
                        const double vp = Vp[i], vq = Vq[i];
                        Vp[i] = c * vp - s * vq;
                        Vq[i] = s * vp + c * vq;
                    }
                    if (lane == 0) *s_rot = 1;
                }
            }
            __syncthreads();
        }
        const int rot = *s_rot;
        __syncthreads();
        if (!rot) break;
    }
    const int Gc = 32 / S;   // columns per warp instruction
    for (int j0 = warp * Gc; j0 < k; j0 += nwarps() * Gc) {
        const int j = j0 + sg;
        const double x = (j < k && i < rows) ? B[j * ldb + i] : 0.0;
        const double a = seg_sum(x * x, S);
        if (j < k && i < rows) B[j * ldb + i] = x * up;
        if (j < k && i == 0) Sraw[j] = sqrt_via_rsqrt(a) * up;
    }
    __syncthreads();
}

// SVD factors from a Jacobi on B itself (B V = U diag(Sraw), B = M for a tall M, B =
// M^T for a wide M): tall: US = columns of B, Vt = rows V^T; wide: US = V
// diag(S), Vt = (B diag(1/S))^T.  Order, tie rule and sign rule as in
// svd_assemble.  rinv: k scratch doubles, perm: k ints.
__device__ __forceinline__ void svd_assemble_direct(const double* B, int ldb, const double* V, int ldv,
                                                    const double* Sraw, double* rinv, int* perm, double* S,
                                                    double* US, double* Vt, int M, int N, int k, int wide, int ldus,
                                                    int ldvt) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < k; i += nthreads()) {
        const double si = Sraw[i];
        const long long ki = nonneg_key(si);
        int rank = 0;
        for (int j = 0; j < k; ++j) {
            const long long kj = nonneg_key(Sraw[j]);
            rank += (kj > ki || (kj == ki && j < i)) ? 1 : 0;
        }
        perm[rank] = i;
        if (wide) {
            const double r = rsqrt(si);
            rinv[i] = si > 0.0 ? r * r : 0.0;
        }
    }
    __syncthreads();
    for (int64_t e = threadIdx.x; e < (int64_t)M * k; e += nthreads()) {
        const int i = (int)(e / k), r = (int)(e % k);
        const int p = perm[r];
        US[(int64_t)i * ldus + r] = wide ? V[(int64_t)p * ldv + i] * Sraw[p] : B[(int64_t)p * ldb + i];
    }
    for (int64_t e = threadIdx.x; e < (int64_t)k * N; e += nthreads()) {
        const int r = (int)(e / N), c = (int)(e % N);
        const int p = perm[r];
        Vt[(int64_t)r * ldvt + c] = wide ? B[(int64_t)p * ldb + c] * rinv[p] : V[(int64_t)p * ldv + c];
    }
    for (int r = threadIdx.x; r < k; r += nthreads()) S[r] = Sraw[perm[r]];
    __syncthreads();
    for (int r = warp; r < k; r += nwarps()) {
        long long best = -1;
        int bi = 0;
        for (int c = lane; c < N; c += 32) {
            const long long a = abs_key(Vt[(int64_t)r * ldvt + c]);
            if (a > best) {
                best = a;
                bi = c;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ob > best || (ob == best && oi < bi)) {
                best = ob;
                bi = oi;
            }
        }
        if (Vt[(int64_t)r * ldvt + bi] < 0.0) {
            for (int c = lane; c < N; c += 32) Vt[(int64_t)r * ldvt + c] = -Vt[(int64_t)r * ldvt + c];
            for (int i = lane; i < M; i += 32) US[(int64_t)i * ldus + r] = -US[(int64_t)i * ldus + r];
        }
    }
}

__device__ __forceinline__ float seg8_sum(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}
// Leading dimension of columns of n <= 64 rows in jacobi_pre(): they are
// padded with zero rows to an odd multiple of 8, so that the 8-lane segments of a
// warp, which work on neighbouring columns, meet distinct banks (64-byte pieces of
// columns 64 bytes apart modulo 128), and whole segments of rows need no bounds check.
__host__ __device__ constexpr int jacobi_ld(int n) {
    return n <= 8 ? 8 : n <= 24 ? 24 : n <= 40 ? 40 : n <= 56 ? 56 : 72;
}

__device__ __forceinline__ float rsqrt_fast(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// tan of the angle that makes columns of squared norms a, b (d = b - a) and
// inner product g (g2 = 2 g) orthogonal; d and g2 scaled so that the larger is near 1.
__device__ __forceinline__ float jacobi_tan(float d, float g2) {
    const float w = fmaf(d, d, g2 * g2);
    const float r = w * rsqrt_fast(w);
    const float t = __fdividef(fabsf(g2), fabsf(d) + r);
    return __uint_as_float(__float_as_uint(t) | ((__float_as_uint(d) ^ __float_as_uint(g2)) & 0x80000000u));
}

// jacobi_tan() of FP64 norms and inner product, d = b - a and 2 g scaled by the larger exponent.
__device__ __forceinline__ float jacobi_angle(double d, double g) {
    const int ed = (__double2hiint(d) >> 20) & 0x7ff, eg = ((__double2hiint(g) >> 20) & 0x7ff) + 1;
    const int sh = 1023 - max(ed, eg);
    return jacobi_tan(to_float_scaled(d, sh), to_float_scaled(g, sh + 1));
}

// Round-robin over k columns, one pair per 8-lane segment u: the pair of a round
// follows from the one before (position 0 stands still, the others move on by one).
// get(): false, and columns that other segments may be writing, for a segment without a pair.
struct SegPair {
    int a, b, n2, k;
    bool fixed;
    __device__ __forceinline__ SegPair(int u, int k_) : n2(k_ + (k_ & 1)), k(k_) {
        fixed = u == 0;
        a = u;
        b = u < n2 / 2 ? n2 - 1 - u : n2;   // out of range: never valid
    }
    __device__ __forceinline__ bool get(int* p, int* q) const {
        const bool on = b < n2 && a < k && b < k;
        *p = on ? min(a, b) : 0;
        *q = on ? max(a, b) : 0;
        return on;
    }
    __device__ __forceinline__ void next() {
        if (!fixed) a = a == n2 - 1 ? 1 : a + 1;
        if (b < n2) b = b == n2 - 1 ? 1 : b + 1;
    }
};

// Barrier 1 among the first n threads of the CTA (a multiple of 32).
__device__ __forceinline__ void bar_first(int n) { asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); }

// FP32 one-sided Jacobi of G (k columns of 8 RG rows, ||G||_F ~ 1, overwritten), the
// rotations accumulated in V (k columns of 8 RV rows, identity on entry): one pair per 8-lane segment.
// Bound by the latency of a round (loads, three shuffles, two reciprocal square
// roots, stores, a barrier of the working warps).  Tolerance 4 sqrt(k) eps_32; a
// sweep rotating at most 1/32 of the pairs ends.  Needs 4 warps per 32 columns.
template <int RG, int RV>
__device__ __forceinline__ void jacobi_f32_segments(float* G, float* V, int k, int ldg, int ldv, int* s_cnt) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sl = lane & 7;
    const int n2 = k + (k & 1);
    const int nact = (n2 / 2 + 3) / 4;
    const float tol = 4.0f * sqrtf((float)k) * FLT_EPSILON;
    for (int sweep = 0; sweep < 20; ++sweep) {
        if (threadIdx.x == 0) *s_cnt = 0;
        int cnt = 0;
        if (warp < nact) {
            SegPair pr(4 * warp + (lane >> 3), k);
            for (int round = 0; round < n2 - 1; ++round, pr.next()) {
                int p, q;
                const bool on = pr.get(&p, &q);
                float* Gp = G + p * ldg;
                float* Gq = G + q * ldg;
                float* Vp = V + p * ldv;
                float* Vq = V + q * ldv;
                float xp[RG], xq[RG], vp[RV], vq[RV];
                float a = 0.0f, b = 0.0f, g = 0.0f;
#pragma unroll
                for (int r = 0; r < RG; ++r) {
                    const int i = sl + 8 * r;
                    xp[r] = on ? Gp[i] : 0.0f;
                    xq[r] = on ? Gq[i] : 0.0f;
                    a = fmaf(xp[r], xp[r], a);
                    b = fmaf(xq[r], xq[r], b);
                    g = fmaf(xp[r], xq[r], g);
                }
#pragma unroll
                for (int r = 0; r < RV; ++r) {
                    const int i = sl + 8 * r;
                    vp[r] = on ? Vp[i] : 0.0f;
                    vq[r] = on ? Vq[i] : 0.0f;
                }
                a = seg8_sum(a);
                b = seg8_sum(b);
                g = seg8_sum(g);
                // cos and sin of the rotation from cos(2 theta) = |d| / sqrt(d^2 + 4 g^2)
                const float d = b - a, g2 = g + g;
                const unsigned mb = max(__float_as_uint(fabsf(d)), __float_as_uint(fabsf(g2))) >> 23;
                const float sc = __uint_as_float((254u - min(mb, 253u)) << 23);
                const float dn = d * sc, gn = g2 * sc;
                const float ri = rsqrt_fast(fmaf(dn, dn, gn * gn));
                const float c2 = fmaf(0.5f, fabsf(dn) * ri, 0.5f);
                const float rc = rsqrt_fast(c2);
                // one Newton step on c^2 + s^2 = 1: the approximate reciprocal roots are off by up
                // to 2^-22, which hundreds of rotations would add up in the columns' lengths
                const float cr = c2 * rc, hr = 0.5f * gn * ri * rc;
                const float fix = fmaf(-0.5f, fmaf(cr, cr, hr * hr), 1.5f);
                const float c = cr * fix, h = hr * fix;
                const float sn = __uint_as_float(__float_as_uint(h) ^ (__float_as_uint(d) & 0x80000000u));
                const bool rot = on && fminf(a, b) > 1e-30f && fabsf(g) > tol * (a * rsqrt_fast(a)) * (b * rsqrt_fast(b));
                if (rot) {
#pragma unroll
                    for (int r = 0; r < RG; ++r) {
                        const int i = sl + 8 * r;
                        Gp[i] = c * xp[r] - sn * xq[r];
                        Gq[i] = sn * xp[r] + c * xq[r];
                    }
#pragma unroll
                    for (int r = 0; r < RV; ++r) {
                        const int i = sl + 8 * r;
                        Vp[i] = c * vp[r] - sn * vq[r];
                        Vq[i] = sn * vp[r] + c * vq[r];
                    }
                    cnt += sl == 0;
                }
                bar_first(32 * nact);
            }
        }
        __syncthreads();
        if (cnt) atomicAdd(s_cnt, cnt);
        __syncthreads();
        const int total = *s_cnt;
        __syncthreads();
        if (64 * total <= k * (k - 1)) break;
    }
}

// Rotation of one pair as the G warps hand it to the V warps.
struct SegRot {
    double fp, sq, sp, fq;   // x_p' = fp x_p - sq x_q, x_q' = sp x_p + fq x_q
    int p, q;
    int mode;                // 0: none, 1: fp = fq = 1, 2: full
    int pad;
};

// FP64 one-sided Jacobi of G (rows x k, column-major, ||G||_F in [1/2, 1)) rotating
// the columns of V along: one pair per 8-lane segment, the columns' squared norms
// tracked in nrm (recomputed every sweep), the tests and angles in FP32 (only the
// inner product, the norms and the rotation itself need FP64).  A rotation by a
// small angle is applied as x_p - alpha x_q, x_q + beta x_p (two FMAs per row
// instead of four operations): that is the rotation times 1 / cos, and the cosines
// are gathered per column in del (column = (1 + del) x stored; alpha and beta
// carry the ratio of the two scales, terms below 2^-57 dropped).  Larger angles
// (and columns with |del| >= 2^-30) take the full rotation, which clears del.
// Pairs rotate while |g| > rows eps sqrt(a b), min(a, b) > (rows eps)^2 ||G||_F^2.
// Between sweeps all warps form the inner products of all pairs.  Where none is over the
// limit the iteration ends; where all cosines |g| / sqrt(a b) and tangents over it are below
// m = 2^-28, it ends with one step of first order, G += G X and V += V X with the tangents in
// the antisymmetric X: what is left of a cosine are terms of second order, X_rp g_rq and X_rp
// X_rq |g_r|^2, at most m^2 sqrt(a b) each and 5 k together, 0.3 k eps, under the
// limit.  X is below 2^-28 times a ratio of norms, so the two products take FP32.  That step
// costs a third of the sweep it replaces (k = 60: 65 us for 198).
// The first nact warps work on G; the next nact rotate V one round behind them,
// which fills the FP64 pipe while the G warps wait for loads, shuffles and
// angles.  ring: 2 x 32 rotations.  Needs 2 nact warps.
template <int RG, int RV>
__device__ __forceinline__ void jacobi_f64_segments(double* G, double* V, double* nrm, float* del, int k, int rows, int ldg,
                                                    int ldv, double fro, double* scr, SegRot* ring, int* s_rot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sl = lane & 7;
    const int n2 = k + (k & 1);
    const int nact = (n2 / 2 + 3) / 4;
    const float tol = (float)rows * 2.220446e-16f * 0x1p48f;   // compared with g 2^48
    const float tiny = (float)rows * 2.220446e-16f * (float)rows * 2.220446e-16f * to_float_scaled(fro, 0);
    float* Gf = (float*)scr;
    float* Vf = Gf + k * ldg;
    float* Xf = Vf + k * ldv;
    for (int j = threadIdx.x; j < k; j += nthreads()) del[j] = 0.0f;
    __syncthreads();
    for (int sweep = 0; sweep < kMaxSweeps && k > 1; ++sweep) {
        if (threadIdx.x == 0) *s_rot = 0;
        for (int jb = 4 * warp; jb < k; jb += 4 * nwarps()) {
            const int j = jb + (lane >> 3);
            double a = 0.0;
#pragma unroll
            for (int r = 0; r < RG; ++r) {
                const int i = sl + 8 * r;
                const double x = j < k ? G[j * ldg + i] : 0.0;
                a = fma(x, x, a);
            }
            a = seg8_sum(a);
            if (j < k && sl == 0) nrm[j] = a;
        }
        __syncthreads();
        if (sweep > 0) {
            const int np = k * (k - 1) / 2;
            int over = 0;
            for (int eb = 4 * warp; eb < np; eb += 4 * nwarps()) {
                const int e = min(eb + (lane >> 3), np - 1);
                int q = (int)((sqrtf(8.0f * e + 1.0f) + 1.0f) * 0.5f);   // e = q (q - 1) / 2 + p, p < q
                q += q * (q + 1) / 2 <= e;
                q -= q * (q - 1) / 2 > e;
                const int p = e - q * (q - 1) / 2;
                double g = 0.0;
#pragma unroll
                for (int r = 0; r < RG; ++r) g = fma(G[p * ldg + sl + 8 * r], G[q * ldg + sl + 8 * r], g);
                g = seg8_sum(g);
                const double a = nrm[p], b = nrm[q];
                const float af = to_float_scaled(a, 0), bf = to_float_scaled(b, 0), gs = fabsf(to_float_scaled(g, 48));
                const float nab = (af * rsqrt_fast(af)) * (bf * rsqrt_fast(bf));
                float t = 0.0f;
                if (fminf(af, bf) > tiny && gs > tol * nab) {
                    t = jacobi_angle(b - a, g);
                    over |= gs > 0x1p20f * nab || fabsf(t) > 0x1p-28f ? 3 : 1;
                }
                if (sl == 0 && eb + (lane >> 3) < np) {
                    Xf[q * k + p] = -t;
                    Xf[p * k + q] = t;
                }
            }
            if (over) atomicOr(s_rot, over);
            __syncthreads();
            const int state = *s_rot;
            if (state == 0) break;
            if (state == 1) {
                for (int j = threadIdx.x; j < k; j += nthreads()) Xf[j * k + j] = 0.0f;
                for (int e = threadIdx.x; e < k * ldg; e += nthreads()) Gf[e] = to_float_scaled(G[e], 0);
                for (int e = threadIdx.x; e < k * ldv; e += nthreads()) Vf[e] = to_float_scaled(V[e], 0);
                __syncthreads();
                for (int e = threadIdx.x; e < k * 8 * RG; e += nthreads()) {
                    const int p = e / (8 * RG), i = e % (8 * RG);
                    float acc = 0.0f;
                    for (int q = 0; q < k; ++q) acc = fmaf(Gf[q * ldg + i], Xf[q * k + p], acc);
                    G[p * ldg + i] += to_double(acc);
                }
                for (int e = threadIdx.x; e < k * 8 * RV; e += nthreads()) {
                    const int p = e / (8 * RV), i = e % (8 * RV);
                    float acc = 0.0f;
                    for (int q = 0; q < k; ++q) acc = fmaf(Vf[q * ldv + i], Xf[q * k + p], acc);
                    V[p * ldv + i] += to_double(acc);
                }
                break;
            }
        }
        if (warp < nact) {
            const int u = 4 * warp + (lane >> 3);
            SegPair pr(u, k);
            for (int round = 0; round < n2 - 1; ++round, pr.next()) {
                int p, q;
                const bool on = pr.get(&p, &q);
                double* Gp = G + p * ldg;
                double* Gq = G + q * ldg;
                double xp[RG], xq[RG];
                double g = 0.0;
#pragma unroll
                for (int r = 0; r < RG; ++r) {
                    const int i = sl + 8 * r;
                    xp[r] = on ? Gp[i] : 0.0;
                    xq[r] = on ? Gq[i] : 0.0;
                    g = fma(xp[r], xq[r], g);
                }
                const double a = on ? nrm[p] : 0.0, b = on ? nrm[q] : 0.0;
                const float dp = on ? del[p] : 0.0f, dq = on ? del[q] : 0.0f;
                const float af = to_float_scaled(a, 0), bf = to_float_scaled(b, 0);
                const float nab = (af * rsqrt_fast(af)) * (bf * rsqrt_fast(bf));
                const double d = b - a;
                g = seg8_sum(g);
                const float gs = fabsf(to_float_scaled(g, 48));
                const bool rot = on && fminf(af, bf) > tiny && gs > tol * nab;
                SegRot* out = ring + (round & 1) * 32 + u;
                if (!__any_sync(0xffffffffu, rot)) {
                    if (sl == 0) out->mode = 0;
                    bar_first(64 * nact);
                    continue;
                }
                const float t = rot ? jacobi_angle(d, g) : 0.0f;
                const bool small = fabsf(t) < 0x1p-14f && fabsf(dp) < 0x1p-30f && fabsf(dq) < 0x1p-30f;
                const double td = to_double(t);
                double fp = 1.0, fq = 1.0;
                double sq = fma(td, to_double(dq - dp), td);
                double sp = fma(td, to_double(dp - dq), td);
                if (__any_sync(0xffffffffu, rot && !small)) {
                    if (!small) {
                        const double c = rsqrt(fma(td, td, 1.0)), s = c * td;
                        const double ep = to_double(dp), eq = to_double(dq);
                        fp = fma(c, ep, c);
                        fq = fma(c, eq, c);
                        sq = fma(s, eq, s);
                        sp = fma(s, ep, s);
                    }
                    if (rot) {
#pragma unroll
                        for (int r = 0; r < RG; ++r) {
                            const int i = sl + 8 * r;
                            Gp[i] = fma(-sq, xq[r], fp * xp[r]);
                            Gq[i] = fma(sp, xp[r], fq * xq[r]);
                        }
                    }
                } else if (rot) {
#pragma unroll
                    for (int r = 0; r < RG; ++r) {
                        const int i = sl + 8 * r;
                        Gp[i] = fma(-sq, xq[r], xp[r]);
                        Gq[i] = fma(sp, xp[r], xq[r]);
                    }
                }
                if (sl == 0) {
                    out->mode = rot ? (small ? 1 : 2) : 0;
                    if (rot) {
                        out->fp = fp;
                        out->sq = sq;
                        out->sp = sp;
                        out->fq = fq;
                        out->p = p;
                        out->q = q;
                        nrm[p] = fma(-td, g, a);
                        nrm[q] = fma(td, g, b);
                        const float h = 0.5f * t * t;
                        del[p] = small ? dp - h : 0.0f;
                        del[q] = small ? dq - h : 0.0f;
                    }
                }
                bar_first(64 * nact);
            }
        } else if (warp < 2 * nact) {
            const int u = 4 * (warp - nact) + (lane >> 3);
            for (int round = 0; round < n2 - 1; ++round) {
                bar_first(64 * nact);
                const SegRot* in = ring + (round & 1) * 32 + u;
                const int mode = in->mode;
                if (!__any_sync(0xffffffffu, mode != 0)) continue;
                if (mode) {
                    const double fp = in->fp, sq = in->sq, sp = in->sp, fq = in->fq;
                    double* Vp = V + in->p * ldv;
                    double* Vq = V + in->q * ldv;
                    if (mode == 1) {
#pragma unroll
                        for (int r = 0; r < RV; ++r) {
                            const int i = sl + 8 * r;
                            const double vp = Vp[i], vq = Vq[i];
                            Vp[i] = fma(-sq, vq, vp);
                            Vq[i] = fma(sp, vp, vq);
                        }
                    } else {
#pragma unroll
                        for (int r = 0; r < RV; ++r) {
                            const int i = sl + 8 * r;
                            const double vp = Vp[i], vq = Vq[i];
                            Vp[i] = fma(-sq, vq, fp * vp);
                            Vq[i] = fma(sp, vp, fq * vq);
                        }
                    }
                }
                __syncwarp();
            }
        }
        __syncthreads();
    }
    __syncthreads();
}

// V (k x k row-major, k <= 64) <- an orthogonal matrix Qp = P (I - E/2 + 3/8 E^2 - 5/16 E^3) next
// to P = V, E = P^T P - I, with the square and cube of E in FP32 (they take a third of the FP64
// instructions otherwise).  What one pass leaves of Qp^T Qp - I is bounded through ||E||_F, which
// bounds ||E||_2 whatever the signs of the entries: the dropped term, 35/64 ||E||^4, and the FP32
// rounding of 3/4 E^2, at most (4 + k) 2^-24 of it (sums of k terms; sqrt(k) in place of k where
// roundings are random).  ||E||_F^2 < 6e-11 k keeps the first below 2e-21 k^2 and the second
// below k eps (k eps / 6 at random roundings), the limit to which the Jacobi itself takes cosines;
// otherwise another pass follows.  false: E is not small (non-finite entries, no rotations to speak of).
// scr: 2 k^2 doubles; own: this thread's entries threadIdx.x + n blockDim of the result; red: 33 doubles.
// (One pass with the cube instead of two without it: k = 60 330 -> 134 us, k = 20 22 -> 9.5 us.)
constexpr float kOrthOnePass = 6e-11f;
constexpr int kOwn = 8;   // outputs of a product per thread: rows k <= 8 blockDim (blockDim >= min(16 k, 512))
__device__ __forceinline__ bool orthogonalise(double* V, int k, double* scr, double (&own)[kOwn], double* red) {
    const int T = nthreads(), kk = k * k, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* Ef = (float*)(scr + kk);   // E in FP32
    float* Tf = Ef + kk;
    float* part = (float*)red;
    for (int pass = 0; pass < 3; ++pass) {
        __syncthreads();
        float f2 = 0.0f;
        for (int e = threadIdx.x; e < k * (k + 1) / 2; e += T) {
            // row i, column j <= i of the symmetric E
            int i = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
            i += (i + 1) * (i + 2) / 2 <= e;
            i -= i * (i + 1) / 2 > e;
            const int j = e - i * (i + 1) / 2;
            double acc = i == j ? -1.0 : 0.0;
            for (int r = 0; r < k; ++r) acc = fma(V[r * k + i], V[r * k + j], acc);
            scr[i * k + j] = scr[j * k + i] = acc;
            const float af = to_float_scaled(acc, 0);
            Ef[i * k + j] = Ef[j * k + i] = af;
            f2 = fmaf(i == j ? af : 2.0f * af, af, f2);
        }
        for (int o = 16; o > 0; o >>= 1) f2 += __shfl_xor_sync(0xffffffffu, f2, o);
        if (lane == 0) part[warp] = f2;
        __syncthreads();
        f2 = 0.0f;
        for (int w = 0; w < nwarps(); ++w) f2 += part[w];
        if (!(f2 < 0.0625f)) return false;
        // Tf = -3/8 E + 5/16 E^2, then F = E/2 + E Tf
        for (int e = threadIdx.x; e < kk; e += T) {
            const int i = e % k, j = e / k;
            float acc = 0.0f;
            for (int m = 0; m < k; ++m) acc = fmaf(Ef[m * k + i], Ef[j * k + m], acc);
            Tf[e] = fmaf(0.3125f, acc, -0.375f * Ef[e]);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < kk; e += T) {
            const int i = e % k, j = e / k;
            float acc = 0.0f;
            for (int m = 0; m < k; ++m) acc = fmaf(Ef[m * k + i], Tf[j * k + m], acc);
            scr[e] = fma(0.5, scr[e], to_double(acc));
        }
        __syncthreads();
        // P (I - F): row i of V (row-major) times the symmetric F
#pragma unroll
        for (int n = 0; n < kOwn; ++n) {
            const int e = threadIdx.x + n * T;
            if (e < kk) {
                const int c = e % k, i = e / k;
                double acc = 0.0;
                for (int j = 0; j < k; ++j) acc = fma(V[i * k + j], scr[j * k + c], acc);
                own[n] = V[e] - acc;
            }
        }
        __syncthreads();
#pragma unroll
        for (int n = 0; n < kOwn; ++n) {
            const int e = threadIdx.x + n * T;
            if (e < kk) V[e] = own[n];
        }
        if (f2 < kOrthOnePass * (float)k) return true;
    }
    return false;
}

// One-sided Jacobi of G (rows x k, column-major, k <= rows <= 64) as jacobi(): G ends
// as U diag(Sraw), V (k x k) accumulates the rotations.  The FP64 sweeps are few because an
// FP32 Jacobi of G comes first (FP32 arithmetic runs at 64 times the FP64 rate
// here): its rotations P, orthogonal to about 3e-6, are orthogonalised in FP64
// (orthogonalise()), and the FP64 Jacobi starts from G Qp with V = Qp: one sweep and a
// step of first order.  Where the FP32
// iteration gives nothing (non-finite entries) it starts from G and I.
// RG, RV: rows of G and V in units of 8 (8 RG >= rows, 8 RV >= k).  Leading dimensions:
// jacobi_ld of max(rows, 8 RG - 7) for G (its padding zero on entry) and of
// max(k, 8 RV - 7) for V, so that the 8 RG (8 RV) rows a lane segment walks stay
// within the column.  scr: jacobi_scratch(ldg, ldv, k) shared doubles; del: k of them.
// Tri: G is lower triangular (rows = k).  pre: with the FP32 start.
template <int RG, int RV, bool Tri>
__device__ __forceinline__ void jacobi_pre(double* G, double* V, double* Sraw, int rows, int k, double* scr,
                                           double* del, SegRot* ring, double* red, int* s_int, bool pre) {
    const int T = nthreads(), kk = k * k;
    const int ldg = jacobi_ld(max(rows, 8 * RG - 7)), ldv = jacobi_ld(max(k, 8 * RV - 7));   // >= 8 RG, 8 RV
    double f = 0.0;
    for (int e = threadIdx.x; e < k * ldg; e += T) f = fma(G[e], G[e], f);
    f = block_sum(f, red);
    // exact scaling to ||G||_F in [1/2, 1)
    int ex = 0;
    if (f > 0.0 && f < DBL_MAX) frexp(sqrt(f), &ex);
    const double sc = ldexp(1.0, -ex);
    const double fro = f * sc * sc;
    float* Gf = (float*)scr;
    float* Vf = Gf + k * ldg;
    for (int e = threadIdx.x; e < k * ldg; e += T) {
        const double x = G[e] * sc;
        G[e] = x;
        Gf[e] = (float)x;
    }
    for (int e = threadIdx.x; e < k * ldv; e += T) Vf[e] = e % ldv == e / ldv ? 1.0f : 0.0f;
    __syncthreads();
    double own[kOwn];
    bool ok = false;
    if (pre) {
        jacobi_f32_segments<RG, RV>(Gf, Vf, k, ldg, ldv, s_int);
        // V row-major <- P
        for (int e = threadIdx.x; e < kk; e += T) V[(e % k) * k + e / k] = to_double(Vf[(e / k) * ldv + e % k]);
        ok = orthogonalise(V, k, scr, own, red);
    }
    __syncthreads();
    if (ok) {
        // G <- G Qp, row i to consecutive threads (rows k <= 8 blockDim outputs); V to column-major
        double gq[kOwn];
#pragma unroll
        for (int n = 0; n < kOwn; ++n) {
            const int e = threadIdx.x + n * T;
            if (e < rows * k) {
                const int i = e / k, c = e % k;
                const int jn = Tri ? i + 1 : k;
                double acc = 0.0;
                for (int j = 0; j < jn; ++j) acc = fma(G[j * ldg + i], V[j * k + c], acc);
                gq[n] = acc;
            }
        }
        __syncthreads();
#pragma unroll
        for (int n = 0; n < kOwn; ++n) {
            const int e = threadIdx.x + n * T;
            if (e < rows * k) G[(e % k) * ldg + e / k] = gq[n];
            if (e < kk) V[(e % k) * ldv + e / k] = own[n];
        }
    } else {
        for (int e = threadIdx.x; e < k * ldv; e += T) V[e] = e % ldv == e / ldv ? 1.0 : 0.0;
    }
    for (int e = threadIdx.x; e < k * (ldv - k); e += T) V[(e / (ldv - k)) * ldv + k + e % (ldv - k)] = 0.0;
    __syncthreads();
    float* dl = (float*)del;
    jacobi_f64_segments<RG, RV>(G, V, Sraw, dl, k, rows, ldg, ldv, fro, scr, ring, s_int);
    // the columns' scales, and the norms of the result
    const double up = ldexp(1.0, ex);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sl = lane & 7;
    for (int jb = 4 * warp; jb < k; jb += 4 * nwarps()) {
        const int j = jb + (lane >> 3);
        double a = 0.0;
        if (j < k) {
            const double s1 = 1.0 + to_double(dl[j]);
            for (int i = sl; i < rows; i += 8) {
                const double x = G[j * ldg + i] * s1;
                a = fma(x, x, a);
                G[j * ldg + i] = x * up;
            }
            for (int i = sl; i < k; i += 8) V[j * ldv + i] *= s1;
        }
        a = seg8_sum(a);
        if (j < k && sl == 0) Sraw[j] = sqrt_via_rsqrt(a) * up;
    }
    __syncthreads();
}

// Shared doubles of jacobi_pre()'s scratch: G, V and a k x k matrix in FP32, or a k x k
// matrix in FP64 and two in FP32.
__host__ __device__ constexpr int jacobi_scratch(int ldg, int ldv, int k) {
    const int f = (k * (ldg + ldv + k) + 1) / 2;
    return f > 2 * k * k ? f : 2 * k * k;
}

// jacobi_pre() on a square lower triangular G of k <= 64 columns (blockDim as svd_block_for() gives it).
// G and V: leading dimension jacobi_ld(k).
__device__ __forceinline__ void jacobi_auto(double* G, double* V, double* Sraw, int k, double* scr, double* del,
                                            SegRot* ring, double* red, int* s_rot, bool pre) {
    if (k <= 8)
        jacobi_pre<1, 1, true>(G, V, Sraw, k, k, scr, del, ring, red, s_rot, pre);
    else if (k <= 16)
        jacobi_pre<2, 2, true>(G, V, Sraw, k, k, scr, del, ring, red, s_rot, pre);
    else if (k <= 24)
        jacobi_pre<3, 3, true>(G, V, Sraw, k, k, scr, del, ring, red, s_rot, pre);
    else if (k <= 32)
        jacobi_pre<4, 4, true>(G, V, Sraw, k, k, scr, del, ring, red, s_rot, pre);
    else if (k <= 40)
        jacobi_pre<5, 5, true>(G, V, Sraw, k, k, scr, del, ring, red, s_rot, pre);
    else if (k <= 56)
        jacobi_pre<7, 7, true>(G, V, Sraw, k, k, scr, del, ring, red, s_rot, pre);
    else
        jacobi_pre<8, 8, true>(G, V, Sraw, k, k, scr, del, ring, red, s_rot, pre);
}

// One-sided (Hestenes) Jacobi on the columns of G (k x k, column-major) with the
// rotations accumulated in V (initialised here), parallel round-robin pair
// order.  zeta = (b - a)/(2 g), t = sign(zeta)/(|zeta| + sqrt(1 + zeta^2)),
// c = 1/sqrt(1 + t^2), s = c t.  A pair is rotated while |g| > k eps sqrt(a b)
// and both columns are above the numerical-zero level k eps ||G||_F; a sweep
// without rotations ends the iteration.  Sraw: column norms of the result.
__device__ __forceinline__ void jacobi(double* G, double* V, double* Sraw, int k, double* red, int* s_rot) {
    if (k <= 16) {
        jacobi_small(G, V, Sraw, k, red, s_rot);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double f = 0.0;
    for (int64_t e = threadIdx.x; e < (int64_t)k * k; e += nthreads()) {
        const double v = G[e];
        f += v * v;
        V[e] = (e % k) == (e / k) ? 1.0 : 0.0;
    }
    f = block_sum(f, red);
    const double tol = (double)k * DBL_EPSILON;
    const double tiny2 = tol * tol * f;
    const int n2 = k + (k & 1);
    for (int sweep = 0; sweep < kMaxSweeps && k > 1; ++sweep) {
        if (threadIdx.x == 0) *s_rot = 0;
        __syncthreads();
        for (int round = 0; round < n2 - 1; ++round) {
            for (int pi = warp; pi < n2 / 2; pi += nwarps()) {
                int p = rr_player(pi, round, n2), q = rr_player(n2 - 1 - pi, round, n2);
                if (p >= k || q >= k) continue;
                if (p > q) {
                    const int tmp = p;
                    p = q;
                    q = tmp;
                }
                double a = 0.0, b = 0.0, g = 0.0;
                for (int i = lane; i < k; i += 32) {
                    const double xp = G[(int64_t)p * k + i], xq = G[(int64_t)q * k + i];
                    a += xp * xp;
                    b += xq * xq;
                    g += xp * xq;
                }
                a = warp_sum(a);
                b = warp_sum(b);
                g = warp_sum(g);
                if (g != 0.0 && fabs(g) > tol * sqrt(a * b) && fmin(a, b) > tiny2) {
                    const double zeta = (b - a) / (2.0 * g);
                    const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                    const double c = 1.0 / sqrt(1.0 + t * t), s = c * t;
                    for (int i = lane; i < k; i += 32) {
                        const double xp = G[(int64_t)p * k + i], xq = G[(int64_t)q * k + i];
                        G[(int64_t)p * k + i] = c * xp - s * xq;
                        G[(int64_t)q * k + i] = s * xp + c * xq;
                        const double vp = V[(int64_t)p * k + i], vq = V[(int64_t)q * k + i];
                        V[(int64_t)p * k + i] = c * vp - s * vq;
                        V[(int64_t)q * k + i] = s * vp + c * vq;
                    }
                    if (lane == 0) *s_rot = 1;
                }
            }
            __syncthreads();
        }
        const int rot = *s_rot;
        __syncthreads();
        if (!rot) break;
    }
    for (int j = warp; j < k; j += nwarps()) {
        double a = 0.0;
        for (int i = lane; i < k; i += 32) {
            const double x = G[(int64_t)j * k + i];
            a += x * x;
        }
        a = warp_sum(a);
        if (lane == 0) Sraw[j] = sqrt(a);
    }
    __syncthreads();
}

// SVD of an M x N matrix from QR + Jacobi of its k x k triangular factor:
// tall (M >= N): M = Q R, R^T = G, G V = U' S  =>  U = Q V, Vt = U'^T;
// wide (M < N):  M^T = Q R, R^T = G, G V = U' S => U = U', Vt = (Q V)^T.
// QV: column-major len x k (QV[p*len + i] = (Q V)(i, p)).  Writes S (k,
// descending, ties by index), US = U diag(S) (M x k row-major) and Vt (k x N
// row-major, row strides ldus / ldvt) with the largest-|.| entry of every Vt
// row positive.  This CTA writes the singular triples r0 .. r1 - 1.  perm: k ints,
// rinv: k doubles (the same values from every CTA).
__device__ __forceinline__ void svd_assemble(const double* G, int ldg, const double* QV, const double* Sraw,
                                             double* rinv, int* perm, double* S, double* US, double* Vt, int M,
                                             int N, int k, int len, int wide, int ldus, int ldvt, int r0, int r1) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < k; i += nthreads()) {
        // compared as integers: a permutation also when a value is not a number
        const long long si = nonneg_key(Sraw[i]);
        int rank = 0;
        for (int j = 0; j < k; ++j) {
            const long long sj = nonneg_key(Sraw[j]);
            rank += (sj > si || (sj == si && j < i)) ? 1 : 0;
        }
        perm[rank] = i;
        if (!wide) {
            const double r = rsqrt(Sraw[i]);
            rinv[i] = Sraw[i] > 0.0 ? r * r : 0.0;
        }
    }
    __syncthreads();
    const int nr = r1 - r0;
    for (int64_t e = threadIdx.x; e < (int64_t)M * nr; e += nthreads()) {
        const int i = (int)(e / nr), r = r0 + (int)(e % nr);
        const int p = perm[r];
        US[(int64_t)i * ldus + r] = wide ? G[(int64_t)p * ldg + i] : Sraw[p] * QV[(int64_t)p * len + i];
    }
    for (int64_t e = threadIdx.x; e < (int64_t)nr * N; e += nthreads()) {
        const int r = r0 + (int)(e / N), c = (int)(e % N);
        const int p = perm[r];
        Vt[(int64_t)r * ldvt + c] = wide ? QV[(int64_t)p * len + c] : G[(int64_t)p * ldg + c] * rinv[p];
    }
    for (int r = r0 + (int)threadIdx.x; r < r1; r += nthreads()) S[r] = Sraw[perm[r]];
    __syncthreads();
    for (int r = r0 + warp; r < r1; r += nwarps()) {
        long long best = -1;
        int bi = 0;
        for (int c = lane; c < N; c += 32) {
            const long long a = abs_key(Vt[(int64_t)r * ldvt + c]);
            if (a > best) {
                best = a;
                bi = c;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ob > best || (ob == best && oi < bi)) {
                best = ob;
                bi = oi;
            }
        }
        if (Vt[(int64_t)r * ldvt + bi] < 0.0) {
            for (int c = lane; c < N; c += 32) Vt[(int64_t)r * ldvt + c] = -Vt[(int64_t)r * ldvt + c];
            for (int i = lane; i < M; i += 32) US[(int64_t)i * ldus + r] = -US[(int64_t)i * ldus + r];
        }
    }
}

}  // namespace dev
}  // namespace bsm
