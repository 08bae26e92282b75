// One-sided Jacobi of a k x k matrix G (k up to kClusterJacobiMax) on one
// thread-block cluster of C CTAs (C = 16, else 8), in a block-cyclic ordering.
//
// The k columns form 2C blocks of b = ceil(k / 2C) columns.  A sweep is a
// round-robin tournament of the blocks by the circle method (position 0 keeps
// block 0, positions 1 .. 2C-1 rotate by one per step; 2C - 1 steps).  In a step
// CTA c holds the blocks at positions c and 2C-1-c in its shared memory and
// rotates every column pair between them in local rounds (round r pairs column
// j of the first block with column (j + r) mod B of the second, one warp per
// pair, __syncthreads between rounds); in the first step of a sweep it also
// rotates the pairs inside both blocks (the round-robin ordering of
// dev::jacobi).  One cluster barrier ends a step; then every CTA pulls the two
// blocks of its next positions from the other CTAs' shared memory into its
// second buffer.  So a sweep still meets every pair of columns once, with 2C
// cluster barriers instead of one per round of k / 2 pairs, and the rotations
// read and write the CTA's own shared memory.  The accumulated rotations V
// (k x k) stay in global memory (L2-resident, read with __ldcg because another
// CTA of the cluster wrote them in an earlier step).
//
// A pair rotates while |g| > k eps sqrt(a b) and min(a, b) > (k eps)^2 ||G||_F^2
// (the rule of dev::jacobi).  A sweep whose rotated pairs all had cosines |g| / sqrt(a b) and
// tangents below m = 2^-28 is the last (at most dev::kMaxSweeps): rotating column p
// against r changes the cosine of p and q by at most 2 m^2, so after the other 2 (k - 2) rotations
// of p and q it is below 4 k m^2 = k eps / 4, and the next sweep would rotate nothing.  On this GPU an SM retires one
// FP64 warp instruction per 16 cycles, so the Jacobi is bound by the number of
// FP64 instructions: the cluster brings the FP64 units of C SMs to one matrix,
// and a rotation takes few of them, as in dev::jacobi_f64_segments: squared norms
// tracked per column (recomputed every sweep), tests and angles in FP32, the
// inner product summed over the warp by integer reductions, small angles
// applied with two FMAs per row and their cosines gathered per column.  Half of
// the warps rotate V one round behind the others, so that its L2 latency and
// G's chain of product, sum and angle overlap (k = 200: 36 instead of 112 FP64
// instructions per pair; a rank-1024 truncation over one charge: 26.7 -> 22.4 ms).  Every CTA takes the same decisions (the rotation flags
// and ||G||_F^2 are combined in a fixed order), so all of them pass the same barriers.
#include <cooperative_groups.h>

#include <algorithm>

#include "dense_dev.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace bsm {
namespace {

constexpr int kClusterThreads = 512;
constexpr int kClusterWarps = kClusterThreads / 32;
constexpr size_t kClusterSmemMax = 222 * 1024;   // beside the static arrays, within 227 KB
constexpr int kRingMax = 24;                     // column pairs of a round
static_assert((kClusterJacobiMax + 15) / 16 + 1 <= kRingMax, "b columns a block on 8 CTAs: at most b + 1 pairs a round");

// Slot strides, in elements, rounded up to 16 bytes so that blocks move between
// the CTAs' shared memories in 16-byte units: FP64 slot = b columns of G, then b
// squared norms and b scales (float); FP32 slot = b columns of G, then b columns
// of V, each part 16-byte aligned.
__host__ __device__ __forceinline__ size_t cols_f64(int b, int k) { return ((size_t)b * k + 1) & ~size_t(1); }
__host__ __device__ __forceinline__ size_t slot_f64(int b, int k) { return cols_f64(b, k) + 2 * (size_t)b; }
__host__ __device__ __forceinline__ size_t part_f32(int b, int k) { return ((size_t)b * k + 3) & ~size_t(3); }

// shared memory of one CTA: two buffers of two block slots
size_t cluster_smem(int k, int ctas, bool f32) {
    const int b = (k + 2 * ctas - 1) / (2 * ctas);
    return f32 ? 4 * 2 * part_f32(b, k) * sizeof(float) : 4 * slot_f64(b, k) * sizeof(double);
}

// Copy n16 16-byte units from src (another CTA's shared memory) to dst, with
// four loads in flight per thread; both 16-byte aligned.
__device__ __forceinline__ void pull16(float4* __restrict__ dst, const float4* __restrict__ src, int n16) {
    constexpr int T = kClusterThreads;
    int e = threadIdx.x;
    for (; e + 3 * T < n16; e += 4 * T) {
        const float4 v0 = src[e], v1 = src[e + T], v2 = src[e + 2 * T], v3 = src[e + 3 * T];
        dst[e] = v0;
        dst[e + T] = v1;
        dst[e + 2 * T] = v2;
        dst[e + 3 * T] = v3;
    }
    for (; e < n16; e += T) dst[e] = src[e];
}

// Block at tournament position p in step s (n2m1 = 2C - 1; position 0 fixed).
__device__ __forceinline__ int block_at(int p, int s, int n2m1) {
    return p == 0 ? 0 : (p - 1 + s) % n2m1 + 1;
}
// Position of block beta in step s (the inverse of block_at).
__device__ __forceinline__ int pos_of(int beta, int s, int n2m1) {
    return beta == 0 ? 0 : ((beta - 1 - s) % n2m1 + n2m1) % n2m1 + 1;
}

// A rotation on its way from a warp that rotated G to one that rotates V.
struct Rot {
    double fp, sq, sp, fq;   // x_p' = fp x_p - sq x_q, x_q' = sp x_p + fq x_q
    int p, q;                // columns of V
    int mode;                // 0: none, 1: fp = fq = 1, 2: full
    int pad;
};

// One warp: rotate columns Gp, Gq (k rows, shared memory), whose squared norms
// and scales stand at np, nq and dp, dq; the rotation to *out.
// lim: k eps 2^48; tiny: (k eps)^2 ||G||_F^2.
__device__ __forceinline__ void rotate_g(double* Gp, double* Gq, double* np, double* nq, float* dp, float* dq, int k,
                                         float lim, float tiny, int gp, int gq, int lane, Rot* out, int* s_rot) {
    double g = 0.0;
    for (int i = lane; i < k; i += 32) g = fma(Gp[i], Gq[i], g);
    const double a = *np, b = *nq;
    const float ep = *dp, eq = *dq;
    const float af = dev::to_float_scaled(a, 0), bf = dev::to_float_scaled(b, 0);
    g = dev::warp_sum_fixed(g);
    const float nab = (af * dev::rsqrt_fast(af)) * (bf * dev::rsqrt_fast(bf)), gs = fabsf(dev::to_float_scaled(g, 48));
    const bool rot = fminf(af, bf) > tiny && gs > lim * nab;
    if (!rot) {
        if (lane == 0) out->mode = 0;
        return;
    }
    const float t = dev::jacobi_angle(b - a, g);
    const bool small = fabsf(t) < 0x1p-14f && fabsf(ep) < 0x1p-30f && fabsf(eq) < 0x1p-30f;
    const double td = dev::to_double(t);
    double fp = 1.0, fq = 1.0, sq, sp;
    if (small) {
        sq = fma(td, dev::to_double(eq - ep), td);
        sp = fma(td, dev::to_double(ep - eq), td);
        for (int i = lane; i < k; i += 32) {
            const double xp = Gp[i], xq = Gq[i];
            Gp[i] = fma(-sq, xq, xp);
            Gq[i] = fma(sp, xp, xq);
        }
    } else {
        const double c = rsqrt(fma(td, td, 1.0)), s = c * td;
        fp = fma(c, dev::to_double(ep), c);
        fq = fma(c, dev::to_double(eq), c);
        sq = fma(s, dev::to_double(eq), s);
        sp = fma(s, dev::to_double(ep), s);
        for (int i = lane; i < k; i += 32) {
            const double xp = Gp[i], xq = Gq[i];
            Gp[i] = fma(-sq, xq, fp * xp);
            Gq[i] = fma(sp, xp, fq * xq);
        }
    }
    __syncwarp();   // every lane has read the norms and scales
    if (lane == 0) {
        out->fp = fp;
        out->sq = sq;
        out->sp = sp;
        out->fq = fq;
        out->p = gp;
        out->q = gq;
        out->mode = small ? 1 : 2;
        *np = fma(-td, g, a);
        *nq = fma(td, g, b);
        const float h = 0.5f * t * t;
        *dp = small ? ep - h : 0.0f;
        *dq = small ? eq - h : 0.0f;
        if (gs > 0x1p20f * nab || fabsf(t) > 0x1p-28f) *s_rot = 1;
    }
}

// One warp: the rotation *in applied to its columns of V (global memory, four row
// groups in flight).
__device__ __forceinline__ void rotate_v(double* V, const Rot* in, int k, int lane) {
    const int mode = in->mode;
    if (!mode) return;
    double* Vp = V + (int64_t)in->p * k;
    double* Vq = V + (int64_t)in->q * k;
    const double fp = in->fp, sq = in->sq, sp = in->sp, fq = in->fq;
    for (int i0 = lane; i0 < k; i0 += 128) {
        double vp[4], vq[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = i0 + 32 * r;
            vp[r] = i < k ? __ldcg(Vp + i) : 0.0;
            vq[r] = i < k ? __ldcg(Vq + i) : 0.0;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = i0 + 32 * r;
            if (i < k) {
                Vp[i] = fma(-sq, vq[r], mode == 1 ? vp[r] : fp * vp[r]);
                Vq[i] = fma(sp, vp[r], mode == 1 ? vq[r] : fq * vq[r]);
            }
        }
    }
}

template <int C>
__global__ void __launch_bounds__(kClusterThreads, 1) k_jacobi_cluster(const JacTask* __restrict__ tasks) {
    extern __shared__ double jc_smem[];
    __shared__ double s_part[C];     // CTA 0's slots: partial ||G||^2 of every CTA
    __shared__ int s_flag[2][C];     // CTA 0's slots: rotation flags, by sweep parity
    __shared__ int s_rot;            // this CTA had a larger rotation in the current sweep
    __shared__ double red[33];
    __shared__ Rot ring[2][kRingMax];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const JacTask tk = tasks[blockIdx.x / C];
    const int k = tk.k;
    constexpr int nblk = 2 * C, n2m1 = 2 * C - 1, kHalf = kClusterWarps / 2;
    const int b = (k + nblk - 1) / nblk;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // slot sl of buffer buf: b columns of k rows, their squared norms and scales
    const size_t ncol = cols_f64(b, k), sstride = slot_f64(b, k);
    auto slot = [&](int buf, int sl) { return jc_smem + (size_t)(buf * 2 + sl) * sstride; };
    auto bcols = [&](int beta) { return max(0, min(b, k - beta * b)); };
    // step 0: CTA c holds blocks c (slot 0) and 2C-1-c (slot 1); load them, set
    // their columns of V to the identity, partial ||G||_F^2
    double f = 0.0;
    for (int sl = 0; sl < 2; ++sl) {
        const int beta = sl == 0 ? rank : nblk - 1 - rank;
        const int nc = bcols(beta);
        double* dst = slot(0, sl);
        const int64_t off = (int64_t)beta * b * k;
        for (int64_t e = threadIdx.x; e < (int64_t)nc * k; e += kClusterThreads) {
            const double v = tk.G[off + e];
            dst[e] = v;
            f = fma(v, v, f);
            const int j = (int)(e / k), i = (int)(e % k);
            if (!tk.v_given) tk.V[off + e] = i == beta * b + j ? 1.0 : 0.0;
        }
    }
    f = dev::block_sum(f, red);
    double* part0 = cluster.map_shared_rank(s_part, 0);
    if (threadIdx.x == 0) {
        part0[rank] = f;
        s_rot = 0;
    }
    cluster.sync();
    double fro = 0.0;
    for (int c = 0; c < C; ++c) fro += part0[c];
    // exact scaling to ||G||_F in [1/2, 1): norms and tests stay in FP32's range
    int ex = 0;
    if (fro > 0.0 && fro < DBL_MAX) frexp(sqrt(fro), &ex);
    const double sc = ldexp(1.0, -ex);
    for (int sl = 0; sl < 2; ++sl) {
        double* X = slot(0, sl);
        const int nc = bcols(sl == 0 ? rank : nblk - 1 - rank);
        for (int e = threadIdx.x; e < nc * k; e += kClusterThreads) X[e] *= sc;
        float* del = (float*)(X + ncol + b);
        for (int j = threadIdx.x; j < b; j += kClusterThreads) del[j] = 0.0f;
    }
    const float epsk = (float)k * 2.220446e-16f;
    const float lim = epsk * 0x1p48f, tiny = epsk * epsk * dev::to_float_scaled(fro * sc * sc, 0);
    int* flag0 = cluster.map_shared_rank(&s_flag[0][0], 0);
    int gstep = 0;   // steps taken: buffer gstep & 1 holds the current blocks
    int par = 0;     // ring half of the current round
    for (int sweep = 0; sweep < dev::kMaxSweeps && k > 1; ++sweep) {
        for (int s = 0; s < n2m1; ++s, ++gstep) {
            const int cur = gstep & 1;
            const int bL = block_at(rank, s, n2m1), bR = block_at(nblk - 1 - rank, s, n2m1);
            const int nL = bcols(bL), nR = bcols(bR);
            double* L = slot(cur, 0);
            double* R = slot(cur, 1);
            int prev = 0;   // rotations of the round before, in the other half of the ring
            // V units spread so that G and V work meet on as many schedulers as possible
            auto rotate_prev = [&]() {
                for (int u = (warp - kHalf - prev) & (kHalf - 1); u < prev; u += kHalf)
                    rotate_v(tk.V, &ring[par ^ 1][u], k, lane);
            };
            if (s == 0) {
                __syncthreads();
                for (int c = warp; c < nL + nR; c += kClusterWarps) {
                    double* X = c < nL ? L : R;
                    const int j = c < nL ? c : c - nL;
                    double a = 0.0;
                    for (int i = lane; i < k; i += 32) a = fma(X[(size_t)j * k + i], X[(size_t)j * k + i], a);
                    a = dev::warp_sum_fixed(a);
                    if (lane == 0) X[ncol + j] = a;
                }
                __syncthreads();
                // pairs inside each block: round-robin over nb2 players per block
                const int nb = max(nL, nR), nb2 = nb + (nb & 1), half = nb2 / 2;
                for (int round = 0; round < nb2 - 1; ++round) {
                    if (warp < kHalf) {
                        for (int u = warp; u < nb2; u += kHalf) {
                            const int pi = u % half, side = u / half;
                            int p = dev::rr_player(pi, round, nb2), q = dev::rr_player(nb2 - 1 - pi, round, nb2);
                            if (p > q) {
                                const int t = p;
                                p = q;
                                q = t;
                            }
                            if (q >= (side == 0 ? nL : nR)) {
                                if (lane == 0) ring[par][u].mode = 0;
                                continue;
                            }
                            double* X = side == 0 ? L : R;
                            float* del = (float*)(X + ncol + b);
                            const int c0 = (side == 0 ? bL : bR) * b;
                            rotate_g(X + (size_t)p * k, X + (size_t)q * k, X + ncol + p, X + ncol + q, del + p, del + q,
                                     k, lim, tiny, c0 + p, c0 + q, lane, &ring[par][u], &s_rot);
                        }
                    } else {
                        rotate_prev();
                    }
                    __syncthreads();
                    par ^= 1;
                    prev = nb2;
                }
            }
            // pairs between the two blocks
            const int B = max(nL, nR);
            float* dL = (float*)(L + ncol + b);
            float* dR = (float*)(R + ncol + b);
            for (int r = 0; r < B; ++r) {
                if (warp < kHalf) {
                    for (int j = warp; j < B; j += kHalf) {
                        const int q = (j + r) % B;
                        if (j >= nL || q >= nR) {
                            if (lane == 0) ring[par][j].mode = 0;
                            continue;
                        }
                        rotate_g(L + (size_t)j * k, R + (size_t)q * k, L + ncol + j, R + ncol + q, dL + j, dR + q, k,
                                 lim, tiny, bL * b + j, bR * b + q, lane, &ring[par][j], &s_rot);
                    }
                } else {
                    rotate_prev();
                }
                __syncthreads();
                par ^= 1;
                prev = B;
            }
            for (int u = warp; u < prev; u += kClusterWarps) rotate_v(tk.V, &ring[par ^ 1][u], k, lane);
            cluster.sync();
            // pull the blocks of the next step's positions into the other buffer
            const int s1 = s + 1 == n2m1 ? 0 : s + 1;
            for (int sl = 0; sl < 2; ++sl) {
                const int beta = block_at(sl == 0 ? rank : nblk - 1 - rank, s1, n2m1);
                const int hp = pos_of(beta, s, n2m1);   // its position in this step
                const int holder = hp < C ? hp : nblk - 1 - hp;
                const double* src = cluster.map_shared_rank(slot(cur, hp < C ? 0 : 1), holder);
                if (bcols(beta) > 0) pull16((float4*)slot(cur ^ 1, sl), (const float4*)src, (int)(sstride / 2));
            }
            __syncthreads();
        }
        // combine the CTAs' rotation flags in CTA 0's slots (parity-indexed, so the
        // slots of one sweep are never reset while another CTA still reads them)
        const int fpar = sweep & 1;
        if (threadIdx.x == 0) {
            flag0[fpar * C + rank] = s_rot;
            s_rot = 0;
        }
        cluster.sync();
        int rot = 0;
        for (int c = 0; c < C; ++c) rot |= flag0[fpar * C + c];
        if (!rot) break;
    }
    // the current blocks (step gstep mod 2C-1 of the tournament) back to global
    // memory times their columns' scales, with the column norms
    const int cur = gstep & 1, s_now = gstep % n2m1;
    const double up = ldexp(1.0, ex);
    for (int sl = 0; sl < 2; ++sl) {
        const int beta = block_at(sl == 0 ? rank : nblk - 1 - rank, s_now, n2m1);
        const int nc = bcols(beta);
        const double* X = slot(cur, sl);
        const float* del = (const float*)(X + ncol + b);
        for (int j = warp; j < nc; j += kClusterWarps) {
            const double s1 = 1.0 + dev::to_double(del[j]);
            const int64_t off = ((int64_t)beta * b + j) * k;
            double a = 0.0;
            for (int i = lane; i < k; i += 32) {
                const double x = X[(size_t)j * k + i] * s1;
                a = fma(x, x, a);
                tk.G[off + i] = x * up;
                tk.V[off + i] = __ldcg(tk.V + off + i) * s1;
            }
            a = dev::warp_sum(a);
            if (lane == 0) tk.Sraw[beta * b + j] = sqrt(a) * up;
        }
    }
    // no CTA leaves while another may still read its shared memory
    cluster.sync();
}

// One-sided Jacobi in FP32 of the k x k FP64 matrix G, as a preconditioner:
// the same block-cyclic tournament as k_jacobi_cluster, with G (scaled by a
// power of two to ||G||_F ~ 1, rounded to FP32) and the accumulated rotations
// V both in the CTAs' shared memory (a block moves with its columns of V).
// FP32 arithmetic runs at 64 times the FP64 rate of this GPU.  A pair rotates
// while |g| > tol sqrt(a) sqrt(b), tol = 4 sqrt(k) eps_32 (above the rounding
// noise of the FP32 inner products), and min(a, b) > 1e-36 (of ||G||_F^2 ~ 1):
// floating point resolves the small columns of a graded G relative to their
// own norms, so they are rotated too, which leaves the FP64 Jacobi only the
// last quadratic sweeps at every scale.  The rotation is that of
// dev::jacobi_f32_segments.  A sweep that rotates at most 1/32 of the pairs ends
// the iteration (at most kMaxSweepsF32).  Output: tk.V = the FP32 V as FP64 (orthogonal to about 1e-6); tk.G is read only; tk.Sraw unused.
constexpr int kMaxSweepsF32 = 20;

__device__ __forceinline__ void rotate_pair_f32(float* Gp, float* Gq, float* Vp, float* Vq, int k, float tol,
                                                int lane, int* s_rot) {
    float a = 0.0f, b = 0.0f, g = 0.0f;
    for (int i = lane; i < k; i += 32) {
        const float xp = Gp[i], xq = Gq[i];
        a = fmaf(xp, xp, a);
        b = fmaf(xq, xq, b);
        g = fmaf(xp, xq, g);
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        g += __shfl_xor_sync(0xffffffffu, g, o);
    }
    if (fabsf(g) > tol * (a * dev::rsqrt_fast(a)) * (b * dev::rsqrt_fast(b)) && fminf(a, b) > 1e-36f) {
        // cos and sin of the rotation from cos(2 theta) = |d| / sqrt(d^2 + 4 g^2), and one
        // Newton step on c^2 + s^2 = 1, as in dev::jacobi_f32_segments
        const float d = b - a, g2 = g + g;
        const unsigned mb = max(__float_as_uint(fabsf(d)), __float_as_uint(fabsf(g2))) >> 23;
        const float sc = __uint_as_float((254u - min(mb, 253u)) << 23);
        const float dn = d * sc, gn = g2 * sc;
        const float ri = dev::rsqrt_fast(fmaf(dn, dn, gn * gn));
        const float c2 = fmaf(0.5f, fabsf(dn) * ri, 0.5f);
        const float rc = dev::rsqrt_fast(c2);
        const float cr = c2 * rc, hr = 0.5f * gn * ri * rc;
        const float fix = fmaf(-0.5f, fmaf(cr, cr, hr * hr), 1.5f);
        const float c = cr * fix, h = hr * fix;
        const float sn = __uint_as_float(__float_as_uint(h) ^ (__float_as_uint(d) & 0x80000000u));
        for (int i = lane; i < k; i += 32) {
            const float xp = Gp[i], xq = Gq[i];
            Gp[i] = c * xp - sn * xq;
            Gq[i] = sn * xp + c * xq;
            const float vp = Vp[i], vq = Vq[i];
            Vp[i] = c * vp - sn * vq;
            Vq[i] = sn * vp + c * vq;
        }
        if (lane == 0) atomicAdd(s_rot, 1);
    }
}

template <int C>
__global__ void __launch_bounds__(kClusterThreads, 1) k_jacobi_cluster_f32(const JacTask* __restrict__ tasks) {
    extern __shared__ float jf_smem[];
    __shared__ double s_part[C];
    __shared__ int s_flag[2][C];
    __shared__ int s_rot;
    __shared__ double red[33];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const JacTask tk = tasks[blockIdx.x / C];
    const int k = tk.k;
    constexpr int nblk = 2 * C, n2m1 = 2 * C - 1;
    const int b = (k + nblk - 1) / nblk;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // slot sl of buffer buf: b columns of G, then b columns of V (k rows each)
    const size_t vpart = part_f32(b, k);   // offset of the V columns in a slot
    auto slot = [&](int buf, int sl) { return jf_smem + (size_t)(buf * 2 + sl) * 2 * vpart; };
    auto bcols = [&](int beta) { return max(0, min(b, k - beta * b)); };
    double f = 0.0;
    for (int sl = 0; sl < 2; ++sl) {
        const int beta = sl == 0 ? rank : nblk - 1 - rank;
        const int64_t off = (int64_t)beta * b * k;
        for (int64_t e = threadIdx.x; e < (int64_t)bcols(beta) * k; e += kClusterThreads) {
            const double v = tk.G[off + e];
            f += v * v;
        }
    }
    f = dev::block_sum(f, red);
    double* part0 = cluster.map_shared_rank(s_part, 0);
    if (threadIdx.x == 0) {
        part0[rank] = f;
        s_rot = 0;
    }
    cluster.sync();
    double fro = 0.0;
    for (int c = 0; c < C; ++c) fro += part0[c];
    int ex = 0;
    if (fro > 0.0) frexp(sqrt(fro), &ex);
    const double sc = ldexp(1.0, -ex);   // exact power of two: ||sc G||_F in [1/2, 1)
    for (int sl = 0; sl < 2; ++sl) {
        const int beta = sl == 0 ? rank : nblk - 1 - rank;
        const int nc = bcols(beta);
        const int64_t off = (int64_t)beta * b * k;
        float* dst = slot(0, sl);
        for (int64_t e = threadIdx.x; e < (int64_t)nc * k; e += kClusterThreads) {
            dst[e] = (float)(tk.G[off + e] * sc);
            const int j = (int)(e / k), i = (int)(e % k);
            dst[vpart + e] = i == beta * b + j ? 1.0f : 0.0f;
        }
    }
    __syncthreads();
    const float tol = 4.0f * sqrtf((float)k) * FLT_EPSILON;
    int* flag0 = cluster.map_shared_rank(&s_flag[0][0], 0);
    int gstep = 0;
    for (int sweep = 0; sweep < kMaxSweepsF32 && k > 1; ++sweep) {
        for (int s = 0; s < n2m1; ++s, ++gstep) {
            const int cur = gstep & 1;
            const int bL = block_at(rank, s, n2m1), bR = block_at(nblk - 1 - rank, s, n2m1);
            const int nL = bcols(bL), nR = bcols(bR);
            float* L = slot(cur, 0);
            float* R = slot(cur, 1);
            float* LV = L + vpart;
            float* RV = R + vpart;
            if (s == 0) {
                const int nb = max(nL, nR), nb2 = nb + (nb & 1), half = nb2 / 2;
                for (int round = 0; round < nb2 - 1; ++round) {
                    for (int u = warp; u < nb2; u += kClusterWarps) {
                        const int pi = u % half, side = u / half;
                        int p = dev::rr_player(pi, round, nb2), q = dev::rr_player(nb2 - 1 - pi, round, nb2);
                        if (p > q) {
                            const int t = p;
                            p = q;
                            q = t;
                        }
                        if (q >= (side == 0 ? nL : nR)) continue;
                        float* X = side == 0 ? L : R;
                        float* XV = side == 0 ? LV : RV;
                        rotate_pair_f32(X + (size_t)p * k, X + (size_t)q * k, XV + (size_t)p * k, XV + (size_t)q * k,
                                        k, tol, lane, &s_rot);
                    }
                    __syncthreads();
                }
            }
            const int B = max(nL, nR);
            for (int r = 0; r < B; ++r) {
                for (int j = warp; j < B; j += kClusterWarps) {
                    const int q = (j + r) % B;
                    if (j >= nL || q >= nR) continue;
                    rotate_pair_f32(L + (size_t)j * k, R + (size_t)q * k, LV + (size_t)j * k, RV + (size_t)q * k, k,
                                    tol, lane, &s_rot);
                }
                __syncthreads();
            }
            cluster.sync();
            const int s1 = s + 1 == n2m1 ? 0 : s + 1;
            for (int sl = 0; sl < 2; ++sl) {
                const int beta = block_at(sl == 0 ? rank : nblk - 1 - rank, s1, n2m1);
                const int hp = pos_of(beta, s, n2m1);
                const int holder = hp < C ? hp : nblk - 1 - hp;
                const float* src = cluster.map_shared_rank(slot(cur, hp < C ? 0 : 1), holder);
                float* dst = slot(cur ^ 1, sl);
                const int n16 = (bcols(beta) * k + 3) / 4;
                pull16((float4*)dst, (const float4*)src, n16);
                pull16((float4*)(dst + vpart), (const float4*)(src + vpart), n16);
            }
            __syncthreads();
        }
        // rotation counts of the sweep; a sweep that rotated at most 1/32 of the
        // pairs ends the FP32 iteration (the FP64 Jacobi takes the rest)
        const int par = sweep & 1;
        if (threadIdx.x == 0) {
            flag0[par * C + rank] = s_rot;
            s_rot = 0;
        }
        cluster.sync();
        int64_t rot = 0;
        for (int c = 0; c < C; ++c) rot += flag0[par * C + c];
        if (32 * rot <= (int64_t)k * (k - 1) / 2) break;
    }
    const int cur = gstep & 1, s_now = gstep % n2m1;
    for (int sl = 0; sl < 2; ++sl) {
        const int beta = block_at(sl == 0 ? rank : nblk - 1 - rank, s_now, n2m1);
        const float* XV = slot(cur, sl) + vpart;
        const int64_t off = (int64_t)beta * b * k;
        for (int64_t e = threadIdx.x; e < (int64_t)bcols(beta) * k; e += kClusterThreads) tk.V[off + e] = XV[e];
    }
    cluster.sync();
}

// One launch of a C-CTA kernel (the FP64 Jacobi, or the FP32 one when f32);
// false (nothing launched) when such clusters cannot be scheduled.
template <int C>
bool launch_cluster_size(Context* ctx, const std::vector<JacTask>& tasks, int kmax, bool f32 = false) {
    const size_t smem = cluster_smem(kmax, C, f32);
    if (smem > kClusterSmemMax) return false;
    void (*kern)(const JacTask*) = f32 ? k_jacobi_cluster_f32<C> : k_jacobi_cluster<C>;
    static bool attr[2] = {false, false};
    if (!attr[f32]) {
        BSM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterSmemMax));
        if (C > 8) BSM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        attr[f32] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tasks.size() * C));
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr_l[1];
    attr_l[0].id = cudaLaunchAttributeClusterDimension;
    attr_l[0].val.clusterDim.x = C;
    attr_l[0].val.clusterDim.y = 1;
    attr_l[0].val.clusterDim.z = 1;
    cfg.attrs = attr_l;
    cfg.numAttrs = 1;
    int n_clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&n_clusters, kern, &cfg) != cudaSuccess || n_clusters < 1) {
        (void)cudaGetLastError();
        return false;
    }
    Scratch s(ctx);
    const JacTask* d = s.up(tasks);
    BSM_CUDA(cudaLaunchKernelEx(&cfg, kern, d));
    check_launch(ctx);
    return true;
}

}  // namespace

// Tasks with k <= kClusterJacobiMax, one cluster each: 16 CTAs per cluster when
// such clusters can be scheduled (more FP64 units per matrix), else 8; false
// (nothing launched) when neither can.
bool launch_jacobi_cluster(Context* ctx, const std::vector<JacTask>& tasks) {
    if (tasks.empty()) return true;
    int kmax = 0;
    for (const JacTask& t : tasks) kmax = std::max(kmax, t.k);
    if (kmax > kClusterJacobiMax) return false;
    return launch_cluster_size<16>(ctx, tasks, kmax) || launch_cluster_size<8>(ctx, tasks, kmax);
}

// The FP32 preconditioning Jacobi (k_jacobi_cluster_f32) of the same tasks, on
// 8-CTA clusters first: the FP32 sweeps are bound by round latency, not by the
// arithmetic of the SMs, and 8 CTAs halve the tournament steps (cluster
// barriers and block pulls) per sweep (measured: full-rank step 12.23 -> 11.86 s).
bool launch_jacobi_cluster_f32(Context* ctx, const std::vector<JacTask>& tasks) {
    if (tasks.empty()) return true;
    int kmax = 0;
    for (const JacTask& t : tasks) kmax = std::max(kmax, t.k);
    if (kmax > kClusterJacobiMax) return false;
    return launch_cluster_size<8>(ctx, tasks, kmax, true) || launch_cluster_size<16>(ctx, tasks, kmax, true);
}

}  // namespace bsm
