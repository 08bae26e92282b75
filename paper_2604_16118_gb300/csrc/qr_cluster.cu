// Householder QR of one M x N matrix on one thread-block cluster: the columns of
// A and of Q are spread cyclically over the shared memories of the cluster's
// CTAs (column p on CTA p mod C), so the trailing updates of a column use the
// FP64 units of C SMs (one SM retires one FP64 warp instruction per 16 cycles
// on this GPU, which bounds a one-CTA QR).
//
// What bounds it is the chain from one reflector to the next (two reductions, a
// reciprocal square root and a reciprocal, the hand-over to the other CTAs), so
// that chain runs ahead: in step j the owner of column j + 1 applies H_j to that
// column first, forms H_{j+1} (dev::reflector_vector()) and
// writes v, tau and v_{j+1} straight into every CTA's shared memory, while all
// other warps of the cluster apply H_j to the columns beyond.  One cluster
// barrier per column ends the step.  A column of a trailing update is worked on by
// 8, 16 or 32 lanes, the fewer the more columns a CTA holds (fewer reduction
// steps per column), so that all four schedulers stay busy.
// Q = H_0 ... H_{k-1} applied to the first k columns of I is formed afterwards
// by every CTA for its own Q columns, the reflectors pulled from their owners a
// few at a time.  diag(R) >= 0: row j of R and column j of Q change sign when
// beta_j < 0.  Output as QrTask of k_qr: Q (M x k, column-major), R (k x N,
// row-major).
#include <cooperative_groups.h>

#include <algorithm>

#include "dense_dev.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace bsm {
namespace {

constexpr int kQcThreads = 256;
constexpr int kQcWarps = kQcThreads / 32;
constexpr size_t kQcSmemMax = 220 * 1024;
constexpr int kQcLongRows = 256;   // from this many rows on four warps share a column's chain

// shared memory of one CTA: its A and Q columns, one pulled reflector, tau and the reflectors' diagonals
size_t qc_smem(int M, int N, int C) {
    const int k = std::min(M, N);
    const size_t na = (size_t)(N + C - 1) / C, nq = (size_t)(k + C - 1) / C;
    return sizeof(double) * ((na + nq + 1) * (size_t)M + 2 * (size_t)k);
}
// The kernel pulls up to 8 reflectors at a time where shared memory has room for more than one.
constexpr int kQcPull = 8;
int qc_pull(int M, int N, int C) {
    const size_t base = qc_smem(M, N, C);
    if (base >= kQcSmemMax) return 1;
    return (int)std::min<size_t>(kQcPull, 1 + (kQcSmemMax - base) / (sizeof(double) * (size_t)M));
}

template <int L>
__device__ __forceinline__ double seg_sum_of(double v) {
#pragma unroll
    for (int o = L >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Local columns lp (global rank + lp C), lp0 <= lp < n, lp != skip: a -= tau (v^T a) v
// over the rows j .. M-1 (v_j = vj), L lanes per column, by worker w of nw.
template <int L>
__device__ __forceinline__ void qc_update(double* Al, const double* v, double tj, double vj, int M, int j, int lp0,
                                          int n, int skip, int w, int nw, int lane) {
    const int sl = lane & (L - 1);
    for (int cb = lp0 + w * (32 / L); cb < n; cb += nw * (32 / L)) {
        const int lp = cb + lane / L;
        const bool on = lp < n && lp != skip;
        double* a = Al + (size_t)(on ? lp : lp0) * M;
        double d = 0.0;
        if (on) {   // (a segment without a column reads none: another one may be writing it)
            if (sl == 0) d = vj * a[j];
            for (int i = j + 1 + sl; i < M; i += L) d = fma(v[i], a[i], d);
        }
        const double tw = tj * seg_sum_of<L>(d);
        if (on) {
            if (sl == 0) a[j] = fma(-tw, vj, a[j]);
            for (int i = j + 1 + sl; i < M; i += L) a[i] = fma(-tw, v[i], a[i]);
        }
    }
}

// This CTA's columns of Q, L lanes each, through the reflectors j0 + n - 1 .. j0 held in vb (rows from j on).
template <int L, int C>
__device__ __forceinline__ void qc_form(double* Ql, const double* vb, const double* taus, const double* vds, int M,
                                        int j0, int n, int q_loc, int rank, int warp, int lane) {
    const int sl = lane & (L - 1);
    for (int cb = warp * (32 / L); cb < q_loc; cb += kQcWarps * (32 / L)) {
        const int lq = cb + lane / L;
        const int p = lq < q_loc ? rank + lq * C : -1;
        double* q = Ql + (size_t)(lq < q_loc ? lq : 0) * M;
        for (int b = n - 1; b >= 0; --b) {
            const int j = j0 + b;
            const double tj = taus[j];
            if (tj == 0.0) continue;
            const double vj = vds[j];
            const double* v = vb + (size_t)b * M;
            const int i0 = j + ((sl - j) & (L - 1));
            double d = 0.0;
            if (p >= j)
                for (int i = i0; i < M; i += L) d = fma(i == j ? vj : v[i], q[i], d);
            const double tw = tj * seg_sum_of<L>(d);
            if (p >= j)
                for (int i = i0; i < M; i += L) q[i] = fma(-tw, i == j ? vj : v[i], q[i]);
        }
    }
}

// Two CTAs per SM at least: without the figure the compiler aims for four, at 64 registers and
// with spills (three wide workloads: 95.4 -> 94.1, 23.0 -> 20.2 and 113.7 -> 110.9 ms).
template <int C>
__global__ void __launch_bounds__(kQcThreads, 2) k_qr_cluster(const QrTask* __restrict__ tasks) {
    extern __shared__ double qc_sm[];
    __shared__ double part[2][4];
    __shared__ double s_alpha;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const QrTask tk = tasks[blockIdx.x / C];
    const int M = tk.M, N = tk.N, k = M < N ? M : N;
    const int na = (N + C - 1) / C, nq = (k + C - 1) / C;
    double* Al = qc_sm;                          // local column lp = global column rank + lp C
    double* Ql = Al + (size_t)na * M;            // while A is factorised: two reflectors in flight
    double* taus = Ql + (size_t)nq * M;          // tau_j and v_j(j) of every column
    double* vds = taus + k;                      // (tau_j = 0: -R(j, j)); beta_j < 0 exactly when vds[j] > 0
    double* vb = vds + k;                        // pulled reflectors
    const int n_pull = tk.pull;
    const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_loc = rank < N ? (N - 1 - rank) / C + 1 : 0;
    const int nch = M >= kQcLongRows ? 4 : 1;    // warps of the chain
    for (int64_t e = tid; e < (int64_t)n_loc * M; e += kQcThreads) {
        const int lp = (int)(e / M), i = (int)(e % M);
        Al[e] = tk.A[(int64_t)(rank + lp * C) * M + i];
    }
    cluster.sync();   // every CTA runs before the first reflector is written into it
    // sum over the chain's warps; slot: two reductions in a row use different slots
    auto chain_sum = [&](double v, int slot) {
        v = dev::warp_sum_fixed(v);
        if (nch == 1) return v;
        if (lane == 0) part[slot][warp] = v;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        return (part[slot][0] + part[slot][1]) + (part[slot][2] + part[slot][3]);
    };
    // H_{j-1} applied to column j (j > 0), H_j formed and handed to every CTA
    auto chain = [&](int j) {
        double* x = Al + (size_t)(j / C) * M;
        const int t0 = tid, step = 32 * nch;
        double tw = 0.0, vj = 0.0;
        const double* v = Ql + (size_t)((j - 1) & 1) * M;
        if (j > 0) {
            const double tj = taus[j - 1];
            vj = vds[j - 1];
            if (tj != 0.0) {
                double d = t0 == 0 ? vj * x[j - 1] : 0.0;
                for (int i = j + t0; i < M; i += step) d = fma(v[i], x[i], d);
                tw = tj * chain_sum(d, 0);
                if (t0 == 0) x[j - 1] = fma(-tw, vj, x[j - 1]);
            }
        }
        double s = 0.0, alpha = 0.0;
        double* dst = Ql + (size_t)(j & 1) * M;
        for (int i = j + t0; i < M; i += step) {
            const double y = tw != 0.0 ? fma(-tw, v[i], x[i]) : x[i];
            x[i] = y;
            if (i == j) {
                alpha = y;
                continue;
            }
            s = fma(y, y, s);
#pragma unroll
            for (int c = 0; c < C; ++c) cluster.map_shared_rank(dst, c)[i] = y;
        }
        if (nch > 1 && t0 == 0) s_alpha = alpha;   // visible after the reduction's barrier
        s = chain_sum(s, 1);
        alpha = nch > 1 ? s_alpha : __shfl_sync(0xffffffffu, alpha, 0);
        double tj = 0.0, vd = -alpha;
        if (s != 0.0) {
            double beta;
            int shift;
            dev::reflector_vector(alpha, s, &tj, &vd, &beta, &shift);
            if (shift)
                for (int i = j + t0; i < M; i += step) {   // the rows this thread wrote
                    if (i == j) continue;
                    x[i] = ldexp(x[i], -shift);
                    for (int c = 0; c < C; ++c) cluster.map_shared_rank(dst, c)[i] = x[i];
                }
            if (t0 == 0) x[j] = beta;
        }
        if (t0 < C) {
            cluster.map_shared_rank(taus, t0)[j] = tj;
            cluster.map_shared_rank(vds, t0)[j] = vd;
        }
    };
    if (rank == 0 && warp < nch) chain(0);
    cluster.sync();
    for (int j = 0; j < k; ++j) {
        const double tj = taus[j], vj = vds[j];
        const bool own = j + 1 < k && rank == (j + 1) % C;
        if (own && warp < nch) {
            chain(j + 1);
        } else if (tj != 0.0) {
            // in the owner's CTA the other warps, without those on the chain's scheduler when it has one
            int w = warp, nw = kQcWarps;
            if (own && nch == 1) {
                w = (warp & 3) ? (warp >> 2) * 3 + (warp & 3) - 1 : -1;
                nw = kQcWarps / 4 * 3;
            } else if (own) {
                w = warp - nch;
                nw = kQcWarps - nch;
            }
            const int lp0 = j + 1 <= rank ? 0 : (j + 1 - rank + C - 1) / C;
            const int left = n_loc - lp0, skip = own ? (j + 1) / C : -1;
            const double* v = Ql + (size_t)(j & 1) * M;
            if (w >= 0 && left > 0) {
                if (left <= 4)
                    qc_update<32>(Al, v, tj, vj, M, j, lp0, n_loc, skip, w, nw, lane);
                else if (left <= 8)
                    qc_update<16>(Al, v, tj, vj, M, j, lp0, n_loc, skip, w, nw, lane);
                else
                    qc_update<8>(Al, v, tj, vj, M, j, lp0, n_loc, skip, w, nw, lane);
            }
        }
        cluster.sync();
    }
    // Q: this CTA's columns p < k (p = rank + lq C), from the identity, reflectors backwards
    const int q_loc = rank < k ? (k - 1 - rank) / C + 1 : 0;
    for (int64_t e = tid; e < (int64_t)q_loc * M; e += kQcThreads) {
        const int lq = (int)(e / M), i = (int)(e % M);
        Ql[e] = i == rank + lq * C ? 1.0 : 0.0;
    }
    const int half = n_pull >= 2 ? n_pull / 2 : 1;
    auto pull = [&](int j1, double* dst) {   // reflectors max(0, j1 - half) .. j1 - 1
        const int j0 = max(0, j1 - half);
        for (int e = tid; e < (j1 - j0) * M; e += kQcThreads) {
            const int b = e / M, i = e % M, j = j0 + b;
            if (i > j) dst[e] = cluster.map_shared_rank(Al + (size_t)(j / C) * M, j % C)[i];
        }
    };
    pull(k, vb);
    __syncthreads();
    for (int j1 = k, it = 0; j1 > 0; j1 -= half, ++it) {
        const int j0 = max(0, j1 - half);
        const double* cur = vb + (n_pull >= 2 ? (size_t)(it & 1) * half * M : 0);
        double* nxt = vb + (n_pull >= 2 ? (size_t)((it + 1) & 1) * half * M : 0);
        if (n_pull >= 2) pull(j0, nxt);
        if (q_loc <= 4)
            qc_form<32, C>(Ql, cur, taus, vds, M, j0, j1 - j0, q_loc, rank, warp, lane);
        else if (q_loc <= 8)
            qc_form<16, C>(Ql, cur, taus, vds, M, j0, j1 - j0, q_loc, rank, warp, lane);
        else
            qc_form<8, C>(Ql, cur, taus, vds, M, j0, j1 - j0, q_loc, rank, warp, lane);
        __syncthreads();
        if (n_pull < 2) {
            pull(j0, nxt);
            __syncthreads();
        }
    }
    // R (row-major k x N) from this CTA's A columns and Q columns, with the sign rule
    for (int64_t e = tid; e < (int64_t)n_loc * k; e += kQcThreads) {
        const int lp = (int)(e / k), r = (int)(e % k);
        const int c = rank + lp * C;
        tk.R[(int64_t)r * N + c] = c >= r ? (vds[r] > 0.0 ? -1.0 : 1.0) * Al[(size_t)lp * M + r] : 0.0;
    }
    for (int64_t e = tid; e < (int64_t)q_loc * M; e += kQcThreads) {
        const int lq = (int)(e / M), i = (int)(e % M);
        const int p = rank + lq * C;
        tk.Q[(int64_t)p * M + i] = (vds[p] > 0.0 ? -1.0 : 1.0) * Ql[e];
    }
    // no CTA leaves while another may still read its shared memory
    cluster.sync();
}

template <int C>
bool launch_qc(Context* ctx, const std::vector<QrTask>& tasks_in) {
    size_t smem = 0;
    std::vector<QrTask> tasks = tasks_in;
    for (QrTask& t : tasks) {
        if (qc_smem(t.M, t.N, C) > kQcSmemMax) return false;
        t.pull = qc_pull(t.M, t.N, C);
        smem = std::max(smem, qc_smem(t.M, t.N, C) + sizeof(double) * (size_t)(t.pull - 1) * t.M);
    }
    static bool attr = false;
    if (!attr) {
        BSM_CUDA(cudaFuncSetAttribute(k_qr_cluster<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQcSmemMax));
        if (C > 8) BSM_CUDA(cudaFuncSetAttribute(k_qr_cluster<C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        attr = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tasks.size() * C));
    cfg.blockDim = dim3(kQcThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n_clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&n_clusters, k_qr_cluster<C>, &cfg) != cudaSuccess || n_clusters < 1) {
        (void)cudaGetLastError();
        return false;
    }
    Scratch s(ctx);
    const QrTask* d = s.up(tasks);
    BSM_CUDA(cudaLaunchKernelEx(&cfg, k_qr_cluster<C>, d));
    check_launch(ctx);
    return true;
}

}  // namespace

bool qr_cluster_eligible(int M, int N) {
    const int k = std::min(M, N);
    return k >= kClusterQrMin && qc_smem(M, N, 16) <= kQcSmemMax;
}

bool launch_qr_cluster(Context* ctx, const std::vector<QrTask>& tasks, bool narrow_on_8) {
    if (tasks.empty()) return true;
    int nmax = 0;
    for (const QrTask& t : tasks) nmax = std::max(nmax, std::min(t.M, t.N));
    if (narrow_on_8 && nmax <= kClusterNarrowMax && launch_qc<8>(ctx, tasks)) return true;
    return launch_qc<16>(ctx, tasks) || launch_qc<8>(ctx, tasks);
}

}  // namespace bsm
