// Device kernels: block scatter/copy, segmented FP64 grouped GEMM, batched
// Householder QR and batched one-sided Jacobi SVD for the small dense blocks of
// a block-sparse MPS.  All arithmetic is float64.
#include <cfloat>
#include <cmath>
#include <cstring>

#include "dense_dev.cuh"
#include "kernels.h"

namespace bsm {
namespace {

using dev::block_sum;
using dev::kThreads;
using dev::kWarps;
using dev::warp_sum;

constexpr int64_t kCopyChunk = 16384;

struct CopyChunk {
    int task;
    int64_t beg, end;
};

__global__ void __launch_bounds__(kThreads) k_copy(const CopyTask* __restrict__ tasks,
                                                   const CopyChunk* __restrict__ chunks) {
    const CopyChunk ch = chunks[blockIdx.x];
    const CopyTask tk = tasks[ch.task];
    for (int64_t e = ch.beg + threadIdx.x; e < ch.end; e += blockDim.x) {
        const int i = (int)(e / tk.cols), j = (int)(e % tk.cols);
        const int64_t si = tk.src_cm ? (int64_t)j * tk.src_ld + i : (int64_t)i * tk.src_ld + j;
        const int64_t di = tk.dst_cm ? (int64_t)j * tk.dst_ld + i : (int64_t)i * tk.dst_ld + j;
        const double v = tk.f * tk.src[si];
        if (tk.accumulate)
            tk.dst[di] += v;
        else
            tk.dst[di] = v;
    }
}

struct GemmTile {
    int out, m0, n0;
};

constexpr int kTile = dev::kGemmTile;
constexpr int kSmallGemmThreads = 128;

// Contributions that read the same B block (untransposed): their A blocks are summed first,
// sum_c alpha_c A_c B = (sum_c alpha_c A_c) B.  In the zip-up contraction every output has at
// most two B blocks (one per occupation of the site) and as many contributions as operator
// entries, so the products shrink from one per entry to two.
__host__ __device__ __forceinline__ bool same_b(const GemmIn& x, const GemmIn& y) {
    return x.B == y.B && x.K == y.K && x.ldb == y.ldb && !x.transA && !y.transA;
}

// One run in[0 .. n) of such contributions (n = 1 when transposed) added to a tile of tm x tn
// entries, which the threads own flat (entry e = thread + 256 q at row em, column en: a small
// block then fills whole warps); the sum of the A blocks is formed while they are staged.
__device__ __forceinline__ void tile_accumulate_run(const GemmIn* in, int n, int m0, int n0, int tm, int tn,
                                                    const int* em, const int* en, double (*As)[kTile + 1],
                                                    double (*Bs)[kTile + 1], double acc[4]) {
    const int K = in[0].K, ldb = in[0].ldb, tid = (int)threadIdx.x;
    const double* B = in[0].B;
    for (int k0 = 0; k0 < K; k0 += kTile) {
        const int kk_end = min(kTile, K - k0);
        if (in[0].transA) {
            for (int e = tid; e < kk_end * tm; e += kThreads) {
                const int kk = e / tm, mm = e - kk * tm;
                As[kk][mm] = in[0].alpha * in[0].A[(int64_t)(k0 + kk) * in[0].lda + m0 + mm];
            }
        } else {
            for (int e = tid; e < tm * kk_end; e += kThreads) {
                const int mm = e / kk_end, kk = e - mm * kk_end;
                double v = 0.0;
#pragma unroll 4
                for (int u = 0; u < n; ++u)
                    v = fma(in[u].alpha, in[u].A[(int64_t)(m0 + mm) * in[u].lda + k0 + kk], v);
                As[kk][mm] = v;
            }
        }
        for (int e = tid; e < kk_end * tn; e += kThreads) {
            const int kk = e / tn, nn = e - kk * tn;
            Bs[kk][nn] = B[(int64_t)(k0 + kk) * ldb + n0 + nn];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (tid + q * kThreads < tm * tn)
                for (int kk = 0; kk < kk_end; ++kk) acc[q] = fma(As[kk][em[q]], Bs[kk][en[q]], acc[q]);
        __syncthreads();
    }
}

// 32 x 32 output tile per CTA.
constexpr int kGemmIns = 64;   // descriptors staged at a time
__global__ void __launch_bounds__(kThreads) k_gemm(const GemmOut* __restrict__ outs,
                                                   const GemmIn* __restrict__ ins,
                                                   const GemmTile* __restrict__ tiles) {
    __shared__ double As[kTile][kTile + 1];   // [k][m]
    __shared__ double Bs[kTile][kTile + 1];   // [k][n]
    __shared__ GemmIn s_in[kGemmIns];
    const GemmTile tl = tiles[blockIdx.x];
    const GemmOut o = outs[tl.out];
    const int tm = min(kTile, o.M - tl.m0), tn = min(kTile, o.N - tl.n0);
    int em[4], en[4];
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int e = threadIdx.x + q * kThreads;
        em[q] = e / tn;
        en[q] = e - em[q] * tn;
    }
    for (int cb = o.beg; cb < o.end; cb += kGemmIns) {
        const int n = min(kGemmIns, o.end - cb);
        constexpr int kWords = (int)(sizeof(GemmIn) / sizeof(long long));
        for (int i = threadIdx.x; i < n * kWords; i += kThreads) ((long long*)s_in)[i] = ((const long long*)(ins + cb))[i];
        __syncthreads();
        for (int u = 0; u < n;) {
            int v = u + 1;
            while (v < n && same_b(s_in[v], s_in[u])) ++v;
            tile_accumulate_run(s_in + u, v - u, tl.m0, tl.n0, tm, tn, em, en, As, Bs, acc);
            u = v;
        }
        __syncthreads();   // the descriptors are replaced
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (threadIdx.x + q * kThreads < tm * tn) {
            double* cp = o.C + (int64_t)(tl.m0 + em[q]) * o.ldc + tl.n0 + en[q];
            *cp = o.beta == 0.0 ? acc[q] : o.beta * (*cp) + acc[q];
        }
}

// Small outputs (M, N <= 32): one CTA per output, one thread per output
// element, the K loop reading A and B directly, so that no FP64 instruction is
// spent on tile padding.
__global__ void __launch_bounds__(kSmallGemmThreads) k_gemm_small(const GemmOut* __restrict__ outs,
                                                                  const GemmIn* __restrict__ ins,
                                                                  const int* __restrict__ ids) {
    const GemmOut o = outs[ids[blockIdx.x]];
    const int n_el = o.M * o.N;
    for (int e = threadIdx.x; e < n_el; e += kSmallGemmThreads) {
        const int m = e / o.N, n = e % o.N;
        double acc = 0.0;
        for (int c = o.beg; c < o.end; ++c) {
            const GemmIn in = ins[c];
            double part = 0.0;
            if (in.transA)
                part = dev::dot_global<false, false>(in.A + m, in.lda, in.B + n, in.ldb, in.K, 0.0);
            else
                part = dev::dot_global<false, false>(in.A + (int64_t)m * in.lda, 1, in.B + n, in.ldb, in.K, 0.0);
            acc = fma(in.alpha, part, acc);
        }
        double* cp = o.C + (int64_t)m * o.ldc + n;
        *cp = o.beta == 0.0 ? acc : o.beta * (*cp) + acc;
    }
}

// Householder QR, one CTA per matrix; the working set (A, Q, tau) lives in
// shared memory when it fits (smem = 1), else in global memory.  Reflector
// H = I - tau v v^T with v_j = 1, beta = -sign(alpha) ||x||,
// tau = (beta - alpha)/beta, v = x/(alpha - beta).
__global__ void __launch_bounds__(kThreads) k_qr(const QrTask* __restrict__ tasks) {
    extern __shared__ double sm[];
    __shared__ double red[33];
    const QrTask tk = tasks[blockIdx.x];
    const int M = tk.M, N = tk.N, k = M < N ? M : N;
    double* A = tk.smem ? sm : tk.A;
    double* Q = tk.smem ? sm + (int64_t)M * N : tk.Q;
    double* tau = tk.smem ? sm + (int64_t)M * N + (int64_t)M * k : tk.tau;
    double* vd = tau + k;   // the reflectors' diagonals, until Q is formed (in shared memory only)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (tk.smem) {
        for (int64_t e = threadIdx.x; e < (int64_t)M * N; e += kThreads) A[e] = tk.A[e];
        __syncthreads();
        dev::householder(A, tau, vd, M, N);
        dev::form_q(A, tau, vd, Q, M, k);
    } else {
        dev::householder_global(A, tau, M, N, red);
        dev::form_q_global(A, tau, Q, M, k);
    }
    __syncthreads();
    // R (k x N row-major) from the upper trapezoid
    for (int64_t e = threadIdx.x; e < (int64_t)k * N; e += kThreads) {
        const int r = (int)(e / N), c = (int)(e % N);
        tk.R[e] = c >= r ? A[(int64_t)c * M + r] : 0.0;
    }
    __syncthreads();
    // diag(R) >= 0 (R is in global memory; every thread sees the final R after the barrier)
    for (int j = warp; j < k; j += kWarps) {
        const double rjj = A[(int64_t)j * M + j];
        if (rjj < 0.0) {
            for (int c = lane; c < N; c += 32) tk.R[(int64_t)j * N + c] = -tk.R[(int64_t)j * N + c];
            for (int i = lane; i < M; i += 32) Q[(int64_t)j * M + i] = -Q[(int64_t)j * M + i];
        }
    }
    if (tk.smem) {
        __syncthreads();
        for (int64_t e = threadIdx.x; e < (int64_t)M * k; e += kThreads) tk.Q[e] = Q[e];
    }
}

constexpr int kSmemJacobiMax = 110;   // 2 k^2 doubles <= 193 KB of shared memory

// One-sided Jacobi task on a k x k matrix G (column-major, overwritten by the
// rotated columns) with the accumulated rotations in V (column-major).

// One-sided Jacobi (dev::jacobi), one CTA per matrix, in shared memory when k <= kSmemJacobiMax.
__global__ void __launch_bounds__(kThreads) k_jacobi(const JacTask* __restrict__ tasks) {
    extern __shared__ double sm[];
    __shared__ double red[33];
    __shared__ int s_rot;
    const JacTask tk = tasks[blockIdx.x];
    const int k = tk.k;
    double* G = tk.smem ? sm : tk.G;
    double* V = tk.smem ? sm + (int64_t)k * k : tk.V;
    if (tk.smem) {
        for (int64_t e = threadIdx.x; e < (int64_t)k * k; e += kThreads) G[e] = tk.G[e];
        __syncthreads();
    }
    dev::jacobi(G, V, tk.Sraw, k, red, &s_rot);
    if (tk.smem) {
        for (int64_t e = threadIdx.x; e < (int64_t)k * k; e += kThreads) {
            tk.G[e] = G[e];
            tk.V[e] = V[e];
        }
    }
}

// Assemble the SVD of M (M x N) from QR + Jacobi of the triangular factor:
// tall (M >= N): M = Q R, R^T = G, G V = U' S  =>  U = Q V, Vt = U'^T;
// wide (M < N):  M^T = Q R, R^T = G, G V = U' S => U = U', Vt = (Q V)^T.
// QVt = (Q V)^T (k x len, row-major) comes from a grouped GEMM.
struct SvdFin {
    const double* G;
    const double* QVt;
    const double* Sraw;
    double* S;
    double* US;
    double* Vt;
    double* rinv;
    int* perm;
    int M, N, k, len, wide;
};

// kFinSplit CTAs per matrix, a range of its singular triples each: bound by the strided
// copies, which one CTA per matrix left to one SM (k = 200: 230 us).
constexpr int kFinSplit = 16;
__global__ void __launch_bounds__(kThreads) k_svd_finalize(const SvdFin* __restrict__ tasks) {
    const SvdFin tk = tasks[blockIdx.x];
    dev::svd_assemble(tk.G, tk.k, tk.QVt, tk.Sraw, tk.rinv, tk.perm, tk.S, tk.US, tk.Vt, tk.M, tk.N, tk.k, tk.len, tk.wide,
                      tk.k, tk.N, (int)((int64_t)tk.k * blockIdx.y / kFinSplit), (int)((int64_t)tk.k * (blockIdx.y + 1) / kFinSplit));
}

__global__ void __launch_bounds__(kThreads) k_sumsq(const double* const* __restrict__ xs,
                                                    const int64_t* __restrict__ ns,
                                                    double* __restrict__ out) {
    __shared__ double red[33];
    const double* x = xs[blockIdx.x];
    const int64_t n = ns[blockIdx.x];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += kThreads) s += x[i] * x[i];
    s = block_sum(s, red);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
}


// Every kernel of the library prefers the same L1/shared-memory split (maximum
// shared memory), so consecutive launches never wait for the SM to re-partition.
void configure_carveout() {
    static bool done = false;
    if (done) return;
    const int carve = cudaSharedmemCarveoutMaxShared;
    BSM_CUDA(cudaFuncSetAttribute(k_copy, cudaFuncAttributePreferredSharedMemoryCarveout, carve));
    BSM_CUDA(cudaFuncSetAttribute(k_gemm, cudaFuncAttributePreferredSharedMemoryCarveout, carve));
    BSM_CUDA(cudaFuncSetAttribute(k_qr, cudaFuncAttributePreferredSharedMemoryCarveout, carve));
    BSM_CUDA(cudaFuncSetAttribute(k_jacobi, cudaFuncAttributePreferredSharedMemoryCarveout, carve));
    BSM_CUDA(cudaFuncSetAttribute(k_svd_finalize, cudaFuncAttributePreferredSharedMemoryCarveout, carve));
    BSM_CUDA(cudaFuncSetAttribute(k_sumsq, cudaFuncAttributePreferredSharedMemoryCarveout, carve));
    done = true;
}

}  // namespace

void check_launch(Context* ctx) {
    ctx->launches++;
    BSM_CUDA(cudaGetLastError());
}

cudaEvent_t Context::take_event() {
    cudaEvent_t e;
    if (!event_pool.empty()) {
        e = event_pool.back();
        event_pool.pop_back();
    } else {
        BSM_CUDA(cudaEventCreate(&e));
    }
    return e;
}

void Context::prof_begin(cudaEvent_t* e0) {
    *e0 = take_event();
    BSM_CUDA(cudaEventRecord(*e0, stream));
}

void Context::prof_end(int kind, double fl, double by, cudaEvent_t e0, double executed) {
    cudaEvent_t e1 = take_event();
    BSM_CUDA(cudaEventRecord(e1, stream));
    prof.push_back({kind, fl, by, executed < 0.0 ? fl : executed, e0, e1});
}

struct ZeroChunk {
    double* p;
    int64_t n;
};

__global__ void __launch_bounds__(kThreads) k_zero(const ZeroChunk* __restrict__ chunks) {
    const ZeroChunk c = chunks[blockIdx.x];
    for (int64_t e = threadIdx.x; e < c.n; e += kThreads) c.p[e] = 0.0;
}

// Up to kFlatCores cores per launch, their pointers in the kernel's arguments (no task upload).
constexpr int kFlatCores = 120;
struct FlatCores {
    double* core[kFlatCores];
    int64_t beg[kFlatCores + 1];   // offsets in the flat array
    int n;
};

// Entries lo_e .. hi_e of the concatenated cores, entry e at flat[e - flat0].
__global__ void __launch_bounds__(kThreads) k_flat_cores(const FlatCores fc, double* __restrict__ flat, int64_t flat0,
                                                         int64_t lo_e, int64_t hi_e, int to_cores) {
    for (int64_t e = lo_e + (int64_t)blockIdx.x * kThreads + threadIdx.x; e < hi_e;
         e += (int64_t)gridDim.x * kThreads) {
        int lo = 0, hi = fc.n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (fc.beg[mid] <= e) lo = mid;
            else hi = mid - 1;
        }
        double* c = fc.core[lo] + (e - fc.beg[lo]);
        if (to_cores) *c = flat[e - flat0];
        else flat[e - flat0] = *c;
    }
}

void launch_flat_cores(Context* ctx, const std::vector<double*>& core, const std::vector<int64_t>& n, double* flat,
                       int64_t beg, int64_t end, bool to_cores) {
    configure_carveout();
    int64_t off = 0;
    for (size_t t = 0; t < core.size();) {
        FlatCores fc{};
        for (; t < core.size() && fc.n < kFlatCores; ++t) {
            if (n[t] > 0) {
                fc.core[fc.n] = core[t];
                fc.beg[fc.n++] = off;
            }
            off += n[t];
        }
        fc.beg[fc.n] = off;
        if (fc.n == 0) continue;
        const int64_t lo = std::max(beg, fc.beg[0]), hi = std::min(end, off), total = hi - lo;
        if (total <= 0) continue;
        const unsigned ctas = (unsigned)std::min<int64_t>((total + 4 * kThreads - 1) / (4 * kThreads), 1024);
        ProfScope ps(ctx, KK_COPY, 0.0, 16.0 * (double)total);
        k_flat_cores<<<ctas, kThreads, 0, ctx->stream>>>(fc, flat, beg, lo, hi, to_cores ? 1 : 0);
        check_launch(ctx);
        ps.done();
    }
}

void launch_zero(Context* ctx, const std::vector<double*>& ptr, const std::vector<int64_t>& n, int kind) {
    std::vector<ZeroChunk> chunks;
    for (size_t i = 0; i < ptr.size(); ++i)
        for (int64_t b = 0; b < n[i]; b += kCopyChunk) chunks.push_back({ptr[i] + b, std::min(n[i] - b, kCopyChunk)});
    if (chunks.empty()) return;
    configure_carveout();
    Scratch s(ctx);
    const ZeroChunk* d = s.up(chunks);
    ProfScope ps(ctx, kind, 0.0, 8.0 * [&] {
        double t = 0.0;
        for (int64_t v : n) t += (double)v;
        return t;
    }());
    k_zero<<<(unsigned)chunks.size(), kThreads, 0, ctx->stream>>>(d);
    check_launch(ctx);
    ps.done();
}

void launch_copy(Context* ctx, const std::vector<CopyTask>& tasks, int kind) {
    if (tasks.empty()) return;
    configure_carveout();
    std::vector<CopyChunk> chunks;
    for (int i = 0; i < (int)tasks.size(); ++i) {
        const int64_t n = (int64_t)tasks[i].rows * tasks[i].cols;
        for (int64_t b = 0; b < n; b += kCopyChunk) chunks.push_back({i, b, std::min(n, b + kCopyChunk)});
    }
    if (chunks.empty()) return;
    double by = 0.0;
    for (const CopyTask& t : tasks) by += (t.accumulate ? 24.0 : 16.0) * t.rows * (double)t.cols;
    Scratch s(ctx);
    CopyTask* dt = s.up(tasks);
    CopyChunk* dc = s.up(chunks);
    ProfScope ps(ctx, kind, 0.0, by);
    k_copy<<<(unsigned)chunks.size(), kThreads, 0, ctx->stream>>>(dt, dc);
    check_launch(ctx);
    ps.done();
}


namespace {

// The FP64 grouped GEMM with outputs of max(M, N) <= small_max on the
// one-thread-per-entry kernel and the rest on 32 x 32 tiles (small_max <= 32).
void launch_gemm_fp64(Context* ctx, const std::vector<GemmOut>& outs, const std::vector<GemmIn>& ins, int kind,
                      int small_max) {
    configure_carveout();
    std::vector<GemmTile> tiles;
    std::vector<int> small, emulated;
    // fl: of the terms, a product each; ex: what the kernels run for them (k_gemm sums the left factors of a
    // run before it multiplies, once per tile column, and reads the right factor once)
    double fl = 0.0, ex = 0.0, by = 0.0;
    for (int o = 0; o < (int)outs.size(); ++o) {
        const GemmOut& g = outs[o];
        // outputs of at least 2^gemm_emulation_log2 flops with one untransposed
        // contribution (overwritten) go to the tensor-core FP64 emulation; the
        // emulation takes untransposed operands only (the sweeps' large R X and
        // U S X products are untransposed)
        if (ctx->gemm_emulation_log2 > 0 && g.end == g.beg + 1 && g.beta == 0.0 && !ins[g.beg].transA &&
            2.0 * g.M * (double)g.N * ins[g.beg].K >= std::ldexp(1.0, ctx->gemm_emulation_log2)) {
            emulated.push_back(o);
            continue;
        }
        if (std::max(g.M, g.N) <= small_max) {
            if (g.M > 0 && g.N > 0) small.push_back(o);
        } else {
            for (int m0 = 0; m0 < g.M; m0 += kTile)
                for (int n0 = 0; n0 < g.N; n0 += kTile) tiles.push_back({o, m0, n0});
        }
        const bool one_by_one = std::max(g.M, g.N) <= small_max;
        for (int c = g.beg; c < g.end && !ctx->profiling; ++c) fl += 2.0 * g.M * g.N * (double)ins[c].K;
        for (int c = g.beg; c < g.end && ctx->profiling;) {
            const int end = std::min(g.end, c + kGemmIns - (c - g.beg) % kGemmIns);   // descriptors staged together
            int v = c + 1;
            while (!one_by_one && v < end && same_b(ins[v], ins[c])) ++v;
            const double n = v - c, mk = (double)g.M * ins[c].K;
            fl += 2.0 * mk * g.N * n;
            ex += 2.0 * mk * g.N + (n > 1 ? 2.0 * mk * n * ((g.N + kTile - 1) / kTile) : 0.0);
            by += 8.0 * (mk * n + (double)ins[c].K * g.N);
            c = v;
        }
        by += 8.0 * g.M * (double)g.N * (g.beta == 0.0 ? 1.0 : 2.0);
    }
    if (!emulated.empty()) {
        std::vector<OzGemm> og;
        double efl = 0.0;
        for (int o : emulated) {
            const GemmOut& g = outs[o];
            const GemmIn& in = ins[g.beg];
            og.push_back({in.A, in.B, g.C, g.M, g.N, in.K, in.lda, in.ldb, g.ldc, in.alpha});
            efl += 2.0 * g.M * (double)g.N * in.K;
        }
        ProfScope pe(ctx, kind, efl, 0.0);
        launch_gemm_ozaki_group(ctx, og, 8);
        pe.done();
    }
    if (tiles.empty() && small.empty()) return;
    ctx->flops += fl;
    // one staged upload for all task arrays
    std::vector<unsigned char> pack;
    auto add = [&](const void* src, size_t bytes) {
        const size_t off = (pack.size() + 15) & ~size_t(15);
        pack.resize(off + bytes);
        if (bytes) std::memcpy(pack.data() + off, src, bytes);
        return off;
    };
    const size_t oo = add(outs.data(), outs.size() * sizeof(GemmOut));
    const size_t oi = add(ins.data(), ins.size() * sizeof(GemmIn));
    const size_t os = add(small.data(), small.size() * sizeof(int));
    const size_t ot = add(tiles.data(), tiles.size() * sizeof(GemmTile));
    Scratch s(ctx);
    unsigned char* d = s.up(pack);
    const GemmOut* d_o = (const GemmOut*)(d + oo);
    const GemmIn* d_i = (const GemmIn*)(d + oi);
    ProfScope ps(ctx, kind, fl, by);
    ps.executed = ex;
    if (!small.empty()) {
        k_gemm_small<<<(unsigned)small.size(), kSmallGemmThreads, 0, ctx->stream>>>(d_o, d_i, (const int*)(d + os));
        check_launch(ctx);
    }
    if (!tiles.empty()) {
        k_gemm<<<(unsigned)tiles.size(), kThreads, 0, ctx->stream>>>(d_o, d_i, (const GemmTile*)(d + ot));
        check_launch(ctx);
    }
    ps.done();
}

// Size class of a contraction launch for the autotuner: the fractions of
// outputs with max(M, N) <= 8, <= 16, <= 32 (in quarters) and log2 of the flops.
int64_t gemm_size_class(const std::vector<GemmOut>& outs, const std::vector<GemmIn>& ins) {
    int64_t c8 = 0, c16 = 0, c32 = 0;
    double fl = 0.0;
    for (const GemmOut& g : outs) {
        const int mx = std::max(g.M, g.N);
        c8 += mx <= 8;
        c16 += mx <= 16;
        c32 += mx <= 32;
        for (int c = g.beg; c < g.end; ++c) fl += 2.0 * g.M * g.N * (double)ins[c].K;
    }
    const int64_t n = std::max<int64_t>((int64_t)outs.size(), 1);
    const int64_t q8 = 4 * c8 / n, q16 = 4 * c16 / n, q32 = 4 * c32 / n;
    const int64_t lf = fl > 1.0 ? (int64_t)std::log2(fl) : 0;
    return ((q8 * 5 + q16) * 5 + q32) * 64 + std::min<int64_t>(lf, 63);
}

}  // namespace

// The zip-up contraction (kind KK_APPLY) in FP64 is autotuned: the split
// between the one-thread-per-entry kernel and the 32 x 32 tiled kernel
// (small_max in {0, 8, 16, 32}) is chosen per context and size class by timing
// every candidate on the first launch of that class (the contraction overwrites
// its outputs, so the repeats change nothing) and kept for later launches.
void launch_gemm(Context* ctx, const std::vector<GemmOut>& outs, const std::vector<GemmIn>& ins, int kind) {
    if (outs.empty()) return;
    if (kind == KK_APPLY && ctx->apply_precision == BSMPS_PREC_TF32X3 && gemm_tf32x3_eligible(outs, ins)) {
        launch_gemm_tf32x3(ctx, outs, ins, kind);
        return;
    }
    if (kind != KK_APPLY || !ctx->autotune) {
        launch_gemm_fp64(ctx, outs, ins, kind, kTile);
        return;
    }
    for (const GemmOut& g : outs)
        if (g.beta != 0.0) {   // accumulating outputs cannot be repeated
            launch_gemm_fp64(ctx, outs, ins, kind, kTile);
            return;
        }
    const int64_t key = gemm_size_class(outs, ins);
    auto it = ctx->gemm_tuned.find(key);
    if (it != ctx->gemm_tuned.end() || ctx->rec) {
        // a graph being recorded takes the tuned split (its sizing run tuned every
        // class) and never times candidates
        launch_gemm_fp64(ctx, outs, ins, kind, it != ctx->gemm_tuned.end() ? it->second : kTile);
        return;
    }
    const int cand[4] = {0, 8, 16, 32};
    float best_ms = 0.0f;
    int best = kTile;
    const bool prof = ctx->profiling;
    ctx->profiling = false;   // tuning launches are not part of the profile
    cudaEvent_t e0 = ctx->take_event(), e1 = ctx->take_event();
    for (int c : cand) {
        BSM_CUDA(cudaEventRecord(e0, ctx->stream));
        launch_gemm_fp64(ctx, outs, ins, kind, c);
        BSM_CUDA(cudaEventRecord(e1, ctx->stream));
        BSM_CUDA(cudaEventSynchronize(e1));
        float ms = 0.0f;
        BSM_CUDA(cudaEventElapsedTime(&ms, e0, e1));
        if (c == cand[0] || ms < best_ms) {
            best_ms = ms;
            best = c;
        }
    }
    ctx->event_pool.push_back(e0);
    ctx->event_pool.push_back(e1);
    ctx->profiling = prof;
    ctx->gemm_tuned[key] = best;
    // the launch that counts (and is profiled)
    launch_gemm_fp64(ctx, outs, ins, kind, best);
}

constexpr size_t kSmemBudget = 220 * 1024;

void launch_qr(Context* ctx, const std::vector<QrTask>& tasks_in, int kind) {
    if (tasks_in.empty()) return;
    configure_carveout();
    double fl = 0.0, by = 0.0;
    std::vector<QrTask> small, large, clustered;
    size_t smem_max = 0;
    for (QrTask t : tasks_in) {
        if (qr_cluster_eligible(t.M, t.N)) {
            const double m = t.M, n = t.N, k = std::min(m, n);
            fl += 2.0 * m * n * k - (m + n) * k * k + 2.0 / 3.0 * k * k * k + 2.0 * m * k * k - 2.0 / 3.0 * k * k * k;
            by += 8.0 * (m * n + m * k + k * n);
            clustered.push_back(t);
            continue;
        }
        const double m = t.M, n = t.N, k = std::min(m, n);
        fl += 2.0 * m * n * k - (m + n) * k * k + 2.0 / 3.0 * k * k * k;   // factorisation
        fl += 2.0 * m * k * k - 2.0 / 3.0 * k * k * k;                     // forming Q
        by += 8.0 * (m * n + m * k + k * n);
        const size_t need = sizeof(double) * ((size_t)t.M * t.N + (size_t)t.M * std::min(t.M, t.N) +
                                              (size_t)std::min(t.M, t.N));
        if (need <= kSmemBudget) {
            t.smem = 1;
            small.push_back(t);
            smem_max = std::max(smem_max, need + sizeof(double) * (size_t)std::min(t.M, t.N));
        } else {
            t.smem = 0;
            large.push_back(t);
        }
    }
    ctx->flops += fl;
    Scratch s(ctx);
    ProfScope ps(ctx, kind, fl, by);
    bool cluster_ran = false;
    if (!clustered.empty()) {
        cluster_ran = launch_qr_cluster(ctx, clustered, kind == KK_APPLY_QR);
        if (!cluster_ran) {
            for (QrTask t : clustered) {   // no cluster could be scheduled: one CTA per matrix
                const size_t need = sizeof(double) * ((size_t)t.M * t.N + (size_t)t.M * std::min(t.M, t.N) +
                                                      (size_t)std::min(t.M, t.N));
                t.smem = need <= kSmemBudget ? 1 : 0;
                if (t.smem) smem_max = std::max(smem_max, need + sizeof(double) * (size_t)std::min(t.M, t.N));
                (t.smem ? small : large).push_back(t);
            }
        }
    }
    // the one-CTA QRs overlap the cluster QRs on the context's second stream:
    // their task lists are uploaded first, the fork follows, the join precedes
    // the release of s
    QrTask* d_small = small.empty() ? nullptr : s.up(small);
    QrTask* d_large = large.empty() ? nullptr : s.up(large);
    const bool overlap = cluster_ran && (d_small || d_large) && !ctx->profiling && !ctx->rec && !ctx->side_open;
    SideJoin guard(overlap ? ctx : nullptr);   // after s: joins before s releases the task lists
    const cudaStream_t st = overlap ? ctx->fork_side() : ctx->stream;
    if (d_small) {
        BSM_CUDA(cudaFuncSetAttribute(k_qr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max));
        k_qr<<<(unsigned)small.size(), kThreads, smem_max, st>>>(d_small);
        check_launch(ctx);
    }
    if (d_large) {
        k_qr<<<(unsigned)large.size(), kThreads, 0, st>>>(d_large);
        check_launch(ctx);
    }
    if (overlap) ctx->join_side();
    ps.done();
}

void launch_svd(Context* ctx, const std::vector<SvdTask>& tasks) {
    if (tasks.empty()) return;
    configure_carveout();
    Scratch s(ctx);
    // 1. Householder QR of M (tall) or M^T (wide): Q is len x k, R is k x k
    std::vector<QrTask> qr;
    std::vector<double*> Q(tasks.size()), R(tasks.size()), V(tasks.size()), Sraw(tasks.size()), QVt(tasks.size());
    std::vector<int*> perm(tasks.size());
    for (size_t i = 0; i < tasks.size(); ++i) {
        const SvdTask& t = tasks[i];
        const int k = std::min(t.M, t.N), len = std::max(t.M, t.N);
        Q[i] = s.dbl((size_t)len * k);
        R[i] = s.dbl((size_t)k * k);
        V[i] = s.dbl((size_t)k * k);
        Sraw[i] = s.dbl((size_t)k);
        QVt[i] = s.dbl((size_t)k * len);
        perm[i] = (int*)ctx->alloc(sizeof(int) * (size_t)k);
        s.ptrs.push_back(perm[i]);
        qr.push_back({t.G, Q[i], R[i], s.dbl((size_t)k), t.wide ? t.N : t.M, t.wide ? t.M : t.N});
    }
    launch_qr(ctx, qr);
    // 2. one-sided Jacobi on G = R^T (the row-major R is G column-major): one
    // thread-block cluster per matrix for kClusterJacobiMin <= k <= kClusterJacobiMax
    // (the FP64 units of several SMs on one matrix); one CTA in shared memory for
    // smaller k (and for k <= kSmemJacobiMax when no cluster can be scheduled);
    // beyond, across the grid (one CTA per matrix when the cooperative launch
    // cannot be resident)
    std::vector<JacTask> small, mid, large;
    std::vector<size_t> mid_i;
    double fl = 0.0, by = 0.0;
    for (size_t i = 0; i < tasks.size(); ++i) {
        const int k = std::min(tasks[i].M, tasks[i].N);
        JacTask jt{R[i], V[i], Sraw[i], k, 0};
        if (k >= kClusterJacobiMin && k <= kClusterJacobiMax) {
            mid.push_back(jt);
            mid_i.push_back(i);
        } else if (k <= kSmemJacobiMax)
            small.push_back(jt);
        else
            large.push_back(jt);
        fl += 54.0 * (double)k * k * k;   // nominal: 6 sweeps of k^2/2 pairs x 18k flops
        by += 8.0 * 3.0 * k * (double)k;
    }
    ctx->flops += fl;
    // 2a. FP32 preconditioning of the cluster tasks with k >= jacobi_precond_min:
    // P = the rotations of an FP32 one-sided Jacobi of G (orthogonal to ~1e-6),
    // Qp = the Q factor of P (FP64 Householder, orthogonal to FP64 rounding,
    // diag R >= 0 keeps it next to P), G <- G Qp.  The FP64 Jacobi below then
    // starts from nearly orthogonal columns and converges in a few sweeps
    // (quadratically), and V <- Qp V afterwards: G Qp V = U S exactly as before,
    // with every step that decides the result in FP64.
    struct Pre {
        size_t m;          // index in mid
        double *Qp, *V1;
    };
    std::vector<Pre> pre;
    if (ctx->jacobi_precond_min > 0 && !mid.empty()) {
        const double fl0 = ctx->flops;   // the preconditioner's work is not algorithmic work of the SVD
        std::vector<JacTask> pj;
        std::vector<double*> P;
        double pb = 0.0;
        for (size_t m = 0; m < mid.size(); ++m) {
            const int k = mid[m].k;
            if (k < ctx->jacobi_precond_min) continue;
            P.push_back(s.dbl((size_t)k * k));
            pj.push_back({mid[m].G, P.back(), nullptr, k, 0});
            pre.push_back({m, s.dbl((size_t)k * k), s.dbl((size_t)k * k)});
            pb += 16.0 * k * (double)k;
        }
        bool ok = pj.empty();
        if (!ok) {
            ProfScope ps(ctx, KK_SVD, 0.0, pb);
            ok = launch_jacobi_cluster_f32(ctx, pj);
            ps.done();
        }
        if (ok && !pre.empty()) {
            std::vector<QrTask> pq;
            for (size_t j = 0; j < pre.size(); ++j) {
                const int k = pj[j].k;
                pq.push_back({P[j], pre[j].Qp, s.dbl((size_t)k * k), s.dbl((size_t)k), k, k});
            }
            launch_qr(ctx, pq, KK_SVD);
            // G1 = G Qp (column-major): G1^T = Qp^T G^T, the buffers read row-major
            std::vector<GemmOut> go;
            std::vector<GemmIn> gi;
            for (Pre& pr : pre) {
                JacTask& jt = mid[pr.m];
                double* G1 = s.dbl((size_t)jt.k * jt.k);
                go.push_back({G1, jt.k, jt.k, jt.k, (int)gi.size(), (int)gi.size() + 1, 0.0});
                gi.push_back({pr.Qp, jt.G, jt.k, jt.k, jt.k, 0, 1.0});
                jt.G = G1;
                R[mid_i[pr.m]] = G1;   // the rotated G that step 4 reads
                // the cluster Jacobi rotates Qp's columns: V = Qp V1 without a product
                jt.V = pr.Qp;
                jt.v_given = 1;
            }
            launch_gemm(ctx, go, gi, KK_SVD);
        } else {
            pre.clear();
        }
        ctx->flops = fl0;
    }
    {
        ProfScope ps(ctx, KK_SVD, fl, by);
        if (!mid.empty() && launch_jacobi_cluster(ctx, mid)) {
            for (const Pre& pr : pre) V[mid_i[pr.m]] = pr.Qp;   // Qp V1, in place
            pre.clear();
        } else if (!mid.empty()) {
            // one CTA per matrix: those kernels start from the identity, so the
            // preconditioned tasks accumulate V1 and V = Qp V1 follows below
            for (size_t m = 0; m < mid.size(); ++m) mid[m].v_given = 0;
            for (const Pre& pr : pre) mid[pr.m].V = pr.V1;
            for (const JacTask& t : mid) (t.k <= kSmemJacobiMax ? small : large).push_back(t);
        }
        if (!small.empty()) {
            int kmax_small = 1;
            for (JacTask& t : small) {
                t.smem = 1;
                kmax_small = std::max(kmax_small, t.k);
            }
            JacTask* d = s.up(small);
            const size_t smem = sizeof(double) * 2 * (size_t)kmax_small * kmax_small;
            BSM_CUDA(cudaFuncSetAttribute(k_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_jacobi<<<(unsigned)small.size(), kThreads, smem, ctx->stream>>>(d);
            check_launch(ctx);
        }
        if (!large.empty() && !launch_jacobi_grid(ctx, large)) {
            JacTask* d = s.up(large);
            k_jacobi<<<(unsigned)large.size(), kThreads, 0, ctx->stream>>>(d);
            check_launch(ctx);
        }
        ps.done();
    }
    if (!pre.empty()) {
        // V = Qp V1 (column-major): V^T = V1^T Qp^T
        const double fl0 = ctx->flops;
        std::vector<GemmOut> go;
        std::vector<GemmIn> gi;
        for (const Pre& pr : pre) {
            const int k = mid[pr.m].k;
            go.push_back({V[mid_i[pr.m]], k, k, k, (int)gi.size(), (int)gi.size() + 1, 0.0});
            gi.push_back({pr.V1, pr.Qp, k, k, k, 0, 1.0});
        }
        launch_gemm(ctx, go, gi, KK_SVD);
        ctx->flops = fl0;
    }
    // 3. (Q V)^T = V^T Q^T: A = V column-major read as V^T row-major, B = Q column-major = Q^T row-major
    std::vector<GemmOut> outs;
    std::vector<GemmIn> ins;
    for (size_t i = 0; i < tasks.size(); ++i) {
        const int k = std::min(tasks[i].M, tasks[i].N), len = std::max(tasks[i].M, tasks[i].N);
        outs.push_back({QVt[i], k, len, len, (int)ins.size(), (int)ins.size() + 1, 0.0});
        ins.push_back({V[i], Q[i], k, k, len, 0, 1.0});
    }
    launch_gemm(ctx, outs, ins);
    // 4. sort, assemble U S and V^T, sign convention
    std::vector<SvdFin> fin;
    double fb = 0.0;
    for (size_t i = 0; i < tasks.size(); ++i) {
        const SvdTask& t = tasks[i];
        const int k = std::min(t.M, t.N), len = std::max(t.M, t.N);
        fin.push_back({R[i], QVt[i], Sraw[i], t.S, t.US, t.Vt, s.dbl((size_t)k), perm[i], t.M, t.N, k, len, t.wide});
        fb += 8.0 * ((double)t.M * k + (double)k * t.N + 2.0 * k * (double)len);
    }
    SvdFin* d = s.up(fin);
    ProfScope ps(ctx, KK_SVD, 0.0, fb);
    k_svd_finalize<<<dim3((unsigned)fin.size(), kFinSplit), kThreads, 0, ctx->stream>>>(d);
    check_launch(ctx);
    ps.done();
}

void launch_sumsq(Context* ctx, const std::vector<const double*>& xs, const std::vector<int64_t>& ns,
                  double* out_dev) {
    if (xs.empty()) return;
    configure_carveout();
    Scratch s(ctx);
    const double** d_x = s.up(xs);
    int64_t* d_n = s.up(ns);
    double by = 0.0;
    for (int64_t n : ns) by += 8.0 * n;
    ProfScope ps(ctx, KK_SUMSQ, 2.0 * by / 8.0, by);
    k_sumsq<<<(unsigned)xs.size(), kThreads, 0, ctx->stream>>>(d_x, d_n, out_dev);
    check_launch(ctx);
    ps.done();
}

}  // namespace bsm
