// lanczos.cu -- g ~ M^{1/2} W by the Lanczos (Krylov) method of Sec. II.C, on the device.
//
// Iteration k (0-based), all float64:
//   w = M v_k                                   (pair kernels, context precision)
//   c = V_{0..k}^T w ;  w -= V c                (classical Gram-Schmidt, pass 1; c_k = alpha_k)
//   c' = V_{0..k}^T w ; w -= V c'               (pass 2: full reorthogonalisation)
//   alpha_k = c_k + c'_k ;  beta_k = |w| ;  v_{k+1} = w / beta_k
//   T_{k+1} = tridiag(beta, alpha, beta);  y_k = |W| T_{k+1}^{1/2} e_1 ;  g_k = V_{0..k} y_k
//   eps_k = |y_k - (y_{k-1}, 0)| / |y_{k-1}|  (equals |g_k - g_{k-1}| / |g_{k-1}| while V stays
//   orthonormal, which the reorthogonalisation maintains), first defined at k = 1.
// The first subtraction of pass 1 already removes alpha_k v_k and beta_{k-1} v_{k-1}, i.e. the
// three-term recurrence is a subset of the reorthogonalisation.
//
// What bounds it: for a small suspension the chain of launches, reductions and float64 latencies of
// an iteration, so everything after the product is one kernel: a thread-block cluster holds w in
// registers, exchanges the partial dot products through distributed shared memory, scales v_{k+1},
// writes it into the packed sources of the next product (whose positions stay packed), and its first
// block does the tridiagonal step.  Separate kernels for the two projections, their dot products, the
// scaling, the packing and the tridiagonal step were seven launches, about 25 us of an iteration at 256
// spheres; 20 steps of 256 spheres in float64 went from 13.7 to 8.4 ms, a step of 4096 in float32 from 960 to
// 845 us.  Larger suspensions spread the same steps over the GPU (gs.cuh).
// Reductions are summed in a fixed order: results do not depend on scheduling.  The stopping decision
// is written to pinned host memory, or, inside a graph-replayed run, taken on the device: the
// iterations after the first are the body of a loop node that each iteration keeps running or ends.
#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <mutex>

#include "gs.cuh"
#include "pair_math.cuh"

namespace rpb {

namespace cg = cooperative_groups;

constexpr int kBlasThreads = 256;

// Spheres of a chunk in the kernels for larger suspensions: small enough to fill the GPU, at most
// 256 partial sums per dot product up to 65536 spheres.
static int64_t gs_chunk(int64_t N)
{
    return N > 32768 ? 256 : (N > 12288 ? 128 : 64);
}

size_t lanczos_red_elems(int64_t max_N, int max_iter)
{
    // partials of the dot products of both passes and of a norm: 12288/64, 32768/128 or N/256 chunks
    return (size_t)(2 * max_iter + 1) * (size_t)std::max<int64_t>(256, (max_N + 255) / 256);
}

size_t lanczos_state_elems(int max_iter)
{
    return LzLayout(max_iter).total + 2 * kSqrtNodes;  // the state block, then the square root's nodes
}

int upload_sqrt_nodes(double *nodes, cudaStream_t st)
{
    static const SqrtNodes host = sqrt_nodes();  // shifts, then weights
    static_assert(sizeof(host) == 2 * kSqrtNodes * sizeof(double), "contiguous");
    return cuda_fail(cudaMemcpyAsync(nodes, &host, sizeof(host), cudaMemcpyHostToDevice, st), "square root nodes");
}

int lanczos_upload(double *lz, int max_iter, cudaStream_t st)
{
    return upload_sqrt_nodes(lz + LzLayout(max_iter).total, st);
}

static int blas_grid(int64_t n, int num_sms)
{
    int64_t g = (n + kBlasThreads - 1) / kBlasThreads;
    const int64_t cap = 2 * (int64_t)num_sms;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

// What the kernels of an iteration work on.
struct GsArgs {
    double *V;         // Krylov basis, rows of ld
    size_t ld;
    int64_t N;
    double *w;         // the product M v_k (with the preconditioner, before its second scaling)
    const double *W;   // initialisation: the vector whose square root product is wanted
    double *vf;        // the load of the next product: v_{k+1}, times P with the preconditioner
    const double *P;   // preconditioner (or null)
    const double *sc;  // s_i (SelfCoefs), for the packed sources
    void *src;         // packed sources whose loads the next product reads (null: it packs itself)
    int fp64;
    double *lz;
    LzLayout L;
    double *red, *red2, *norm2;  // partials (larger suspensions)
    double tol;
    int k, max_iter;
    double *hs;        // pinned host copy of the status words (null: none)
    RunState *rs;      // graph-replayed run: k and the loop's state live here
    cudaGraphConditionalHandle loop;
    __device__ __forceinline__ int iter() const { return rs ? rs->k : k; }
    // s_i of row r's sphere (r = c N + i)
    __device__ __forceinline__ double factor(int64_t r) const
    {
        return src ? sc[r < N ? r : (r < 2 * N ? r - N : r - 2 * N)] : 0.0;
    }
    // v_{k+1} (row r, s_i = si) into the basis and the next product's load
    __device__ __forceinline__ void store(double *v, int64_t r, double x, double si) const
    {
        v[r] = x;
        const double f = P ? x * P[r] : x;
        vf[r] = f;
        if (!src) return;
        const int c = r < N ? 0 : (r < 2 * N ? 1 : 2);
        const int64_t i = r - c * N;
        const double s = si * f;
        if (fp64)
            reinterpret_cast<double *>((SrcF64 *)src + i)[3 + c] = s;
        else
            reinterpret_cast<float *>((SrcF32 *)src + i)[5 + c] = (float)s;
    }
    // status words of a new Krylov space, |W|^2 = s
    __device__ __forceinline__ void begin(double s) const
    {
        double *status = lz + L.status;
        const double nw = sqrt(s);
        status[ST_NW] = nw;
        status[ST_INV_NW] = nw > 0.0 ? 1.0 / nw : 0.0;
        status[ST_EPS] = -1.0;
        status[ST_STOP] = 0.0;
        status[ST_BREAK] = 0.0;
        if (rs) rs->k = 0;
    }
    // after the tridiagonal step of iteration k, by one thread
    __device__ __forceinline__ void end(int k, double beta_k, const TailResult &r, double nW) const
    {
        const bool stop = lanczos_tail_stop(lz, L, k, tol, beta_k, r, nW, hs);
        if (rs) {
            rs->m = k + 1;
            rs->k = k + 1;
            if (k > 0) atomicAdd(&rs->loops, 1ull);
            if (max_iter > 1) cudaGraphSetConditional(loop, !stop && k + 1 < max_iter ? 1u : 0u);
        }
    }
};
// record layout that GsArgs::store writes into: floats 5 .. 7 of SrcF32, doubles 3 .. 5 of SrcF64 hold s F
static_assert(sizeof(SrcF32) == 48 && sizeof(SrcF64) == 80, "packed source records");

// ------------------------------------------------------------------ small suspensions: one cluster
constexpr int kGsCluster = 16;  // blocks of the cluster at most (8 where the device schedules no 16)

constexpr int kGsClusterThreads = kGsThreads + kTailThreads;

// Exchange of the cluster: every block writes its partial sums into all blocks' arrays before the barrier, so
// that the sums read their own shared memory (a read of another block's costs about 600 cycles).
struct ClusterShared {
    double part[2][kGsCluster][kMaxIter];  // dot products of the two passes, by block
    double norm[kGsCluster];
    double coef[kMaxIter];
    double alpha[2];                       // the last vector's coefficients: alpha_k is their sum
};

// coef_j = sum over the cluster's blocks of part[block][j], four threads per j; ends with a barrier of the rows'
// threads
__device__ __forceinline__ void cluster_coefs(const double (*part)[kMaxIter], int blocks, int nvec, double *coef)
{
    const int j = threadIdx.x >> 2, q = threadIdx.x & 3;
    double s = 0.0;
    if (j < nvec)
        for (int r = q; r < blocks; r += 4) s += part[r][j];
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (q == 0 && j < nvec) coef[j] = s;
    gs_sync();
}

// One cluster, block r holding spheres [r per, (r + 1) per): Gram-Schmidt on w and v_{k+1} by the first
// kGsThreads threads of every block; the tridiagonal step by the other kTailThreads of the first block, which
// have loaded its state before alpha_k is known and run beside the second projection, the norm and the
// stores (T has no beta_k): 15.9 -> 13.7 us a launch at 256 spheres, of which the tridiagonal step was about 5.
// init: v_0 = W / |W| instead.
// Every thread of the cluster arrives at its four barriers (two when init) and waits for each; warps are
// converged at all of them.
__global__ void __launch_bounds__(kGsClusterThreads) gs_cluster_kernel(GsArgs A, int per, int init)
{
    static_assert(kGsThreads >= 4 * kMaxIter, "four threads per coefficient");
    __shared__ double sh[kGsWarps][kMaxIter + 8];
    __shared__ ClusterShared cs;
    __shared__ TailShared ts;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), blocks = (int)cl.num_blocks(), tid = threadIdx.x;
    cl.sync();  // every block of the cluster runs: its shared memory may be written
    wait_for_before();
    const int k = init ? -1 : A.iter();
    if (tid >= kGsThreads) {
        const int t = tid - kGsThreads;
        TailRegs reg = {};
        if (rank == 0 && !init) reg = lanczos_tail_load(A.lz, A.L, k, A.lz + A.L.total, ts, t);
        if (!init) {
            cl.sync();
            cl.sync();
        }
        cl.barrier_arrive();
        TailResult r = {};
        if (rank == 0 && !init) {
            asm volatile("bar.sync 3, %0;" ::"n"(kGsClusterThreads) : "memory");  // alpha is there
            r = lanczos_tail_y(A.lz, A.L, k, cs.alpha[0] + cs.alpha[1], reg, ts, t);
        }
        __syncwarp();
        cl.barrier_wait();
        if (rank == 0 && t == 0) {
            double bn = 0.0, nb, inv;
            for (int q = 0; q < blocks; ++q) bn += cs.norm[q];
            root_and_inverse(bn, &nb, &inv);
            if (init)
                A.begin(bn);
            else
                A.end(k, nb, r, reg.nW);
        }
        return;
    }
    const int first = rank * per;
    const int left = (int)A.N - first;
    int64_t row[kGsRows];
    double x[kGsRows], si[kGsRows];
    const GsSpan span = {first, A.N, max(0, min(per, left))};
    const int nu = gs_rows(span, row), nw = gs_warps(span);
#pragma unroll
    for (int u = 0; u < kGsRows; ++u) {
        x[u] = row[u] < 0 ? 0.0 : (init ? A.W[row[u]] : A.w[row[u]]);
        si[u] = row[u] < 0 ? 0.0 : A.factor(row[u]);
        if (A.P && !init && row[u] >= 0) x[u] *= A.P[row[u]];
    }
    for (int pass = 0; pass < 2 && !init; ++pass) {
        const double s = gs_dots(A.V, A.ld, k + 1, row, nu, nw, x, sh);
        if (tid <= k)
            for (int q = 0; q < blocks; ++q) cl.map_shared_rank(&cs, q)->part[pass][rank][tid] = s;
        __syncwarp();
        cl.sync();
        cluster_coefs(cs.part[pass], blocks, k + 1, cs.coef);
        if (rank == 0) {
            if (tid == k) cs.alpha[pass] = cs.coef[k];
            __syncwarp();
            if (pass == 1) asm volatile("bar.arrive 3, %0;" ::"n"(kGsClusterThreads) : "memory");
        }
        gs_project(A.V, A.ld, k + 1, row, nu, cs.coef, x);
    }
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < kGsRows; ++u) s = fma(x[u], x[u], s);
    s = gs_block_sum(s, nu, nw, sh[0]);
    if (tid < blocks) cl.map_shared_rank(&cs, tid)->norm[rank] = s;  // (the sum is in the first warp's threads)
    __syncwarp();
    cl.sync();
    double bn = 0.0, nb, inv;
    for (int q = 0; q < blocks; ++q) bn += cs.norm[q];
    root_and_inverse(bn, &nb, &inv);
    if (init && !(bn > 0.0)) inv = 0.0;
    double *v = A.V + (size_t)(k + 1) * A.ld;
#pragma unroll
    for (int u = 0; u < kGsRows; ++u)
        if (row[u] >= 0) A.store(v, row[u], x[u] * inv, si[u]);
}

// ------------------------------------------------------------------ larger suspensions: chunks over the GPU
__device__ __forceinline__ GsSpan gs_chunk_span(const GsArgs &A, int chunk)
{
    const int64_t first = (int64_t)blockIdx.x * chunk;
    return GsSpan{first, A.N, (int)min((int64_t)chunk, A.N - first)};
}

// partials of <V_j, w>, j <= k (w scaled by the preconditioner first)
__global__ void __launch_bounds__(kGsThreads) gs_dots_kernel(GsArgs A, int chunk)
{
    __shared__ double sh[kGsWarps][kMaxIter + 8];
    const int k = A.iter();
    int64_t row[kGsRows];
    double x[kGsRows];
    const GsSpan span = gs_chunk_span(A, chunk);
    const int nu = gs_rows(span, row), nw = gs_warps(span);
#pragma unroll
    for (int u = 0; u < kGsRows; ++u) {
        x[u] = row[u] >= 0 ? A.w[row[u]] : 0.0;
        if (A.P && row[u] >= 0) A.w[row[u]] = x[u] *= A.P[row[u]];
    }
    const double s = gs_dots(A.V, A.ld, k + 1, row, nu, nw, x, sh);
    if (threadIdx.x <= k) A.red[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = s;
}

// w -= V c; pass 0: then the dot products of pass 2; pass 1: then the partials of |w|^2
__global__ void __launch_bounds__(kGsThreads) gs_project_kernel(GsArgs A, int chunk, int pass)
{
    __shared__ double sh[kGsWarps][kMaxIter + 8];
    __shared__ double coef[kMaxIter];
    const int k = A.iter(), tid = threadIdx.x;
    int64_t row[kGsRows];
    double x[kGsRows];
    const GsSpan span = gs_chunk_span(A, chunk);
    const int nu = gs_rows(span, row), nw = gs_warps(span);
#pragma unroll
    for (int u = 0; u < kGsRows; ++u) x[u] = row[u] >= 0 ? A.w[row[u]] : 0.0;
    gs_coefs(pass ? A.red2 : A.red, gridDim.x, gridDim.x, k + 1, coef);
    if (blockIdx.x == 0 && tid <= k) A.lz[(pass ? A.L.c2 : A.L.c1) + tid] = coef[tid];
    gs_project(A.V, A.ld, k + 1, row, nu, coef, x);
#pragma unroll
    for (int u = 0; u < kGsRows; ++u)
        if (row[u] >= 0) A.w[row[u]] = x[u];
    if (pass == 0) {
        const double s = gs_dots(A.V, A.ld, k + 1, row, nu, nw, x, sh);
        if (tid <= k) A.red2[(size_t)tid * gridDim.x + blockIdx.x] = s;
    } else {
        double s = 0.0;
#pragma unroll
        for (int u = 0; u < kGsRows; ++u) s = fma(x[u], x[u], s);
        s = gs_block_sum(s, nu, nw, sh[0]);
        if (tid == 0) A.norm2[blockIdx.x] = s;
    }
}

// partials of |W|^2
__global__ void __launch_bounds__(kGsThreads) gs_norm_kernel(GsArgs A, int chunk)
{
    __shared__ double sh[kGsWarps];
    int64_t row[kGsRows];
    const GsSpan span = gs_chunk_span(A, chunk);
    const int nu = gs_rows(span, row), nw = gs_warps(span);
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < kGsRows; ++u)
        if (row[u] >= 0) s = fma(A.W[row[u]], A.W[row[u]], s);
    s = gs_block_sum(s, nu, nw, sh);
    if (threadIdx.x == 0) A.norm2[blockIdx.x] = s;
}

// v_{k+1} = w / |w| (init: v_0 = W / |W|)
__global__ void __launch_bounds__(kGsThreads) gs_scale_kernel(GsArgs A, int chunk, int init)
{
    __shared__ double bn;
    gs_coefs(A.norm2, 0, gridDim.x, 1, &bn);
    double nb, inv;
    root_and_inverse(bn, &nb, &inv);
    if (init && !(bn > 0.0)) inv = 0.0;
    const int k = init ? -1 : A.iter();
    int64_t row[kGsRows];
    gs_rows(gs_chunk_span(A, chunk), row);
    double *v = A.V + (size_t)(k + 1) * A.ld;
    const double *w = init ? A.W : A.w;
#pragma unroll
    for (int u = 0; u < kGsRows; ++u)
        if (row[u] >= 0) A.store(v, row[u], w[row[u]] * inv, A.factor(row[u]));
    if (init && blockIdx.x == 0 && threadIdx.x == 0) A.begin(bn);
}

__global__ void __launch_bounds__(kTailThreads) lanczos_tail_kernel(GsArgs A, int parts)
{
    __shared__ TailShared ts;
    const int k = A.iter();
    double bn = 0.0;  // the same in every warp
    for (int b = threadIdx.x & 31; b < parts; b += 32) bn += A.norm2[b];
    for (int o = 16; o > 0; o >>= 1) bn += __shfl_xor_sync(0xffffffffu, bn, o);
    const TailRegs reg = lanczos_tail_load(A.lz, A.L, k, A.lz + A.L.total, ts, threadIdx.x);
    const TailResult r = lanczos_tail_y(A.lz, A.L, k, A.lz[A.L.c1 + k] + A.lz[A.L.c2 + k], reg, ts, threadIdx.x);
    if (threadIdx.x == 0) A.end(k, sqrt(bn), r, reg.nW);
}

// g[r] = sum_{k < m} y[k] V[k][r]   (y already carries |W|); d_m (optional): read m from the device
__global__ void combine_kernel(const double *__restrict__ V, size_t ld, int64_t n, int m, const double *__restrict__ y,
                               double *__restrict__ g, const int *__restrict__ d_m)
{
    __shared__ double ys[kMaxIter];
    if (d_m) m = *d_m;
    for (int k = threadIdx.x; k < m; k += blockDim.x) ys[k] = y[k];
    __syncthreads();
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int k = 0; k < m; ++k) acc = fma(ys[k], V[(size_t)k * ld + r], acc);
        g[r] = acc;
    }
}

// Block-diagonal preconditioner (Sec. II.C reports trying it: each particle's self mobility, with
// its wall interaction, and no interactions between particles).  The translation self block of the
// wall-corrected, regularised mobility is diagonal, s_i^2 / (8 pi eta) (mu_par, mu_par, mu_perp) at
// the clamped height, so P = D^{-1/2} is a vector; P = 0 where D = 0 (spheres on or below the wall
// have no mobility).  Free space: D = mu0.
__global__ void precond_diag_kernel(const double *__restrict__ pos, int64_t N, PairConsts<double> c, double a,
                                    double scale, int wall, double *__restrict__ P)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const double z = pos[2 * N + i];
        double ux = 0.0, uy = 0.0, uz = 0.0;
        double k = scale;
        if (wall) {
            const double si = H0(z / a);
            k *= si * si;
            self_velocity<false, true>(fmax(z, a), 1.0, 1.0, 1.0, 0.0, 0.0, c, ux, uy, uz);
        } else {
            self_velocity<false, false>(z, 1.0, 1.0, 1.0, 0.0, 0.0, c, ux, uy, uz);
        }
        const double dx = k * ux, dz = k * uz;
        P[i] = dx > 0.0 ? 1.0 / sqrt(dx) : 0.0;
        P[N + i] = P[i];
        P[2 * N + i] = dz > 0.0 ? 1.0 / sqrt(dz) : 0.0;
    }
}

// out = x P (inverse: x / P, and 0 where P = 0), elementwise over 3N
// (x and out may be the same vector: no __restrict__ on them)
__global__ void precond_scale_kernel(const double *x, const double *__restrict__ P, int64_t n, int inverse,
                                     double *out)
{
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        const double p = P[r];
        out[r] = inverse ? (p > 0.0 ? x[r] / p : 0.0) : x[r] * p;
    }
}

int lanczos_precond_prepare(rpb_ctx *ctx, int64_t N, const double *pos)
{
    if (!ctx->precond) return RPB_OK;
    const double a = ctx->p.a;
    precond_diag_kernel<<<blas_grid(N, ctx->num_sms), kBlasThreads, 0, ctx->stream>>>(
        pos, N, make_consts<double>(a), a, 1.0 / (8.0 * kPi * ctx->p.eta), ctx->p.wall, ctx->ws.pc);
    count_launches(1);
    return cuda_fail(cudaGetLastError(), "preconditioner");
}

static int precond_scale(rpb_ctx *ctx, int64_t N, const double *x, double *out, bool inverse)
{
    precond_scale_kernel<<<blas_grid(3 * N, ctx->num_sms), kBlasThreads, 0, ctx->stream>>>(x, ctx->ws.pc, 3 * N,
                                                                                         inverse ? 1 : 0, out);
    count_launches(1);
    return cuda_fail(cudaGetLastError(), "preconditioner scale");
}

// Blocks of the cluster that the device can schedule: 16 (beyond the portable 8) where it offers them,
// asked once per device.
static int query_cluster()
{
    int n = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kGsCluster);
    cfg.blockDim = dim3(kGsClusterThreads);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kGsCluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(gs_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, gs_cluster_kernel, &cfg) == cudaSuccess && n >= 1)
        return kGsCluster;
    cudaGetLastError();
    return 8;
}

int lanczos_setup(rpb_ctx *ctx)
{
    static std::mutex mu;
    static int blocks[64] = {};  // per device ordinal, 0: not asked yet
    std::lock_guard<std::mutex> lock(mu);
    if (ctx->device < 0 || ctx->device >= 64) {
        ctx->gs_cluster = query_cluster();
        return RPB_OK;
    }
    if (!blocks[ctx->device]) blocks[ctx->device] = query_cluster();
    ctx->gs_cluster = blocks[ctx->device];
    return RPB_OK;
}

// Blocks of the cluster for N spheres, 0 for the kernels over the whole GPU.  Up to kGsChunk spheres a
// block; 64 and fewer for a small suspension, whose time is the latency of the steps and not their
// arithmetic.  Solves in us by 1 / 4 / 8 blocks, float64: 64 spheres 270 / 264 / 263, 200 292 / 264 / 270, 300 314 /
// 320 / 311, 512 349 / 355 / 345; float32, 256: 394 / 365 / 360.  By 4 / 8 / 16, 800 spheres 459 / 453 / 451, 1024
// 539 / 527 / 523, without the wall in float32 700 / 664 / 645.  Up to 32 spheres (two warps of rows) one block and
// eight do not differ.
static int gs_cluster_blocks(const rpb_ctx *ctx, int64_t N)
{
    if (N <= 32) return 1;
    if (N <= 512) return 8;
    return N <= (int64_t)ctx->gs_cluster * kGsChunk ? ctx->gs_cluster : 0;
}

static GsArgs gs_args(rpb_ctx *ctx, int64_t N, bool pack, LzGraph *gr)
{
    const Workspace &w = ctx->ws;
    GsArgs A = {w.V, (size_t)3 * ctx->max_N, N, w.w, nullptr, w.vf, ctx->precond ? w.pc : nullptr, w.selfc,
                pack ? w.src : nullptr, ctx->p.precision == RPB_FP64, w.lz, LzLayout(ctx->max_iter)};
    const size_t nch = (size_t)((N + gs_chunk(N) - 1) / gs_chunk(N));
    A.red = w.red;
    A.red2 = A.red + (size_t)ctx->max_iter * nch;
    A.norm2 = A.red2 + (size_t)ctx->max_iter * nch;
    A.tol = 0.0;
    A.k = 0;
    A.max_iter = 1;
    A.hs = nullptr;
    A.rs = gr ? gr->state : nullptr;
    A.loop = 0;
    return A;
}

static int gs_cluster_launch(cudaStream_t st, const GsArgs &A, int blocks, int init)
{
    count_launches(1);
    return cuda_fail(launch_after(!init, gs_cluster_kernel, dim3(blocks), kGsClusterThreads, blocks, st, A,
                                  (int)((A.N + blocks - 1) / blocks), init),
                     "lanczos cluster kernel");
}

// Everything of an iteration after its product, on the context's stream.
static int gs_iteration(rpb_ctx *ctx, const GsArgs &A)
{
    cudaStream_t st = ctx->stream;
    if (const int blocks = gs_cluster_blocks(ctx, A.N)) return gs_cluster_launch(st, A, blocks, 0);
    const int chunk = (int)gs_chunk(A.N);
    const int nch = (int)((A.N + chunk - 1) / chunk);
    gs_dots_kernel<<<nch, kGsThreads, 0, st>>>(A, chunk);
    gs_project_kernel<<<nch, kGsThreads, 0, st>>>(A, chunk, 0);
    gs_project_kernel<<<nch, kGsThreads, 0, st>>>(A, chunk, 1);
    gs_scale_kernel<<<nch, kGsThreads, 0, st>>>(A, chunk, 0);
    lanczos_tail_kernel<<<1, kTailThreads, 0, st>>>(A, nch);
    count_launches(5);
    return cuda_fail(cudaGetLastError(), "lanczos kernels");
}

int lanczos_init(rpb_ctx *ctx, int64_t N, const double *W, bool packed, LzGraph *gr)
{
    cudaStream_t st = ctx->stream;
    GsArgs A = gs_args(ctx, N, packed, gr);
    A.W = W;
    if (const int blocks = gs_cluster_blocks(ctx, N)) return gs_cluster_launch(st, A, blocks, 1);
    const int chunk = (int)gs_chunk(N);
    const int nch = (int)((N + chunk - 1) / chunk);
    gs_norm_kernel<<<nch, kGsThreads, 0, st>>>(A, chunk);
    gs_scale_kernel<<<nch, kGsThreads, 0, st>>>(A, chunk, 1);
    count_launches(2);
    return cuda_fail(cudaGetLastError(), "lanczos init");
}

int lanczos_impl(rpb_ctx *ctx, int64_t N, const double *pos, const double *W, double *g, double tol, int max_iter,
                 bool packed, int *iters_out, double *err_out, int *converged_out, LzGraph *gr)
{
    int rc;
    if ((rc = lanczos_precond_prepare(ctx, N, pos)) || (rc = lanczos_init(ctx, N, W, packed, gr))) return rc;
    return lanczos_run(ctx, N, pos, g, tol, max_iter, false, packed, iters_out, err_out, converged_out, gr);
}

int lanczos_run(rpb_ctx *ctx, int64_t N, const double *pos, double *g, double tol, int max_iter, bool first_done,
                bool packed, int *iters_out, double *err_out, int *converged_out, LzGraph *gr)
{
    const cudaStream_t main_st = ctx->stream;
    const int64_t n = 3 * N;
    Workspace &w = ctx->ws;
    const double *hs = w.host_status;
    int rc;
    int m = 0;
    bool stopped = false;
    double eps = -1.0;
    // after the first product the positions are packed and each iteration writes the next load beside
    // them (unless the products are the caller's)
    const bool pk = ctx->hook == nullptr;
    GsArgs A = gs_args(ctx, N, pk, gr);
    A.tol = tol;
    A.max_iter = max_iter;
    auto product = [&](bool again) {
        return mobility_apply_impl(ctx, N, pos, w.vf, nullptr, w.w, !pk ? kPlain : (again ? kAgain : kKeep));
    };
    if (gr) {
        // iteration 0 with the step; the others are the body of a loop node that an iteration's
        // tridiagonal step keeps running (its condition is set in every step before the node is met)
        gr->body_launches = 0;
        if (max_iter > 1) {
            cudaStreamCaptureStatus cs;
            cudaGraph_t cg_ = nullptr;
            if ((rc = cuda_fail(cudaStreamGetCaptureInfo(main_st, &cs, nullptr, &cg_, nullptr, nullptr, nullptr),
                                "capture info")) ||
                (rc = cuda_fail(cudaGraphConditionalHandleCreate(&A.loop, cg_, 0u, cudaGraphCondAssignDefault),
                                "conditional handle")))
                return rc;
        }
        if ((!first_done && (rc = product(packed))) || (rc = gs_iteration(ctx, A))) return rc;
        if (max_iter > 1) {
            if ((rc = graph_begin_cond(main_st, gr->body, A.loop, cudaGraphCondTypeWhile))) return rc;
            ctx->stream = gr->body;
            const uint64_t before = rpb_launch_count();
            rc = product(true);
            if (!rc) rc = gs_iteration(ctx, A);
            gr->body_launches = (int)(rpb_launch_count() - before);
            cudaGraph_t body_graph = nullptr;  // owned by the node
            const int erc = cuda_fail(cudaStreamEndCapture(gr->body, &body_graph), "body capture end");
            ctx->stream = main_st;
            if (rc || (rc = erc)) return rc;
        }
    } else {
        // Host-driven: the tridiagonal step leaves its status in pinned memory and an event tells when.  The next
        // product is enqueued before the host knows whether this iteration stopped: the stream would otherwise
        // idle for the host's answer, about 15 us an iteration.  Its kernels read the status and leave if it did.
        // Products that do not ask (one-way kernels, a caller's) are enqueued where a discarded one costs less than the
        // idling of a solve, from what the evaluated pairs take: float32 1.3 ps, float64 150 ps one-way, 200 ps an image
        // of a pseudo-periodic pair (300, 500 and 800 such spheres discarding one 1.58, 2.89 and 6.81 ms, now 1.49, 2.64
        // and 6.07).
        if (!ctx->lz_ev &&
            (rc = cuda_fail(cudaEventCreateWithFlags(&ctx->lz_ev, cudaEventDisableTiming), "lanczos event")))
            return rc;
        const bool per = ctx->Lx > 0.0;
        const double t_product = (per ? 9.0 : 1.0) * (double)N * (double)N *
                                 (ctx->p.precision == RPB_FP32 ? 1.3e-12 : (per ? 2e-10 : 1.5e-10));
        const bool asks = pk && product_stops(ctx, N), speculate = asks || t_product < 1e-4;
        A.hs = w.host_status;
        bool have = first_done;
        for (int k = 0; k < max_iter && !stopped; ++k) {
            A.k = k;
            if (!have && (rc = product(k == 0 ? packed : true))) return rc;
            if ((rc = gs_iteration(ctx, A)) || (rc = cuda_fail(cudaEventRecord(ctx->lz_ev, main_st), "event record")))
                return rc;
            have = speculate && k + 1 < max_iter;
            int ahead = RPB_OK;
            if (have) {
                if (asks) ctx->stop = w.lz + A.L.status + ST_STOP;
                ahead = product(true);
                ctx->stop = nullptr;
                if (ahead && pk) return ahead;
            }
            if ((rc = cuda_fail(cudaEventSynchronize(ctx->lz_ev), "lanczos iteration"))) return rc;
            if (k == 0 && hs[ST_NW] == 0.0) {  // W = 0
                if (iters_out) *iters_out = 0;
                if (err_out) *err_out = -1.0;
                if (converged_out) *converged_out = 1;
                return cuda_fail(cudaMemsetAsync(g, 0, n * sizeof(double), main_st), "zero g");
            }
            m = k + 1;
            eps = hs[ST_EPS];
            stopped = hs[ST_STOP] != 0.0;
            if (ahead && !stopped) return ahead;
            if (ahead) set_error("%s", "");  // a caller's product failed that the solve does not need
        }
    }
    const int tb = elem_threads(n, ctx->num_sms);
    combine_kernel<<<tb == 32 ? (unsigned)((n + 31) / 32) : blas_grid(n, ctx->num_sms), tb, 0, main_st>>>(
        w.V, A.ld, n, m, w.lz + A.L.y, g, gr ? &gr->state->m : nullptr);
    count_launches(1);
    if (ctx->precond && (rc = precond_scale(ctx, N, g, g, true))) return rc;  // g = D^{1/2} y
    if ((rc = cuda_fail(cudaGetLastError(), "lanczos kernels"))) return rc;
    if (gr) return RPB_OK;
    if (iters_out) *iters_out = m;
    if (err_out) *err_out = eps;
    if (converged_out) *converged_out = stopped ? 1 : 0;
    if (tol > 0.0 && !stopped) {
        set_error("lanczos: no convergence in %d iterations (eps=%g, tol=%g)", m, eps, tol);
        return RPB_ENOCONV;
    }
    return RPB_OK;
}

}  // namespace rpb
