// batch.cu -- one call advances many independent suspensions of different sizes (a ragged batch).
//
// The caller keeps each suspension's state in its own device buffers; a call gathers them into a
// packed structure-of-arrays layout (instance b occupies spheres [off_b, off_b + N_b)), runs every
// stage of the step for all instances at once, and scatters the results back.  Per-instance
// quantities (seed, step counter, Lanczos state, convergence) are kept separately, and the work of
// an instance (its target blocks, its source tiles, its reductions) is laid out the same way
// whatever else is in the batch, so an instance's result does not depend on its companions.
//
//   pair products : one 128-target block of one instance per CTA, all of that instance's sources
//                   in 128-source tiles; the float64 self term and s_i/(8 pi eta) in the epilogue.
//   Lanczos       : dot products and Gram-Schmidt over chunks of 256 spheres (one CTA each), the
//                   tridiagonal step by one CTA per instance, instances drop out as they converge.
//   forces        : the cell lists of cells.cuh over the whole batch.
//   noise         : Philox keyed by each instance's seed, counter (k/2, step_b, stream, 0) -- the
//                   same numbers the single-suspension path draws for that seed and step.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "cells.cuh"
#include "gs.cuh"
#include "pair_math.cuh"

namespace rpb {

struct InstDesc {
    int64_t off;      // first sphere in the packed layout
    int N;            // spheres
    int first;        // 1: first step of this instance (Euler-Maruyama)
    uint32_t seed_lo, seed_hi, step, pad;
    double *pos;      // caller's buffers (SoA, 3N), or null
    double *aux;      // U_prev (step) or F (product)
    double *aux2;     // T (product)
    double *out;      // U (product)
};

// A block's share of an instance in the kernels over chunks of kGsChunk spheres, which are numbered instance by
// instance.
struct ChunkDesc {
    int inst, first;    // instance, its first sphere (instance-local)
    int chunk0, count;  // the instance's first chunk and its number of chunks
};

struct BlockDesc {
    int inst;
    int first;  // first target (instance-local) of this 128-target block
};


// ------------------------------------------------------------------ layout kernels
__global__ void inst_of_kernel(const InstDesc *__restrict__ inst, int B, int *__restrict__ inst_of)
{
    const int b = blockIdx.x;
    if (b >= B) return;
    const InstDesc d = inst[b];
    for (int i = threadIdx.x; i < d.N; i += blockDim.x) inst_of[d.off + i] = b;
}

// Copy (or write back) three-component SoA vectors between the callers' buffers and the packed
// layout.  which: 0 = pos, 1 = aux, 2 = aux2, 3 = out.
__global__ void gather_kernel(const InstDesc *__restrict__ inst, const int *__restrict__ inst_of, int64_t total,
                              int which, double *__restrict__ packed, int to_caller)
{
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < 3 * total; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c = r / total, i = r - c * total;
        const InstDesc &d = inst[inst_of[i]];
        double *p = which == 0 ? d.pos : (which == 1 ? d.aux : (which == 2 ? d.aux2 : d.out));
        const int64_t k = c * d.N + (i - d.off);
        if (to_caller)
            p[k] = packed[r];
        else
            packed[r] = p ? p[k] : 0.0;
    }
}

// ------------------------------------------------------------------ pair products
template <bool TORQUE>
__global__ void __launch_bounds__(kPairThreads, 6) batch_pair_f32x2_kernel(
    const SrcF32 *__restrict__ src, const InstDesc *__restrict__ inst, const BlockDesc *__restrict__ blocks,
    const int *__restrict__ active, int64_t total, X2Consts c, PairConsts<double> cd, double a, double scale,
    const double *__restrict__ pos, const double *__restrict__ F, const double *__restrict__ T, double *__restrict__ U)
{
    constexpr int P = kTile / 2;
    __shared__ float4 sA[P], sB[P], sC[P], sD[P];
    __shared__ float4 sE[TORQUE ? P : 1];
    __shared__ float2 sG[TORQUE ? P : 1];
    const BlockDesc bd = blocks[blockIdx.x];
    if (active && !active[bd.inst]) return;
    const InstDesc d = inst[bd.inst];
    const int tid = threadIdx.x;
    const int il = bd.first + tid;
    const int64_t i = d.off + il;
    const bool valid = il < d.N;
    float4 tp = make_float4(0.f, 0.f, 0.f, 0.f);
    float tz = 1.f;
    if (valid) {
        tp = src[i].p;
        tz = src[i].f.x;
    }
    const float2 txh = make_float2(tp.x, tp.x), tyh = make_float2(tp.y, tp.y);
    const float2 txl = make_float2(tp.z, tp.z), tyl = make_float2(tp.w, tp.w);
    const float2 tz2 = make_float2(tz, tz);
    const float2 zero2 = make_float2(0.f, 0.f);
    float sx = 0.f, sy = 0.f, sz = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
    const int pp = tid >> 1, hh = tid & 1;
    float *fA = reinterpret_cast<float *>(sA);
    float *fB = reinterpret_cast<float *>(sB);
    float *fC = reinterpret_cast<float *>(sC);
    float *fD = reinterpret_cast<float *>(sD);
    float *fE = reinterpret_cast<float *>(sE);
    float *fG = reinterpret_cast<float *>(sG);
    for (int base = 0; base < d.N; base += kTile) {
        const int jl = base + tid;
        float4 sp_ = make_float4(1e18f, 0.f, 0.f, 0.f), sf_ = make_float4(1.f, 0.f, 0.f, 0.f);
        float4 st_ = make_float4(0.f, 0.f, 0.f, 0.f);
        if (jl < d.N) {
            sp_ = src[d.off + jl].p;
            sf_ = src[d.off + jl].f;
            if (TORQUE) st_ = src[d.off + jl].t;
        }
        fA[4 * pp + hh] = sp_.x;
        fA[4 * pp + 2 + hh] = sp_.y;
        fB[4 * pp + hh] = sp_.z;
        fB[4 * pp + 2 + hh] = sp_.w;
        fC[4 * pp + hh] = sf_.x;
        fC[4 * pp + 2 + hh] = sf_.y;
        fD[4 * pp + hh] = sf_.z;
        fD[4 * pp + 2 + hh] = sf_.w;
        if (TORQUE) {
            fE[4 * pp + hh] = st_.x;
            fE[4 * pp + 2 + hh] = st_.y;
            fG[2 * pp + hh] = st_.z;
        }
        __syncthreads();
        float2 ux = zero2, uy = zero2, uz = zero2;
        const bool diag = base == bd.first;
        for (int k = 0; k < P; ++k) {
            const float4 av = sA[k], bv = sB[k], cc = sC[k], dv = sD[k];
            const float4 e = TORQUE ? sE[k] : make_float4(0.f, 0.f, 0.f, 0.f);
            const float2 g = TORQUE ? sG[k] : zero2;
            // instances are small (every warp iteration has some pair within 10a), so the low parts
            // of the positions are always added
            const float2 rx = add2(sub2(txh, make_float2(av.x, av.y)), sub2(txl, make_float2(bv.x, bv.y)));
            const float2 ry = add2(sub2(tyh, make_float2(av.z, av.w)), sub2(tyl, make_float2(bv.z, bv.w)));
            float2 dx = zero2, dy = zero2, dz = zero2;
            pair_velocity_x2<TORQUE>(rx, ry, tz2, make_float2(cc.x, cc.y), make_float2(cc.z, cc.w),
                                     make_float2(dv.x, dv.y), make_float2(dv.z, dv.w), make_float2(e.x, e.y),
                                     make_float2(e.z, e.w), g, c, dx, dy, dz);
            if (diag && k == pp) {  // source 2k + hh of the diagonal tile is this thread's sphere
                if (hh == 0) {
                    dx.x = 0.f;
                    dy.x = 0.f;
                    dz.x = 0.f;
                } else {
                    dx.y = 0.f;
                    dy.y = 0.f;
                    dz.y = 0.f;
                }
            }
            ux = add2(ux, dx);
            uy = add2(uy, dy);
            uz = add2(uz, dz);
        }
        {
            const float tx = ux.x + ux.y, ty = uy.x + uy.y, tzs = uz.x + uz.y;
            float yv = tx - cx, tv = sx + yv;
            cx = (tv - sx) - yv;
            sx = tv;
            yv = ty - cy;
            tv = sy + yv;
            cy = (tv - sy) - yv;
            sy = tv;
            yv = tzs - cz;
            tv = sz + yv;
            cz = (tv - sz) - yv;
            sz = tv;
        }
        __syncthreads();
    }
    if (valid) {
        double ux = (double)sx - (double)cx, uy = (double)sy - (double)cy, uz = (double)sz - (double)cz;
        const double z = pos[2 * total + i];
        const double si = H0(z / a), zc = fmax(z, a);
        const double Fx = F ? si * F[i] : 0.0, Fy = F ? si * F[total + i] : 0.0, Fz = F ? si * F[2 * total + i] : 0.0;
        if (TORQUE)
            self_velocity<true>(zc, Fx, Fy, Fz, si * T[i], si * T[total + i], cd, ux, uy, uz);
        else
            self_velocity<false>(zc, Fx, Fy, Fz, 0.0, 0.0, cd, ux, uy, uz);
        const double k = si * scale;
        U[i] = k * ux;
        U[total + i] = k * uy;
        U[2 * total + i] = k * uz;
    }
}

template <bool TORQUE>
__global__ void __launch_bounds__(kPairThreads) batch_pair_f64_kernel(
    const SrcF64 *__restrict__ src, const InstDesc *__restrict__ inst, const BlockDesc *__restrict__ blocks,
    const int *__restrict__ active, int64_t total, PairConsts<double> c, double a, double scale,
    const double *__restrict__ pos, const double *__restrict__ F, const double *__restrict__ T, double *__restrict__ U)
{
    __shared__ double2 sp[kTile], sq[kTile], sr[kTile];
    __shared__ double2 ss[TORQUE ? kTile : 1], su[TORQUE ? kTile : 1];
    const BlockDesc bd = blocks[blockIdx.x];
    if (active && !active[bd.inst]) return;
    const InstDesc d = inst[bd.inst];
    const int tid = threadIdx.x;
    const int il = bd.first + tid;
    const int64_t i = d.off + il;
    const bool valid = il < d.N;
    double2 tp = make_double2(0.0, 0.0);
    double tz = 1.0;
    if (valid) {
        tp = src[i].p;
        tz = src[i].q.x;
    }
    double ux = 0.0, uy = 0.0, uz = 0.0;
    for (int base = 0; base < d.N; base += kTile) {
        const int jl = base + tid;
        if (jl < d.N) {
            const SrcF64 s = src[d.off + jl];
            sp[tid] = s.p;
            sq[tid] = s.q;
            sr[tid] = s.r;
            if (TORQUE) {
                ss[tid] = s.s;
                su[tid] = s.u;
            }
        }
        __syncthreads();
        const int cnt = min(kTile, d.N - base);
        const bool diag = base == bd.first;
        for (int k = 0; k < cnt; ++k) {
            const double2 p = sp[k], q = sq[k], r = sr[k];
            const double2 s = TORQUE ? ss[k] : make_double2(0.0, 0.0);
            const double2 u = TORQUE ? su[k] : make_double2(0.0, 0.0);
            double dx = 0.0, dy = 0.0, dz = 0.0;
            pair_velocity_f64<TORQUE>(tp.x - p.x, tp.y - p.y, tz, q.x, q.y, r.x, r.y, s.x, s.y, u.x, c, dx, dy, dz);
            if (!(diag && k == tid)) {
                ux += dx;
                uy += dy;
                uz += dz;
            }
        }
        __syncthreads();
    }
    if (valid) {
        const double z = pos[2 * total + i];
        const double si = H0(z / a), zc = fmax(z, a);
        const double Fx = F ? si * F[i] : 0.0, Fy = F ? si * F[total + i] : 0.0, Fz = F ? si * F[2 * total + i] : 0.0;
        if (TORQUE)
            self_velocity<true>(zc, Fx, Fy, Fz, si * T[i], si * T[total + i], c, ux, uy, uz);
        else
            self_velocity<false>(zc, Fx, Fy, Fz, 0.0, 0.0, c, ux, uy, uz);
        const double k = si * scale;
        U[i] = k * ux;
        U[total + i] = k * uy;
        U[2 * total + i] = k * uz;
    }
}

// ------------------------------------------------------------------ noise and elementwise steps
__device__ __forceinline__ uint4 philox4x32_10_b(uint4 c, uint32_t k0, uint32_t k1)
{
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t lo0 = M0 * c.x, hi0 = __umulhi(M0, c.x);
        const uint32_t lo1 = M1 * c.z, hi1 = __umulhi(M1, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// Normals k = 2p and 2p + 1 (k = 3 il + c, il local index) of both noise streams (blockIdx.y: 0 into W, 1 into
// Wt), one block per chunk.  One thread per counter: the logarithm, square root and sincospi (about 80 float64 instructions, which
// bound this kernel) serve the two normals they give; a thread per normal did them twice.
__global__ void __launch_bounds__(256) batch_philox_kernel(const InstDesc *__restrict__ inst,
                                                           const ChunkDesc *__restrict__ chunks, int64_t total,
                                                           double *__restrict__ W, double *__restrict__ Wt)
{
    // a chunk of 256 spheres holds normals 768 q .. 768 q + 767 of its instance: 384 counters
    const ChunkDesc c = chunks[blockIdx.x];
    const InstDesc d = inst[c.inst];
    const uint32_t sid = blockIdx.y;
    double *out = sid ? Wt : W;
    const int n = 3 * d.N, p0 = 3 * c.first / 2;
    const int p1 = min((n + 1) / 2, p0 + 3 * kGsChunk / 2);
    for (int p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        const uint4 w = philox4x32_10_b(make_uint4((uint32_t)p, d.step, sid, 0u), d.seed_lo, d.seed_hi);
        const double two26 = 67108864.0, two_m53 = 1.1102230246251565e-16;
        const double u1 = ((double)(w.x >> 5) * two26 + (double)(w.y >> 6) + 1.0) * two_m53;
        const double u2 = ((double)(w.z >> 5) * two26 + (double)(w.w >> 6) + 1.0) * two_m53;
        const double rad = sqrt(-2.0 * log(u1));
        double sn, cs;
        sincospi(2.0 * u2, &sn, &cs);
        const int ka = 2 * p, kb = ka + 1;
        out[(int64_t)(ka % 3) * total + d.off + ka / 3] = rad * cs;
        if (kb < n) out[(int64_t)(kb % 3) * total + d.off + kb / 3] = rad * sn;
    }
}

__global__ void batch_ab_update_kernel(const InstDesc *__restrict__ inst, const int *__restrict__ inst_of, int64_t total,
                                       double *__restrict__ pos, double *__restrict__ U_prev,
                                       const double *__restrict__ Un, const double *__restrict__ g,
                                       const double *__restrict__ drift, double dt, double noise_scale)
{
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < 3 * total; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = r % total;
        const double un = Un[r];
        const double up = inst[inst_of[i]].first ? un : U_prev[r];
        pos[r] = pos[r] + dt * (1.5 * un - 0.5 * up) + noise_scale * g[r] + dt * drift[r];
        U_prev[r] = un;
    }
}

__global__ void batch_fill3_kernel(double *__restrict__ v, int64_t total, double x, double y, double z)
{
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < 3 * total; r += (int64_t)gridDim.x * blockDim.x)
        v[r] = r < total ? x : (r < 2 * total ? y : z);
}

__global__ void batch_displace_kernel(const double *__restrict__ pos, const double *__restrict__ Wt, int64_t n, double h,
                                      double *__restrict__ plus, double *__restrict__ minus)
{
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        const double q = pos[r], dd = h * Wt[r];
        plus[r] = q + dd;
        minus[r] = q - dd;
    }
}

__global__ void batch_rfd_combine_kernel(double *__restrict__ up_drift, const double *__restrict__ um, int64_t n, double k)
{
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
        up_drift[r] = k * (up_drift[r] - um[r]);
}

// ------------------------------------------------------------------ batched Lanczos
// Every instance's spheres are cut into chunks of kGsChunk, one block each (gs.cuh), numbered instance by
// instance; a reduction writes one partial per chunk and the next kernel adds an instance's own in a
// fixed order, so nothing depends on the companions.  (One block per instance left the largest instances
// to one SM: of a served mix with suspensions of up to 32768 spheres, 24 instances, the dot products and
// projections took 18% of a step; 7.7 of 42 ms.)

__device__ __forceinline__ GsSpan chunk_span(const ChunkDesc &c, const InstDesc &d, int64_t total)
{
    return GsSpan{d.off + c.first, total, min(kGsChunk, d.N - c.first)};
}

// The iteration a kernel of the loop works on: k, or in a replayed graph the one the device is at.
__device__ __forceinline__ int batch_iter(int k, const int *__restrict__ d_k)
{
    return d_k ? *d_k : k;
}

// red[j nchunks + chunk] = the chunk's part of <V_j, w>, j <= k
__global__ void __launch_bounds__(kGsThreads) batch_dots_kernel(const double *__restrict__ V, size_t ld, int k,
                                                                const int *__restrict__ d_k,
                                                                const double *__restrict__ w,
                                                                const InstDesc *__restrict__ inst,
                                                                const ChunkDesc *__restrict__ chunks,
                                                                const int *__restrict__ active, int64_t total,
                                                                double *__restrict__ red)
{
    __shared__ double sh[kGsWarps][kMaxIter + 8];
    const ChunkDesc c = chunks[blockIdx.x];
    if (active && !active[c.inst]) return;  // uniform per block
    const int nvec = batch_iter(k, d_k) + 1;
    int64_t row[kGsRows];
    double x[kGsRows];
    const GsSpan span = chunk_span(c, inst[c.inst], total);
    const int nu = gs_rows(span, row), nw = gs_warps(span);
#pragma unroll
    for (int u = 0; u < kGsRows; ++u) x[u] = row[u] >= 0 ? w[row[u]] : 0.0;
    const double s = gs_dots(V, ld, nvec, row, nu, nw, x, sh);
    if (threadIdx.x < nvec) red[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = s;
}

// w -= sum_j c_j V_j with c_j from the partials `red`; the instance's first chunk stores c in its state block
// (lz_b + coef_off).  Then, with red2, the dot products of the new w (the second pass of Gram-Schmidt) as
// batch_dots_kernel, or the chunk's part of |w|^2 in norm2.
__global__ void __launch_bounds__(kGsThreads) batch_project_kernel(const double *__restrict__ V, size_t ld, int k,
                                                                   const int *__restrict__ d_k,
                                                                   double *__restrict__ w,
                                                                   const InstDesc *__restrict__ inst,
                                                                   const ChunkDesc *__restrict__ chunks,
                                                                   const int *__restrict__ active, int64_t total,
                                                                   const double *__restrict__ red,
                                                                   double *__restrict__ lz, size_t lz_stride,
                                                                   size_t coef_off, double *__restrict__ red2,
                                                                   double *__restrict__ norm2)
{
    __shared__ double sh[kGsWarps][kMaxIter + 8];
    __shared__ double coef[kMaxIter];
    const ChunkDesc c = chunks[blockIdx.x];
    if (active && !active[c.inst]) return;
    const int nvec = batch_iter(k, d_k) + 1;
    int64_t row[kGsRows];
    double x[kGsRows];
    const GsSpan span = chunk_span(c, inst[c.inst], total);
    const int nu = gs_rows(span, row), nw = gs_warps(span);
#pragma unroll
    for (int u = 0; u < kGsRows; ++u) x[u] = row[u] >= 0 ? w[row[u]] : 0.0;
    gs_coefs(red + c.chunk0, gridDim.x, c.count, nvec, coef);
    if (c.first == 0 && threadIdx.x < nvec) lz[(size_t)c.inst * lz_stride + coef_off + threadIdx.x] = coef[threadIdx.x];
    gs_project(V, ld, nvec, row, nu, coef, x);
#pragma unroll
    for (int u = 0; u < kGsRows; ++u)
        if (row[u] >= 0) w[row[u]] = x[u];
    if (red2) {
        const double s = gs_dots(V, ld, nvec, row, nu, nw, x, sh);
        if (threadIdx.x < nvec) red2[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = s;
    } else {
        double s = 0.0;
#pragma unroll
        for (int u = 0; u < kGsRows; ++u) s = fma(x[u], x[u], s);
        s = gs_block_sum(s, nu, nw, sh[0]);
        if (threadIdx.x == 0) norm2[blockIdx.x] = s;
    }
}

// |W_b| per instance from the chunks' squared norms, one warp each; v_0 scale factors; activity.
__global__ void __launch_bounds__(128) batch_norm_init_kernel(const double *__restrict__ red,
                                                              const int2 *__restrict__ inst_chunks, int B,
                                                              double *__restrict__ lz, size_t lz_stride,
                                                              size_t status_off, int *__restrict__ active)
{
    const int b = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= B) return;
    const int2 c = inst_chunks[b];
    double s = 0.0;
    for (int k = lane; k < c.y; k += 32) s += red[c.x + k];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane != 0) return;
    double *st = lz + (size_t)b * lz_stride + status_off;
    const double nw = sqrt(s);
    st[ST_NW] = nw;
    st[ST_INV_NW] = nw > 0.0 ? 1.0 / nw : 0.0;
    st[ST_EPS] = -1.0;
    st[ST_STOP] = nw > 0.0 ? 0.0 : 1.0;
    st[ST_BREAK] = 0.0;
    st[6] = 0.0;  // m (iterations used)
    st[7] = nw > 0.0 ? 0.0 : 1.0;  // converged flag
    active[b] = nw > 0.0 ? 1 : 0;
}

// Basis vector row0 (in a replayed graph the one after the iteration's) = w * status_b[idx] for the active
// instances (all when active is null); also into vf, the next product's load, and times s_i into its
// packed sources, whose positions stay packed through a solve.
__global__ void __launch_bounds__(kGsThreads) batch_scale_kernel(const double *__restrict__ w,
                                                                 const InstDesc *__restrict__ inst,
                                                                 const ChunkDesc *__restrict__ chunks,
                                                                 const int *__restrict__ active, int64_t total,
                                                                 const double *__restrict__ lz, size_t lz_stride,
                                                                 size_t status_off, int idx, double *__restrict__ V,
                                                                 size_t ld, int row0, const int *__restrict__ d_k,
                                                                 double *__restrict__ vf, const double *__restrict__ s,
                                                                 void *__restrict__ src, int fp64)
{
    const ChunkDesc c = chunks[blockIdx.x];
    if (active && !active[c.inst]) return;
    double *v = V + (size_t)(d_k ? *d_k + 1 : row0) * ld;
    const double inv = lz[(size_t)c.inst * lz_stride + status_off + idx];
    int64_t row[kGsRows];
    gs_rows(chunk_span(c, inst[c.inst], total), row);
#pragma unroll
    for (int u = 0; u < kGsRows; ++u) {
        const int64_t r = row[u];
        if (r < 0) continue;
        const double x = w[r] * inv;
        v[r] = x;
        vf[r] = x;
        const int q = r < total ? 0 : (r < 2 * total ? 1 : 2);
        const int64_t i = r - q * total;
        const double f = s[i] * x;
        if (fp64)
            reinterpret_cast<double *>((SrcF64 *)src + i)[3 + q] = f;
        else
            reinterpret_cast<float *>((SrcF32 *)src + i)[5 + q] = (float)f;
    }
}

// One block per instance: the tridiagonal step; converged instances leave the active set.
__global__ void __launch_bounds__(kTailThreads) batch_tail_kernel(double *__restrict__ lz, size_t lz_stride, LzLayout L,
                                                                  int k, const int *__restrict__ d_k, double tol,
                                                                  const double *__restrict__ norm2,
                                                                  const int2 *__restrict__ inst_chunks,
                                                                  const double *__restrict__ nodes,
                                                                  int *__restrict__ active, int *__restrict__ n_active)
{
    __shared__ TailShared sh;
    const int b = blockIdx.x;
    if (!active[b]) return;  // the whole block leaves together
    k = batch_iter(k, d_k);
    double *lzb = lz + (size_t)b * lz_stride;
    const int2 c = inst_chunks[b];
    double s = 0.0;  // |w|^2 from the chunks' parts (every warp, the same in every thread)
    for (int q = threadIdx.x & 31; q < c.y; q += 32) s += norm2[c.x + q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const TailRegs reg = lanczos_tail_load(lzb, L, k, nodes, sh, threadIdx.x);
    const TailResult r = lanczos_tail_y(lzb, L, k, lzb[L.c1 + k] + lzb[L.c2 + k], reg, sh, threadIdx.x);
    if (threadIdx.x == 0) {
        double *st = lzb + L.status;
        st[6] = k + 1;
        if (lanczos_tail_stop(lzb, L, k, tol, sqrt(s), r, reg.nW, nullptr)) {
            st[7] = 1.0;
            active[b] = 0;
        } else {
            atomicAdd(n_active, 1);
        }
    }
}

// g[r] = sum_{k < m_b} y_b[k] V[k][r]
__global__ void batch_combine_kernel(const double *__restrict__ V, size_t ld, const int *__restrict__ inst_of,
                                     int64_t total, const double *__restrict__ lz, size_t lz_stride, LzLayout L,
                                     double *__restrict__ g)
{
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < 3 * total; r += (int64_t)gridDim.x * blockDim.x) {
        const double *lzb = lz + (size_t)inst_of[r % total] * lz_stride;
        const int m = (int)lzb[L.status + 6];
        double acc = 0.0;
        for (int k = 0; k < m; ++k) acc = fma(lzb[L.y + k], V[(size_t)k * ld + r], acc);
        g[r] = acc;
    }
}

}  // namespace rpb

using namespace rpb;

struct rpb_batch {
    rpb_params p;
    int64_t max_total;
    int max_B;
    int max_iter;
    cudaStream_t stream;
    int num_sms;
    size_t lz_stride;
    // device
    InstDesc *d_inst = nullptr;
    BlockDesc *d_blocks = nullptr;
    ChunkDesc *d_chunks = nullptr;   // chunks of the Gram-Schmidt kernels, and each instance's (first, count)
    int2 *d_inst_chunks = nullptr;
    int *d_inst_of = nullptr;
    int *d_active = nullptr;
    int *d_nactive = nullptr;
    void *src = nullptr;
    double *vec[13] = {};  // pos, Up, F, T, Un, W, Wt, g, drift, pos_a, pos_b, w, the next product's load
    double *V = nullptr;
    double *lz = nullptr;
    double *red = nullptr;
    double *norm2 = nullptr;
    double *selfc = nullptr;  // self coefficients of the packed positions (SelfCoefs), 4 max_total_N
    void *cells = nullptr;    // cell lists of the force pass (cell_lists_bytes)
    double *nodes = nullptr;  // nodes and weights of the Lanczos square root
    // host (pinned)
    InstDesc *h_inst = nullptr;
    BlockDesc *h_blocks = nullptr;
    ChunkDesc *h_chunks = nullptr;
    int2 *h_inst_chunks = nullptr;
    int *h_nactive = nullptr;
    double *h_lz = nullptr;
    int64_t total = 0;
    int B = 0;
    int nblocks = 0, nchunks = 0;
    // multi-step runs: a private stream to capture and replay the step graph on, joined to the
    // caller's stream by an event; a device counter of unconverged instance-steps
    cudaStream_t cap = nullptr;
    cudaStream_t loop = nullptr;  // the WHILE node's body (a step) is captured here
    int *d_left = nullptr;        // steps left in the run
    cudaEvent_t join = nullptr;
    unsigned long long *d_unconv = nullptr;
    unsigned long long *h_unconv = nullptr;
    // graph-replayed Lanczos: the iterations after the first run in a loop node of the graph, captured on
    // `body`; d_k is the iteration, d_loops counts the body's runs (for the launch count)
    cudaStream_t body = nullptr;
    int *d_k = nullptr;
    unsigned long long *d_loops = nullptr;
    unsigned long long *h_loops = nullptr;
    int body_launches = 0;
    // float32 products by the symmetric pass (both directions of a pair from one evaluation):
    // schedule and partial-sum scratch for the current batch sizes
    bool sym_enabled = false;
    bool sym_ok = false;
    BatchSymPlan sym;
    int seg_tiles = 8;  // run length of the symmetric pass's row cut (rpb_batch_set_tiles / rpb_batch_tune)
    int sym_env = 1;    // RPB_FP32_BATCH_SYM (the symmetric pass unless "0")
};

namespace rpb {

enum { V_POS, V_UP, V_F, V_T, V_UN, V_W, V_WT, V_G, V_DRIFT, V_PA, V_PB, V_WORK, V_VF };

static void batch_free(rpb_batch *bt)
{
    void *dev[] = {bt->d_inst, bt->d_blocks, bt->d_chunks, bt->d_inst_chunks, bt->d_inst_of, bt->d_active, bt->d_nactive, bt->src, bt->V, bt->lz, bt->red,
                   bt->norm2, bt->selfc, bt->nodes, bt->cells, bt->d_left};
    for (void *p : dev)
        if (p) cudaFree(p);
    for (double *p : bt->vec)
        if (p) cudaFree(p);
    void *host[] = {bt->h_inst, bt->h_blocks, bt->h_chunks, bt->h_inst_chunks, bt->h_nactive, bt->h_lz, bt->h_unconv};
    for (void *p : host)
        if (p) cudaFreeHost(p);
    if (bt->d_unconv) cudaFree(bt->d_unconv);
    if (bt->d_k) cudaFree(bt->d_k);
    if (bt->d_loops) cudaFree(bt->d_loops);
    if (bt->h_loops) cudaFreeHost(bt->h_loops);
    if (bt->body) cudaStreamDestroy(bt->body);
    batch_sym_free(bt->sym);
    if (bt->join) cudaEventDestroy(bt->join);
    if (bt->cap) cudaStreamDestroy(bt->cap);
    if (bt->loop) cudaStreamDestroy(bt->loop);
}

static int grid_for(int64_t n, int sms)
{
    int64_t g = (n + 255) / 256;
    if (g > 16 * (int64_t)sms) g = 16 * sms;
    return g < 1 ? 1 : (int)g;
}

// Describe the batch on the host and copy the descriptors to the device.  Blocks are listed
// largest instance first so that the long CTAs start early.
static int batch_setup(rpb_batch *bt, int B, const int64_t *N, const int64_t *steps, const uint64_t *seeds,
                       double *const *pos, double *const *aux, const double *const *aux2, double *const *out)
{
    if (B < 1 || B > bt->max_B) {
        set_error("batch size B=%d outside [1, %d]", B, bt->max_B);
        return RPB_EINVAL;
    }
    int64_t total = 0;
    for (int b = 0; b < B; ++b) {
        if (N[b] <= 0 || N[b] > (int64_t)1 << 30) {
            set_error("instance %d: N=%lld invalid", b, (long long)N[b]);
            return RPB_EINVAL;
        }
        total += N[b];
    }
    if (total > bt->max_total) {
        set_error("batch of %lld spheres exceeds the context's max_total_N=%lld", (long long)total,
                  (long long)bt->max_total);
        return RPB_EINVAL;
    }
    int64_t off = 0;
    int nblk = 0;
    for (int b = 0; b < B; ++b) {
        InstDesc &d = bt->h_inst[b];
        d.off = off;
        d.N = (int)N[b];
        d.first = steps ? (steps[b] == 0) : 0;
        const uint64_t s = seeds ? seeds[b] : 0;
        d.seed_lo = (uint32_t)(s & 0xffffffffu);
        d.seed_hi = (uint32_t)(s >> 32);
        d.step = steps ? (uint32_t)steps[b] : 0u;
        d.pad = 0;
        d.pos = pos ? pos[b] : nullptr;
        d.aux = aux ? aux[b] : nullptr;
        d.aux2 = aux2 ? const_cast<double *>(aux2[b]) : nullptr;
        d.out = out ? out[b] : nullptr;
        off += N[b];
        nblk += (int)((N[b] + kTile - 1) / kTile);
    }
    std::vector<int> order(B);
    for (int b = 0; b < B; ++b) order[b] = b;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return N[x] > N[y]; });
    int k = 0;
    for (int b : order)
        for (int64_t f = 0; f < N[b]; f += kTile) bt->h_blocks[k++] = BlockDesc{b, (int)f};
    int nc = 0;
    for (int b = 0; b < B; ++b) {
        const int cnt = (int)((N[b] + kGsChunk - 1) / kGsChunk), c0 = nc;
        bt->h_inst_chunks[b] = make_int2(c0, cnt);
        for (int q = 0; q < cnt; ++q) bt->h_chunks[nc++] = ChunkDesc{b, q * kGsChunk, c0, cnt};
    }
    bt->total = total;
    bt->B = B;
    bt->nblocks = nblk;
    bt->nchunks = nc;
    int rc;
    if ((rc = cuda_fail(cudaMemcpyAsync(bt->d_chunks, bt->h_chunks, nc * sizeof(ChunkDesc), cudaMemcpyHostToDevice,
                                        bt->stream),
                        "batch chunks")) ||
        (rc = cuda_fail(cudaMemcpyAsync(bt->d_inst_chunks, bt->h_inst_chunks, B * sizeof(int2), cudaMemcpyHostToDevice,
                                        bt->stream),
                        "batch chunks")))
        return rc;
    if ((rc = cuda_fail(cudaMemcpyAsync(bt->d_inst, bt->h_inst, B * sizeof(InstDesc), cudaMemcpyHostToDevice, bt->stream),
                        "batch descriptors")))
        return rc;
    if ((rc = cuda_fail(cudaMemcpyAsync(bt->d_blocks, bt->h_blocks, nblk * sizeof(BlockDesc), cudaMemcpyHostToDevice,
                                        bt->stream),
                        "batch blocks")))
        return rc;
    inst_of_kernel<<<B, 256, 0, bt->stream>>>(bt->d_inst, B, bt->d_inst_of);
    count_launches(1);
    if ((rc = cuda_fail(cudaGetLastError(), "inst_of"))) return rc;
    bt->sym_ok = false;
    if (bt->sym_enabled && (rc = batch_sym_plan(bt->sym, B, N, bt->stream, &bt->sym_ok, bt->seg_tiles))) return rc;
    return RPB_OK;
}

static int batch_gather(rpb_batch *bt, int which, double *packed, int to_caller)
{
    gather_kernel<<<grid_for(3 * bt->total, bt->num_sms), 256, 0, bt->stream>>>(bt->d_inst, bt->d_inst_of, bt->total,
                                                                               which, packed, to_caller);
    count_launches(1);
    return cuda_fail(cudaGetLastError(), "batch gather");
}

// U = M_tt F + M_tr T over the packed layout; F or T may be null; active masks instances.  packed: the packed
// sources hold these positions and s F already (T null).
static int batch_product(rpb_batch *bt, const double *pos, const double *F, const double *T, double *U,
                         const int *active, bool packed = false)
{
    const int64_t total = bt->total;
    const double a = bt->p.a;
    const double scale = 1.0 / (8.0 * kPi * bt->p.eta);
    const int pb = 256;
    const int gpack = (int)((total + pb - 1) / pb);
    const SelfCoefs sc = {bt->selfc, total, scale, make_consts<double>(a)};
    if (bt->p.precision == RPB_FP32 && bt->sym_ok) {
        SrcF32 *src = (SrcF32 *)bt->src;
        if (!packed) pack_f32_kernel<<<gpack, pb, 0, bt->stream>>>(pos, F, T, (int)total, a, 1, src, sc);
        count_launches(!packed);
        return batch_sym_apply(bt->sym, bt->stream, src, total, F, T, U, active, a, sc);
    } else if (bt->p.precision == RPB_FP32) {
        SrcF32 *src = (SrcF32 *)bt->src;
        if (!packed) pack_f32_kernel<<<gpack, pb, 0, bt->stream>>>(pos, F, T, (int)total, a, 1, src, sc);
        const X2Consts c = make_x2_consts(a);
        const PairConsts<double> cd = make_consts<double>(a);
        if (T)
            batch_pair_f32x2_kernel<true><<<bt->nblocks, kPairThreads, 0, bt->stream>>>(
                src, bt->d_inst, bt->d_blocks, active, total, c, cd, a, scale, pos, F, T, U);
        else
            batch_pair_f32x2_kernel<false><<<bt->nblocks, kPairThreads, 0, bt->stream>>>(
                src, bt->d_inst, bt->d_blocks, active, total, c, cd, a, scale, pos, F, T, U);
    } else {
        SrcF64 *src = (SrcF64 *)bt->src;
        if (!packed) pack_f64_kernel<<<gpack, pb, 0, bt->stream>>>(pos, F, T, (int)total, a, 1, src, sc);
        const PairConsts<double> c = make_consts<double>(a);
        if (T)
            batch_pair_f64_kernel<true><<<bt->nblocks, kPairThreads, 0, bt->stream>>>(
                src, bt->d_inst, bt->d_blocks, active, total, c, a, scale, pos, F, T, U);
        else
            batch_pair_f64_kernel<false><<<bt->nblocks, kPairThreads, 0, bt->stream>>>(
                src, bt->d_inst, bt->d_blocks, active, total, c, a, scale, pos, F, T, U);
    }
    count_launches(packed ? 1 : 2);
    return cuda_fail(cudaGetLastError(), "batch pair kernels");
}

// Inside a replayed graph, the end of an iteration: the next one, counted, and the loop node's body runs again
// while some instance is still active and iterations are left.
__global__ void batch_iter_kernel(cudaGraphConditionalHandle loop, int max_iter, const int *__restrict__ n_active,
                                  int *__restrict__ d_k, unsigned long long *__restrict__ loops)
{
    const int k = *d_k;
    *d_k = k + 1;
    if (k > 0) *loops += 1ull;
    if (max_iter > 1) cudaGraphSetConditional(loop, *n_active > 0 && k + 1 < max_iter ? 1u : 0u);
}

// Lanczos for every instance at once; per-instance m, eps and convergence land in h_lz statuses.
// graph == false: the host reads the number of still-active instances after every iteration and stops
// when it reaches zero, then copies the per-instance statuses to h_lz.  graph == true (inside a CUDA
// graph capture): iteration 0 is captured as is and the others as the body of a loop (WHILE) node that runs
// while some instance is still active (the end of an iteration sets its condition), so a replay does the
// iterations the step needs, at most max_iter; converged instances are masked out of every kernel, and
// nothing is read back.
static int batch_lanczos(rpb_batch *bt, const double *pos, const double *W, double *g, double tol, int max_iter,
                         bool graph = false)
{
    cudaStream_t main_st = bt->stream;
    const int B = bt->B;
    const int64_t total = bt->total;
    const size_t ld = (size_t)3 * bt->max_total;
    const LzLayout L(bt->max_iter);
    double *V = bt->V, *w = bt->vec[V_WORK], *vf = bt->vec[V_VF];
    const int ge = grid_for(3 * total, bt->num_sms), nc = bt->nchunks;
    const int fp64 = bt->p.precision == RPB_FP64;
    double *red2 = bt->red + (size_t)bt->max_iter * nc;
    const int *d_k = graph ? bt->d_k : nullptr;
    int rc;
    cudaGraphConditionalHandle loop = 0;
    if (graph) {
        cudaStreamCaptureStatus cs;
        cudaGraph_t cg = nullptr;
        if ((rc = cuda_fail(cudaStreamGetCaptureInfo(main_st, &cs, nullptr, &cg, nullptr, nullptr, nullptr),
                            "capture info")) ||
            (rc = cuda_fail(cudaGraphConditionalHandleCreate(&loop, cg, 0u, cudaGraphCondAssignDefault),
                            "conditional handle")) ||
            (rc = cuda_fail(cudaMemsetAsync(bt->d_k, 0, sizeof(int), main_st), "memset")))
            return rc;
    }
    batch_dots_kernel<<<nc, kGsThreads, 0, main_st>>>(W, 0, 0, nullptr, W, bt->d_inst, bt->d_chunks, nullptr, total,
                                                      bt->red);
    batch_norm_init_kernel<<<(B + 3) / 4, 128, 0, main_st>>>(bt->red, bt->d_inst_chunks, B, bt->lz, bt->lz_stride,
                                                             L.status, bt->d_active);
    batch_scale_kernel<<<nc, kGsThreads, 0, main_st>>>(W, bt->d_inst, bt->d_chunks, nullptr, total, bt->lz,
                                                       bt->lz_stride, L.status, ST_INV_NW, V, ld, 0, nullptr, vf,
                                                       bt->selfc, bt->src, fp64);
    count_launches(3);
    // everything of an iteration but the host's reading of n_active
    auto iteration = [&](int k, bool scale) {
        cudaStream_t st = bt->stream;
        int r = batch_product(bt, pos, vf, nullptr, w, bt->d_active, true);
        if (r) return r;
        batch_dots_kernel<<<nc, kGsThreads, 0, st>>>(V, ld, k, d_k, w, bt->d_inst, bt->d_chunks, bt->d_active, total,
                                                     bt->red);
        batch_project_kernel<<<nc, kGsThreads, 0, st>>>(V, ld, k, d_k, w, bt->d_inst, bt->d_chunks, bt->d_active, total,
                                                        bt->red, bt->lz, bt->lz_stride, L.c1, red2, nullptr);
        batch_project_kernel<<<nc, kGsThreads, 0, st>>>(V, ld, k, d_k, w, bt->d_inst, bt->d_chunks, bt->d_active, total,
                                                        red2, bt->lz, bt->lz_stride, L.c2, nullptr, bt->norm2);
        if ((r = cuda_fail(cudaMemsetAsync(bt->d_nactive, 0, sizeof(int), st), "memset"))) return r;
        batch_tail_kernel<<<B, kTailThreads, 0, st>>>(bt->lz, bt->lz_stride, L, k, d_k, tol, bt->norm2,
                                                      bt->d_inst_chunks, bt->nodes, bt->d_active, bt->d_nactive);
        count_launches(4);
        if (scale) {
            batch_scale_kernel<<<nc, kGsThreads, 0, st>>>(w, bt->d_inst, bt->d_chunks, bt->d_active, total, bt->lz,
                                                          bt->lz_stride, L.status, ST_INV_BETA, V, ld, k + 1, d_k, vf,
                                                          bt->selfc, bt->src, fp64);
            count_launches(1);
        }
        if (graph) {
            batch_iter_kernel<<<1, 1, 0, st>>>(loop, max_iter, bt->d_nactive, bt->d_k, bt->d_loops);
            count_launches(1);
        }
        return cuda_fail(cudaGetLastError(), "batch lanczos kernels");
    };
    if (graph) {
        if ((rc = iteration(0, max_iter > 1))) return rc;
        if (max_iter > 1) {
            if ((rc = graph_begin_cond(main_st, bt->body, loop, cudaGraphCondTypeWhile))) return rc;
            bt->stream = bt->body;
            const uint64_t before = rpb_launch_count();
            rc = iteration(0, true);
            bt->body_launches = (int)(rpb_launch_count() - before);
            cudaGraph_t body_graph = nullptr;  // owned by the node
            const int erc = cuda_fail(cudaStreamEndCapture(bt->body, &body_graph), "body capture end");
            bt->stream = main_st;
            if (rc || (rc = erc)) return rc;
        }
    }
    for (int k = 0; k < max_iter && !graph; ++k) {
        if ((rc = iteration(k, k + 1 < max_iter)) ||
            (rc = cuda_fail(cudaMemcpyAsync(bt->h_nactive, bt->d_nactive, sizeof(int), cudaMemcpyDeviceToHost, main_st),
                            "n_active copy")) ||
            (rc = cuda_fail(cudaStreamSynchronize(main_st), "batch lanczos iteration")))
            return rc;
        if (*bt->h_nactive == 0) break;
    }
    batch_combine_kernel<<<ge, 256, 0, main_st>>>(V, ld, bt->d_inst_of, total, bt->lz, bt->lz_stride, L, g);
    count_launches(1);
    if (graph) return cuda_fail(cudaGetLastError(), "batch lanczos kernels");
    if ((rc = cuda_fail(cudaMemcpyAsync(bt->h_lz, bt->lz, (size_t)B * bt->lz_stride * sizeof(double),
                                        cudaMemcpyDeviceToHost, main_st),
                        "status copy")))
        return rc;
    return cuda_fail(cudaStreamSynchronize(main_st), "batch lanczos");
}

// After a step replayed from a CUDA graph: advance every instance's step counter and count the
// instances whose Lanczos did not converge within the fixed iteration count.
__global__ void batch_advance_kernel(InstDesc *__restrict__ inst, int B, const int *__restrict__ active,
                                     unsigned long long *__restrict__ unconv)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    inst[b].step += 1u;
    inst[b].first = 0;
    if (active[b]) atomicAdd(unconv, 1ull);
}

// One AB step of the packed batch (state in vec[V_POS], vec[V_UP]).  graph: see batch_lanczos; the
// step then also advances the device-side step counters.
static int batch_step_body(rpb_batch *bt, double dt, double delta, double tol, int max_iter,
                           const rpb_force_params *fp, bool graph)
{
    cudaStream_t st = bt->stream;
    const int64_t total = bt->total, n = 3 * total;
    double **v = bt->vec;
    const int ge = grid_for(n, bt->num_sms);
    int rc;
    const double a = bt->p.a;
    const double rcut = (2.0 * a + kForceCutoffB * fp->b) * 1.01 + 0.01 * a;
    if ((rc = cell_forces<InstDesc>(st, cell_lists(bt->cells, bt->max_total), v[V_POS], total, a, fp->weight, fp->U0, fp->b,
                                    rcut, 2.0 * a + kFarB * fp->b, bt->d_inst, bt->d_inst_of, v[V_F])))
        return rc;
    batch_fill3_kernel<<<ge, 256, 0, st>>>(v[V_T], total, fp->torque[0], fp->torque[1], fp->torque[2]);
    count_launches(1);
    if ((rc = batch_product(bt, v[V_POS], v[V_F], v[V_T], v[V_UN], nullptr))) return rc;
    batch_philox_kernel<<<dim3(bt->nchunks, 2), 256, 0, st>>>(bt->d_inst, bt->d_chunks, total, v[V_W], v[V_WT]);
    count_launches(1);
    if ((rc = batch_lanczos(bt, v[V_POS], v[V_W], v[V_G], tol, max_iter, graph))) return rc;
    // RFD: two products at the displaced configurations, regularised anew
    batch_displace_kernel<<<ge, 256, 0, st>>>(v[V_POS], v[V_WT], n, 0.5 * delta, v[V_PA], v[V_PB]);
    count_launches(1);
    if ((rc = batch_product(bt, v[V_PA], v[V_WT], nullptr, v[V_DRIFT], nullptr))) return rc;
    if ((rc = batch_product(bt, v[V_PB], v[V_WT], nullptr, v[V_WORK], nullptr))) return rc;
    batch_rfd_combine_kernel<<<ge, 256, 0, st>>>(v[V_DRIFT], v[V_WORK], n, bt->p.kT / delta);
    batch_ab_update_kernel<<<ge, 256, 0, st>>>(bt->d_inst, bt->d_inst_of, total, v[V_POS], v[V_UP], v[V_UN], v[V_G],
                                               v[V_DRIFT], dt, sqrt(2.0 * bt->p.kT * dt));
    count_launches(2);
    if (graph) {
        batch_advance_kernel<<<(bt->B + 127) / 128, 128, 0, st>>>(bt->d_inst, bt->B, bt->d_active, bt->d_unconv);
        count_launches(1);
    }
    return cuda_fail(cudaGetLastError(), "batch step kernels");
}

// Per-instance statistics from the host copy of the Lanczos states; returns how many did not converge.
static int batch_read_stats(rpb_batch *bt, double tol, rpb_step_stats *stats)
{
    const LzLayout L(bt->max_iter);
    int noconv = 0;
    for (int b = 0; b < bt->B; ++b) {
        const double *stb = bt->h_lz + (size_t)b * bt->lz_stride + L.status;
        const int conv = stb[7] != 0.0;
        noconv += !conv && tol > 0.0;
        if (stats) {
            stats[b].lanczos_iters = (int)stb[6];
            stats[b].lanczos_err = stb[ST_EPS];
            stats[b].converged = conv;
        }
    }
    return noconv;
}

// nsteps AB steps of the batch: one gather, one launch of a CUDA graph whose WHILE node runs a step
// (converged instances masked) nsteps times without host
// synchronisation, one scatter.
static int batch_run_impl(rpb_batch *bt, int B, const int64_t *N, double *const *pos, double *const *U_prev,
                          const int64_t *steps, const uint64_t *seeds, int nsteps, double dt, double delta, double tol,
                          int lanczos_iters, const rpb_force_params *fp, rpb_step_stats *stats, int64_t *unconverged)
{
    int rc;
    if ((rc = batch_setup(bt, B, N, steps, seeds, pos, U_prev, nullptr, nullptr))) return rc;
    cudaStream_t st = bt->stream;
    double **v = bt->vec;
    if ((rc = batch_gather(bt, 0, v[V_POS], 0)) || (rc = batch_gather(bt, 1, v[V_UP], 0))) return rc;
    if ((rc = cuda_fail(cudaMemsetAsync(bt->d_unconv, 0, sizeof(unsigned long long), st), "memset")) ||
        (rc = cuda_fail(cudaMemsetAsync(bt->d_loops, 0, sizeof(unsigned long long), st), "memset")))
        return rc;
    bt->body_launches = 0;
    int per_step = 0;
    if (nsteps > 0) {
        // one graph launch for all nsteps: a WHILE node whose body is a step, counted down on the device
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        graph_loop_init_kernel<<<1, 1, 0, st>>>(bt->d_left, nsteps);
        count_launches(1);
        const uint64_t before = rpb_launch_count();
        if ((rc = cuda_fail(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal), "begin capture"))) return rc;
        cudaGraphConditionalHandle loop_h = 0;
        int brc = graph_begin_loop(st, bt->loop, &loop_h);
        if (!brc) {
            bt->stream = bt->loop;
            brc = batch_step_body(bt, dt, delta, tol, lanczos_iters, fp, true);
            if (!brc) {
                graph_loop_tail_kernel<<<1, 1, 0, bt->loop>>>(bt->d_left, loop_h);
                count_launches(1);
                brc = cuda_fail(cudaGetLastError(), "loop kernel");
            }
            bt->stream = st;
            cudaGraph_t loop_graph = nullptr;  // owned by the WHILE node
            const cudaError_t el = cudaStreamEndCapture(bt->loop, &loop_graph);
            if (!brc && el != cudaSuccess) brc = cuda_fail(el, "loop body capture end");
        }
        const cudaError_t ec = cudaStreamEndCapture(st, &graph);
        per_step = (int)(rpb_launch_count() - before);
        count_launches(-per_step);  // captured, not executed (counted below from the runs)
        if (brc) {
            if (graph) cudaGraphDestroy(graph);
            cudaGetLastError();
            return brc;
        }
        if ((rc = cuda_fail(ec, "end capture"))) return rc;
        if ((rc = cuda_fail(cudaGraphInstantiate(&exec, graph, 0), "graph instantiate"))) {
            cudaGraphDestroy(graph);
            return rc;
        }
        rc = cuda_fail(cudaGraphLaunch(exec, st), "graph launch");
        cudaGraphExecDestroy(exec);
        cudaGraphDestroy(graph);
        if (rc) return rc;
    }
    if ((rc = batch_gather(bt, 0, v[V_POS], 1)) || (rc = batch_gather(bt, 1, v[V_UP], 1))) return rc;
    if ((rc = cuda_fail(cudaMemcpyAsync(bt->h_lz, bt->lz, (size_t)B * bt->lz_stride * sizeof(double),
                                        cudaMemcpyDeviceToHost, st),
                        "status copy")) ||
        (rc = cuda_fail(cudaMemcpyAsync(bt->h_unconv, bt->d_unconv, sizeof(unsigned long long), cudaMemcpyDeviceToHost,
                                        st),
                        "count copy")) ||
        (rc = cuda_fail(cudaMemcpyAsync(bt->h_loops, bt->d_loops, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st),
                        "iteration count copy")) ||
        (rc = cuda_fail(cudaStreamSynchronize(st), "batch run")))
        return rc;
    if (nsteps > 0)  // kernels executed: the unconditional part every step, the loop's body once per run of it
        count_launches((int)((int64_t)(per_step - bt->body_launches) * nsteps +
                             (int64_t)bt->body_launches * (int64_t)*bt->h_loops));
    batch_read_stats(bt, tol, stats);
    if (unconverged) *unconverged = (int64_t)*bt->h_unconv;
    if (*bt->h_unconv && tol > 0.0) {
        set_error("lanczos: %llu instance-step(s) did not converge in %d iterations", *bt->h_unconv, lanczos_iters);
        return RPB_ENOCONV;
    }
    return RPB_OK;
}

}  // namespace rpb

extern "C" {

int rpb_batch_create(rpb_batch **out, const rpb_params *p, int64_t max_total_N, int max_B, int max_iter, void *stream)
{
    if (!out || !p) {
        set_error("null argument to rpb_batch_create");
        return RPB_EINVAL;
    }
    *out = nullptr;
    if (!(p->a > 0.0) || !(p->eta > 0.0) || !(p->kT >= 0.0) || (p->precision != RPB_FP64 && p->precision != RPB_FP32) ||
        p->wall != 1) {
        set_error("bad parameters (batch contexts need precision RPB_FP64/RPB_FP32 and wall = 1)");
        return RPB_EINVAL;
    }
    if (max_total_N <= 0 || max_total_N > (int64_t)1 << 28 || max_B < 1 || max_B > (1 << 20) || max_iter < 1 ||
        max_iter > kMaxIter) {
        set_error("bad batch limits (max_total_N=%lld max_B=%d max_iter=%d)", (long long)max_total_N, max_B, max_iter);
        return RPB_EINVAL;
    }
    rpb_batch *bt = new (std::nothrow) rpb_batch();
    if (!bt) {
        set_error("host allocation failed");
        return RPB_ENOMEM;
    }
    bt->p = *p;
    bt->max_total = max_total_N;
    bt->max_B = max_B;
    bt->max_iter = max_iter;
    bt->stream = (cudaStream_t)stream;
    {
        // RPB_FP32_BATCH_SYM=0: float32 products by the one-way kernel instead of the symmetric pass
        const char *v = getenv("RPB_FP32_BATCH_SYM");
        bt->sym_env = !(v && strcmp(v, "0") == 0);
        bt->sym_enabled = p->precision == RPB_FP32 && bt->sym_env;
    }
    int dev = 0;
    if (cuda_fail(cudaGetDevice(&dev), "cudaGetDevice") ||
        cuda_fail(cudaDeviceGetAttribute(&bt->num_sms, cudaDevAttrMultiProcessorCount, dev), "SM count")) {
        delete bt;
        return RPB_ECUDA;
    }
    const LzLayout L(max_iter);
    bt->lz_stride = L.total;
    const size_t vb = (size_t)3 * max_total_N * sizeof(double);
    const int64_t max_blocks = max_total_N / kTile + max_B + 1, max_chunks = max_total_N / kGsChunk + max_B + 1;
    bool ok = cudaMalloc(&bt->d_inst, max_B * sizeof(InstDesc)) == cudaSuccess &&
              cudaMalloc(&bt->d_blocks, max_blocks * sizeof(BlockDesc)) == cudaSuccess &&
              cudaMalloc(&bt->d_inst_of, max_total_N * sizeof(int)) == cudaSuccess &&
              cudaMalloc(&bt->d_active, max_B * sizeof(int)) == cudaSuccess &&
              cudaMalloc(&bt->d_nactive, sizeof(int)) == cudaSuccess &&
              cudaMalloc(&bt->src, max_total_N * sizeof(SrcF64)) == cudaSuccess &&
              cudaMalloc(&bt->V, vb * (max_iter + 1)) == cudaSuccess &&
              cudaMalloc(&bt->lz, (size_t)max_B * L.total * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&bt->red, (size_t)2 * max_iter * max_chunks * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&bt->norm2, (size_t)max_chunks * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&bt->d_chunks, max_chunks * sizeof(ChunkDesc)) == cudaSuccess &&
              cudaMalloc(&bt->d_inst_chunks, max_B * sizeof(int2)) == cudaSuccess &&
              cudaMallocHost(&bt->h_chunks, max_chunks * sizeof(ChunkDesc)) == cudaSuccess &&
              cudaMallocHost(&bt->h_inst_chunks, max_B * sizeof(int2)) == cudaSuccess &&
              cudaMalloc(&bt->selfc, (size_t)4 * max_total_N * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&bt->cells, cell_lists_bytes(max_total_N)) == cudaSuccess &&
              cudaMalloc(&bt->nodes, 2 * kSqrtNodes * sizeof(double)) == cudaSuccess &&
              cudaMallocHost(&bt->h_inst, max_B * sizeof(InstDesc)) == cudaSuccess &&
              cudaMallocHost(&bt->h_blocks, max_blocks * sizeof(BlockDesc)) == cudaSuccess &&
              cudaMallocHost(&bt->h_nactive, sizeof(int)) == cudaSuccess &&
              cudaMallocHost(&bt->h_lz, (size_t)max_B * L.total * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&bt->d_unconv, sizeof(unsigned long long)) == cudaSuccess &&
              cudaMallocHost(&bt->h_unconv, sizeof(unsigned long long)) == cudaSuccess &&
              cudaStreamCreateWithFlags(&bt->cap, cudaStreamNonBlocking) == cudaSuccess &&
              cudaStreamCreateWithFlags(&bt->loop, cudaStreamNonBlocking) == cudaSuccess &&
              cudaMalloc(&bt->d_left, sizeof(int)) == cudaSuccess &&
              cudaStreamCreateWithFlags(&bt->body, cudaStreamNonBlocking) == cudaSuccess &&
              cudaMalloc(&bt->d_k, sizeof(int)) == cudaSuccess &&
              cudaMalloc(&bt->d_loops, sizeof(unsigned long long)) == cudaSuccess &&
              cudaMallocHost(&bt->h_loops, sizeof(unsigned long long)) == cudaSuccess &&
              cudaEventCreateWithFlags(&bt->join, cudaEventDisableTiming) == cudaSuccess;
    for (double *&v : bt->vec) ok = ok && cudaMalloc(&v, vb) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        set_error("batch scratch allocation failed (max_total_N=%lld, max_B=%d)", (long long)max_total_N, max_B);
        batch_free(bt);
        delete bt;
        return RPB_ENOMEM;
    }
    if (cuda_fail(cudaMemsetAsync(bt->lz, 0, (size_t)max_B * L.total * sizeof(double), bt->stream), "memset") ||
        upload_sqrt_nodes(bt->nodes, bt->stream)) {
        batch_free(bt);
        delete bt;
        return RPB_ECUDA;
    }
    *out = bt;
    return RPB_OK;
}

int rpb_batch_destroy(rpb_batch *bt)
{
    if (!bt) return RPB_OK;
    const int rc = cuda_fail(cudaStreamSynchronize(bt->stream), "rpb_batch_destroy sync");
    batch_free(bt);
    delete bt;
    return rc;
}

int rpb_batch_set_stream(rpb_batch *bt, void *stream)
{
    if (!bt) {
        set_error("null batch");
        return RPB_EINVAL;
    }
    bt->stream = (cudaStream_t)stream;
    return RPB_OK;
}

int rpb_batch_set_tiles(rpb_batch *bt, const rpb_batch_tiles *t)
{
    if (!bt) {
        set_error("null batch context");
        return RPB_EINVAL;
    }
    rpb_batch_tiles d = {8, 5, bt->sym_env};
    if (!t) t = &d;
    if (t->seg_tiles < 1 || t->seg_tiles > 64 || (t->ctas_per_sm != 4 && t->ctas_per_sm != 5) ||
        (t->symmetric != 0 && t->symmetric != 1)) {
        set_error("bad tile schedule (seg_tiles=%d ctas_per_sm=%d symmetric=%d)", t->seg_tiles, t->ctas_per_sm,
                  t->symmetric);
        return RPB_EINVAL;
    }
    bt->seg_tiles = t->seg_tiles;
    bt->sym.tt_minb = t->ctas_per_sm;
    bt->sym_enabled = bt->p.precision == RPB_FP32 && t->symmetric;
    bt->sym_ok = false;  // planned again by the next call
    return RPB_OK;
}

int rpb_batch_get_tiles(rpb_batch *bt, rpb_batch_tiles *t)
{
    if (!bt || !t) {
        set_error("null argument to rpb_batch_get_tiles");
        return RPB_EINVAL;
    }
    t->seg_tiles = bt->seg_tiles;
    t->ctas_per_sm = bt->sym.tt_minb;
    t->symmetric = bt->sym_enabled ? 1 : 0;
    return RPB_OK;
}

int rpb_batch_tune(rpb_batch *bt, int B, const int64_t *N, const double *const *pos, int reps, rpb_batch_tiles *best,
                   int max_cand, rpb_batch_tiles *cand, double *cand_ms, int *ncand)
{
    if (!bt || !N || !pos || reps < 1) {
        set_error("bad argument to rpb_batch_tune");
        return RPB_EINVAL;
    }
    for (int b = 0; b < B && b < bt->max_B; ++b)
        if (!pos[b]) {
            set_error("instance %d: null pos", b);
            return RPB_EINVAL;
        }
    int rc;
    // candidates: the symmetric pass at every run length and occupancy, and the one-way kernel
    std::vector<rpb_batch_tiles> cs;
    if (bt->p.precision == RPB_FP32) {
        for (int seg : {4, 8, 16, 32})
            for (int minb : {4, 5}) cs.push_back(rpb_batch_tiles{seg, minb, 1});
        cs.push_back(rpb_batch_tiles{8, 5, 0});
    } else {
        cs.push_back(rpb_batch_tiles{8, 5, 0});  // float64: the one-way kernel only
    }
    if ((rc = rpb_batch_set_tiles(bt, &cs[0])) ||
        (rc = batch_setup(bt, B, N, nullptr, nullptr, const_cast<double *const *>(pos), nullptr, nullptr, nullptr)))
        return rc;
    cudaStream_t st = bt->stream;
    double **v = bt->vec;
    const int ge = grid_for(3 * bt->total, bt->num_sms);
    if ((rc = batch_gather(bt, 0, v[V_POS], 0))) return rc;
    batch_fill3_kernel<<<ge, 256, 0, st>>>(v[V_F], bt->total, 0.0, 0.0, -1.0);
    batch_fill3_kernel<<<ge, 256, 0, st>>>(v[V_T], bt->total, 0.0, 1.0, 0.0);
    count_launches(2);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if ((rc = cuda_fail(cudaEventCreate(&e0), "event")) || (rc = cuda_fail(cudaEventCreate(&e1), "event"))) {
        if (e0) cudaEventDestroy(e0);
        return rc;
    }
    double best_cost = -1.0;
    size_t best_k = 0;
    for (size_t k = 0; k < cs.size() && !rc; ++k) {
        if ((rc = rpb_batch_set_tiles(bt, &cs[k]))) break;
        if (bt->sym_enabled && (rc = batch_sym_plan(bt->sym, B, N, st, &bt->sym_ok, bt->seg_tiles))) break;
        // a step makes about ten translation-translation products per fused one
        float t_tt = 0.f, t_fu = 0.f;
        for (int pass = 0; pass < 2 && !rc; ++pass) {  // pass 0 warms up
            for (int which = 0; which < 2 && !rc; ++which) {
                const double *T = which ? v[V_T] : nullptr;
                cudaEventRecord(e0, st);
                for (int r = 0; r < reps && !rc; ++r) rc = batch_product(bt, v[V_POS], v[V_F], T, v[V_UN], nullptr);
                cudaEventRecord(e1, st);
                if (!rc) rc = cuda_fail(cudaEventSynchronize(e1), "tune timing");
                float ms = 0.f;
                if (!rc) rc = cuda_fail(cudaEventElapsedTime(&ms, e0, e1), "tune timing");
                if (pass == 1) (which ? t_fu : t_tt) = ms / reps;
            }
        }
        const double cost = 10.0 * t_tt + t_fu;
        if (cand && cand_ms && (int)k < max_cand) {
            cand[k] = cs[k];
            cand_ms[k] = cost;
        }
        if (!rc && (best_cost < 0.0 || cost < best_cost)) {
            best_cost = cost;
            best_k = k;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc) return rc;
    if (ncand) *ncand = (int)cs.size();
    if (best) *best = cs[best_k];
    return rpb_batch_set_tiles(bt, &cs[best_k]);
}

int rpb_batch_mobility_apply(rpb_batch *bt, int B, const int64_t *N, const double *const *pos, const double *const *F,
                             const double *const *T, double *const *U)
{
    if (!bt || !N || !pos || !U) {
        set_error("null argument to rpb_batch_mobility_apply");
        return RPB_EINVAL;
    }
    for (int b = 0; b < B && b < bt->max_B; ++b)
        if (!pos[b] || !U[b]) {
            set_error("instance %d: null pos or U", b);
            return RPB_EINVAL;
        }
    int rc;
    if ((rc = batch_setup(bt, B, N, nullptr, nullptr, const_cast<double *const *>(pos), const_cast<double *const *>(F),
                          T, U)))
        return rc;
    double *P = bt->vec[V_POS], *Fp = F ? bt->vec[V_F] : nullptr, *Tp = T ? bt->vec[V_T] : nullptr, *Up = bt->vec[V_UN];
    if ((rc = batch_gather(bt, 0, P, 0))) return rc;
    if (Fp && (rc = batch_gather(bt, 1, Fp, 0))) return rc;
    if (Tp && (rc = batch_gather(bt, 2, Tp, 0))) return rc;
    if (!Fp && !Tp) {
        if ((rc = cuda_fail(cudaMemsetAsync(Up, 0, 3 * bt->total * sizeof(double), bt->stream), "memset"))) return rc;
    } else if ((rc = batch_product(bt, P, Fp, Tp, Up, nullptr))) {
        return rc;
    }
    return batch_gather(bt, 3, Up, 1);
}

int rpb_batch_ab_step(rpb_batch *bt, int B, const int64_t *N, double *const *pos, double *const *U_prev,
                      const int64_t *steps, const uint64_t *seeds, double dt, double delta, double tol, int max_iter,
                      const rpb_force_params *fp, rpb_step_stats *stats)
{
    if (!bt || !N || !pos || !U_prev || !steps || !seeds || !fp) {
        set_error("null argument to rpb_batch_ab_step");
        return RPB_EINVAL;
    }
    if (!(fp->b > 0.0) || !(dt > 0.0) || !(delta > 0.0) || max_iter < 1 || max_iter > bt->max_iter) {
        set_error("bad step arguments (dt=%g delta=%g max_iter=%d)", dt, delta, max_iter);
        return RPB_EINVAL;
    }
    for (int b = 0; b < B && b < bt->max_B; ++b)
        if (!pos[b] || !U_prev[b] || steps[b] < 0 || steps[b] > 0xffffffffLL) {
            set_error("instance %d: null buffer or bad step", b);
            return RPB_EINVAL;
        }
    int rc;
    if ((rc = batch_setup(bt, B, N, steps, seeds, pos, U_prev, nullptr, nullptr))) return rc;
    double **v = bt->vec;
    if ((rc = batch_gather(bt, 0, v[V_POS], 0)) || (rc = batch_gather(bt, 1, v[V_UP], 0))) return rc;
    if ((rc = batch_step_body(bt, dt, delta, tol, max_iter, fp, false))) return rc;
    if ((rc = batch_gather(bt, 0, v[V_POS], 1)) || (rc = batch_gather(bt, 1, v[V_UP], 1))) return rc;
    const int noconv = batch_read_stats(bt, tol, stats);
    if (noconv) {
        set_error("lanczos: %d instance(s) did not converge in %d iterations", noconv, max_iter);
        return RPB_ENOCONV;
    }
    return RPB_OK;
}

int rpb_batch_run(rpb_batch *bt, int B, const int64_t *N, double *const *pos, double *const *U_prev,
                  const int64_t *steps, const uint64_t *seeds, int nsteps, double dt, double delta, double tol,
                  int lanczos_iters, const rpb_force_params *fp, rpb_step_stats *stats, int64_t *unconverged)
{
    if (!bt || !N || !pos || !U_prev || !steps || !seeds || !fp) {
        set_error("null argument to rpb_batch_run");
        return RPB_EINVAL;
    }
    if (!(fp->b > 0.0) || !(dt > 0.0) || !(delta > 0.0) || lanczos_iters < 1 || lanczos_iters > bt->max_iter ||
        nsteps < 0) {
        set_error("bad run arguments (dt=%g delta=%g lanczos_iters=%d nsteps=%d)", dt, delta, lanczos_iters, nsteps);
        return RPB_EINVAL;
    }
    for (int b = 0; b < B && b < bt->max_B; ++b)
        if (!pos[b] || !U_prev[b] || steps[b] < 0 || steps[b] + nsteps > 0xffffffffLL) {
            set_error("instance %d: null buffer or bad step", b);
            return RPB_EINVAL;
        }
    // Everything runs on the batch's own capture stream, ordered after the caller's stream.
    cudaStream_t user = bt->stream;
    int rc;
    if ((rc = cuda_fail(cudaEventRecord(bt->join, user), "event record")) ||
        (rc = cuda_fail(cudaStreamWaitEvent(bt->cap, bt->join, 0), "stream wait")))
        return rc;
    bt->stream = bt->cap;
    rc = batch_run_impl(bt, B, N, pos, U_prev, steps, seeds, nsteps, dt, delta, tol, lanczos_iters, fp, stats,
                        unconverged);
    bt->stream = user;
    return rc;
}

}  // extern "C"
