// pair.cu -- the all-pairs Rotne-Prager-Blake product U = M_tt F + M_tr T (and the force kernel).
//
// Mobility (Sec. II.B Eq. mobilityDifferential / mobilityOverlap, Sec. III Eq.
// mobilityDifferentialTR, Appendix A Eq. effMob):
//   M_ij = s_i s_j Mtilde(q~_i, q~_j),  s = H0(z/a),  q~ = (x, y, max(z, a)),
//   Mtilde = free-space RPY (overlap branch for r < 2a) + wall correction.
// The wall correction is the Faxen-operated image system of Blake's half-space Green's function,
// written in closed form on the basis {I, e e, e z, z e, z z} (translation) and
// {T x e, T x z, e (z x e).T, z (z x e).T} (rotation), with R = x_i - x_j* (source mirrored in
// the wall), e = R/|R|, t = z~_j/|R|, s = a^2/|R|^2.  The coefficients were obtained by
// decomposing the Faxen-operated image tensors onto that basis; they reproduce the published
// near-wall self mobilities 1 - 9/(16h) + 1/(8h^3) - 1/(16h^5) and 1 - 9/(8h) + 1/(2h^3) - 1/(8h^5).
//
// Kernel design (GB300, CUDA cores -- the pair work is not a dense contraction):
//   - one target per thread, 128 targets per block, sources staged 128 at a time in shared
//     memory (every thread reads the same source: broadcast, no bank conflicts);
//   - the source range is split into chunks (grid.y) so that small N still fills all SMs; each
//     (target block, chunk) writes a float64 partial, summed in fixed order by the reduce kernel
//     (deterministic, no atomics);
//   - the self pair (j == i) is excluded from the pair loop (only the block's diagonal tile pays
//     for the test) and added in float64 by the reduce kernel, which also applies s_i/(8 pi eta);
//   - float32 mode: positions split x = x_hi + x_lo (two floats), so near-pair offsets keep float32
//     relative accuracy anywhere in a large box; per-tile float32 sums are added with Kahan
//     compensation.
// The float64 products with forces take the symmetric pass of pair64.cu; pair_f64_kernel serves torque-only
// products, row ranges, the allocation-free product and contexts too large for that pass's scratch.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <vector>

#include <cooperative_groups.h>

#include "cells.cuh"
#include "float_sums.h"
#include "grid_plan.h"
#include "pair_math.cuh"
#include "sym_schedule.h"

namespace cg = cooperative_groups;

namespace rpb {

// ------------------------------------------------------------------ packing
__global__ void pack_f32_kernel(const double *__restrict__ pos, const double *__restrict__ F,
                                const double *__restrict__ T, int N, double a, int wall, SrcF32 *__restrict__ out,
                                SelfCoefs sc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double x = pos[i], y = pos[N + i], z = pos[2 * N + i];
    const double s = wall ? H0(z / a) : 1.0;
    const float xh = (float)x, yh = (float)y;
    SrcF32 o;
    o.p = make_float4(xh, yh, (float)(x - (double)xh), (float)(y - (double)yh));
    o.f = make_float4((float)(wall ? fmax(z, a) : z), F ? (float)(s * F[i]) : 0.f, F ? (float)(s * F[N + i]) : 0.f,
                      F ? (float)(s * F[2 * N + i]) : 0.f);
    o.t = make_float4(T ? (float)(s * T[i]) : 0.f, T ? (float)(s * T[N + i]) : 0.f, T ? (float)(s * T[2 * N + i]) : 0.f,
                      0.f);
    out[i] = o;
    if (sc.s) store_self_coefs(sc, i, s, wall ? fmax(z, a) : z, wall);
}

// Second right-hand side of the two-RHS symmetric pass: s_j P_j as float32 (x, y, z, 0).
__global__ void pack_rhs2_kernel(const double *__restrict__ pos, const double *__restrict__ P, int N, double a,
                                 float4 *__restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double s = H0(pos[2 * N + i] / a);
    out[i] = make_float4((float)(s * P[i]), (float)(s * P[N + i]), (float)(s * P[2 * N + i]), 0.f);
}

__global__ void pack_f64_kernel(const double *__restrict__ pos, const double *__restrict__ F,
                                const double *__restrict__ T, int N, double a, int wall, SrcF64 *__restrict__ out,
                                SelfCoefs sc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double z = pos[2 * N + i];
    const double s = wall ? H0(z / a) : 1.0;
    SrcF64 o;
    o.p = make_double2(pos[i], pos[N + i]);
    o.q = make_double2(wall ? fmax(z, a) : z, F ? s * F[i] : 0.0);
    o.r = make_double2(F ? s * F[N + i] : 0.0, F ? s * F[2 * N + i] : 0.0);
    o.s = make_double2(T ? s * T[i] : 0.0, T ? s * T[N + i] : 0.0);
    o.u = make_double2(T ? s * T[2 * N + i] : 0.0, 0.0);
    out[i] = o;
    if (sc.s) store_self_coefs(sc, i, s, wall ? fmax(z, a) : z, wall);
}

// The self coefficients of a context's products, or none (the row-range and allocation-free products
// evaluate their self terms themselves).
SelfCoefs self_coefs(const rpb_ctx *ctx, int64_t N)
{
    return SelfCoefs{ctx->ws.selfc, N, 1.0 / (8.0 * kPi * ctx->p.eta), make_consts<double>(ctx->p.a)};
}
static SelfCoefs no_self_coefs()
{
    return SelfCoefs{nullptr, 0, 0.0, PairConsts<double>{}};
}

// A product enqueued before the host knows whether the Lanczos iteration before it stopped: stop is that
// iteration's status word, and the pair kernels leave when it is set (null: none to ask).  They test it after their
// first loads, beside which it arrives.  A step of 10000 spheres 2145 -> 2095 us, a float64 solve of 2000 1164 ->
// 1122 (there the stream waited for the host); a short discarded product mostly ran while the host answered.
__device__ __forceinline__ bool stopped(const double *stop)
{
    return stop && *stop != 0.0;
}

// ------------------------------------------------------------------ pair kernels
// grid = (ceil(N/128), splits); block (bx, by) covers targets [128 bx, 128 bx + 128) and sources
// [by chunk, (by + 1) chunk); chunk is a multiple of 128, so the tile holding the block's own
// targets (where j == i can occur) is the one starting at 128 bx.
template <bool TORQUE, bool WALL = true>
__global__ void __launch_bounds__(kPairThreads) pair_f32_kernel(const SrcF32 *__restrict__ src, int N, int chunk,
                                                                 PairConsts<float> c, double *__restrict__ part,
                                                                 const double *__restrict__ stop = nullptr)
{
    const bool quit = stopped(stop);
    __shared__ float4 sp[kTile];
    __shared__ float4 sf[kTile];
    __shared__ float4 st[TORQUE ? kTile : 1];
    const int tid = threadIdx.x;
    const int i = blockIdx.x * kPairThreads + tid;
    const int j0 = blockIdx.y * chunk;
    const int j1 = min(N, j0 + chunk);
    float4 tp = make_float4(0.f, 0.f, 0.f, 0.f);
    float tz = 1.f;
    if (i < N) {
        tp = src[i].p;
        tz = src[i].f.x;
    }
    float sx = 0.f, sy = 0.f, sz = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
    const int diag = blockIdx.x * kTile;
    for (int base = j0; base < j1; base += kTile) {
        const int j = base + tid;
        if (j < j1) {
            sp[tid] = src[j].p;
            sf[tid] = src[j].f;
            if (TORQUE) st[tid] = src[j].t;
        }
        __syncthreads();
        if (quit) return;
        const int cnt = min(kTile, j1 - base);
        float ux = 0.f, uy = 0.f, uz = 0.f;
        if (base != diag) {
#pragma unroll 4
            for (int k = 0; k < cnt; ++k) {
                const float4 p = sp[k];
                const float4 f = sf[k];
                const float4 q = TORQUE ? st[k] : make_float4(0.f, 0.f, 0.f, 0.f);
                const float rx = (tp.x - p.x) + (tp.z - p.z);
                const float ry = (tp.y - p.y) + (tp.w - p.w);
                pair_velocity_f32<TORQUE, WALL>(rx, ry, tz, f.x, f.y, f.z, f.w, q.x, q.y, q.z, c, ux, uy, uz);
            }
        } else {
            for (int k = 0; k < cnt; ++k) {
                const float4 p = sp[k];
                const float4 f = sf[k];
                const float4 q = TORQUE ? st[k] : make_float4(0.f, 0.f, 0.f, 0.f);
                const float rx = (tp.x - p.x) + (tp.z - p.z);
                const float ry = (tp.y - p.y) + (tp.w - p.w);
                float dx = 0.f, dy = 0.f, dz = 0.f;
                pair_velocity_f32<TORQUE, WALL>(rx, ry, tz, f.x, f.y, f.z, f.w, q.x, q.y, q.z, c, dx, dy, dz);
                if (k != tid) {
                    ux += dx;
                    uy += dy;
                    uz += dz;
                }
            }
        }
        // compensated (Kahan) accumulation of the tile sums
        {
            float yv = ux - cx, tv = sx + yv;
            cx = (tv - sx) - yv;
            sx = tv;
            yv = uy - cy;
            tv = sy + yv;
            cy = (tv - sy) - yv;
            sy = tv;
            yv = uz - cz;
            tv = sz + yv;
            cz = (tv - sz) - yv;
            sz = tv;
        }
        __syncthreads();
    }
    if (i < N) {
        const size_t o = (size_t)blockIdx.y * 3 * N;
        part[o + i] = (double)sx - (double)cx;
        part[o + N + i] = (double)sy - (double)cy;
        part[o + 2 * N + i] = (double)sz - (double)cz;
    }
}

// Float32 pair pass without the wall for chunks of several tiles (more than 2048 spheres): two targets per
// lane with packed arithmetic, every source read by the whole warp, because the scalar kernel is bound by
// issue (two targets' instructions per source instead of one's for half of the loads and votes).  Block of 64
// threads: targets tid and tid + 64 of 128.  The operations of a pair and the order of a target's sums are
// those of pair_f32_kernel, so the results are the same bits.
// tile_sums (chunk = one tile): the float32 sums of every tile instead of the chunk's, tile_sums[(tile 3 + q) N
// + i], for pair_reduce_tiles_kernel.
// Products in us, scalar kernel -> this one, without / with torques: N = 3001 35.3 -> 31.1 / 35.4 -> 35.3,
// 8000 111 -> 93 / 130 -> 116, 40000 1782 -> 1459 / 2232 -> 1937.  With one tile per CTA a warp is alone on
// its scheduler and two targets per lane double its chain: N = 2048 24.8 -> 29.4, 300 22.8 -> 26.8, so the
// scalar kernel keeps those.
template <bool TORQUE>
__global__ void __launch_bounds__(64) pair_f32_free_kernel(const SrcF32 *__restrict__ src, int N, int chunk, X2Consts c,
                                                           double *__restrict__ part, float *__restrict__ tile_sums,
                                                           const double *__restrict__ stop)
{
    const bool quit = stopped(stop);
    __shared__ float4 sp[kTile], sf[kTile];
    __shared__ float4 st[TORQUE ? kTile : 1];
    const int tid = threadIdx.x;
    const int i0 = blockIdx.x * kTile + tid, i1 = i0 + 64;
    const int j0 = blockIdx.y * chunk;
    const int j1 = min(N, j0 + chunk);
    const float2 zero2 = make_float2(0.f, 0.f), one2 = make_float2(1.f, 1.f);
    float4 p0 = make_float4(0.f, 0.f, 0.f, 0.f), p1 = p0;
    float2 tz = one2;
    if (i0 < N) {
        p0 = src[i0].p;
        tz.x = src[i0].f.x;
    }
    if (i1 < N) {
        p1 = src[i1].p;
        tz.y = src[i1].f.x;
    }
    const float2 tx = make_float2(p0.x, p1.x), ty = make_float2(p0.y, p1.y);
    const float2 txl = make_float2(p0.z, p1.z), tyl = make_float2(p0.w, p1.w);
    float2 s[3] = {zero2, zero2, zero2}, comp[3] = {zero2, zero2, zero2};
    auto dup = [](float v) { return make_float2(v, v); };
    // the targets' velocities from source k added to u
    auto pair = [&](int k, float2 &ux, float2 &uy, float2 &uz) {
        const float4 p = sp[k], f = sf[k];
        const float2 rx = add2(sub2(tx, dup(p.x)), sub2(txl, dup(p.z)));
        const float2 ry = add2(sub2(ty, dup(p.y)), sub2(tyl, dup(p.w)));
        const float2 rz = sub2(tz, dup(f.x));
        const float2 r2 = fma2(rz, rz, fma2(rx, rx, mul2(ry, ry)));
        const float2 ir = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
        const float2 ir2 = mul2(ir, ir), ir3 = mul2(ir, ir2);
        float2 c1 = mul2(ir, fma2(c.two_3_a2, ir2, one2));
        float2 c2 = mul2(ir3, fma2(c.m_two_a2, ir2, one2));
        float2 ct = ir3;
        const bool n0 = r2.x < c.four_a2, n1 = r2.y < c.four_a2;
        if (__any_sync(0xffffffffu, n0 || n1)) {
            if (n0) near_fix(r2.x, ir.x, 0.f, c, c1.x, c2.x, ct.x);
            if (n1) near_fix(r2.y, ir.y, 0.f, c, c1.y, c2.y, ct.y);
        }
        const float2 Fx = dup(f.y), Fy = dup(f.z), Fz = dup(f.w);
        const float2 k2 = mul2(c2, fma2(rz, Fz, fma2(rx, Fx, mul2(ry, Fy))));
        ux = fma2(c1, Fx, fma2(k2, rx, ux));
        uy = fma2(c1, Fy, fma2(k2, ry, uy));
        uz = fma2(c1, Fz, fma2(k2, rz, uz));
        if (TORQUE) {
            const float4 q = st[k];
            const float2 Tx = dup(q.x), Ty = dup(q.y), Tz = dup(q.z);
            ux = fma2(ct, fma2(Ty, rz, neg2(mul2(Tz, ry))), ux);
            uy = fma2(ct, fma2(Tz, rx, neg2(mul2(Tx, rz))), uy);
            uz = fma2(ct, fma2(Tx, ry, neg2(mul2(Ty, rx))), uz);
        }
    };
    for (int base = j0; base < j1; base += kTile) {
        const int cnt = min(kTile, j1 - base);
        for (int k = tid; k < cnt; k += 64) {
            sp[k] = src[base + k].p;
            sf[k] = src[base + k].f;
            if (TORQUE) st[k] = src[base + k].t;
        }
        __syncthreads();
        if (quit) return;
        float2 u[3] = {zero2, zero2, zero2};
        if (base != (int)blockIdx.x * kTile) {
#pragma unroll 4
            for (int k = 0; k < cnt; ++k) pair(k, u[0], u[1], u[2]);
        } else {
            for (int k = 0; k < cnt; ++k) {
                float2 d[3] = {zero2, zero2, zero2};
                pair(k, d[0], d[1], d[2]);
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if (k != tid) u[q].x += d[q].x;
                    if (k != tid + 64) u[q].y += d[q].y;
                }
            }
        }
        if (tile_sums) {
            float *o = tile_sums + (size_t)blockIdx.y * 3 * N;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if (i0 < N) o[(size_t)q * N + i0] = u[q].x;
                if (i1 < N) o[(size_t)q * N + i1] = u[q].y;
            }
            return;
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {  // compensated (Kahan) accumulation of the tile sums
            const float2 y = sub2(u[q], comp[q]), t = add2(s[q], y);
            comp[q] = sub2(sub2(t, s[q]), y);
            s[q] = t;
        }
        __syncthreads();
    }
    double *o = part + (size_t)blockIdx.y * 3 * N;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        if (i0 < N) o[(size_t)q * N + i0] = (double)s[q].x - (double)comp[q].x;
        if (i1 < N) o[(size_t)q * N + i1] = (double)s[q].y - (double)comp[q].y;
    }
}

// Float32 pair pass evaluating two sources per lane and iteration with packed float32x2 arithmetic.
// The shared tile holds the 128 sources as 64 interleaved pairs: float4 (x_hi[2p], x_hi[2p+1],
// y_hi[2p], y_hi[2p+1]), (x_lo.., y_lo..), (z~.., Fx..), (Fy.., Fz..), and for torques (Tx.., Ty..)
// and (Tz[2p], Tz[2p+1]).  Slots past the chunk's end hold a distant source with zero load, whose
// contribution is exactly zero, so every tile is a full 64 iterations.
// Targets t0 .. t0 + nt - 1 (t0 a multiple of kTile; nt < 0: all N), partials indexed by i - t0.
template <bool TORQUE>
__global__ void __launch_bounds__(kPairThreads, 6) pair_f32x2_kernel(const SrcF32 *__restrict__ src, int N, int chunk,
                                                                   X2Consts c, double *__restrict__ part, int t0 = 0,
                                                                   int nt = -1)
{
    constexpr int P = kTile / 2;
    __shared__ float4 sA[P], sB[P], sC[P], sD[P];
    __shared__ float4 sE[TORQUE ? P : 1];
    __shared__ float2 sG[TORQUE ? P : 1];
    if (nt < 0) nt = N;
    const int tid = threadIdx.x;
    const int li = blockIdx.x * kPairThreads + tid;
    const int i = t0 + li;
    const bool live = li < nt && i < N;
    const int j0 = blockIdx.y * chunk;
    const int j1 = min(N, j0 + chunk);
    float4 tp = make_float4(0.f, 0.f, 0.f, 0.f);
    float tz = 1.f;
    if (live) {
        tp = src[i].p;
        tz = src[i].f.x;
    }
    const float2 txh = make_float2(tp.x, tp.x), tyh = make_float2(tp.y, tp.y);
    const float2 txl = make_float2(tp.z, tp.z), tyl = make_float2(tp.w, tp.w);
    const float2 tz2 = make_float2(tz, tz);
    const float2 zero2 = make_float2(0.f, 0.f);
    float sx = 0.f, sy = 0.f, sz = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
    const int diag = t0 + blockIdx.x * kTile;
    const int pp = tid >> 1, hh = tid & 1;
    float *fA = reinterpret_cast<float *>(sA);
    float *fB = reinterpret_cast<float *>(sB);
    float *fC = reinterpret_cast<float *>(sC);
    float *fD = reinterpret_cast<float *>(sD);
    float *fE = reinterpret_cast<float *>(sE);
    float *fG = reinterpret_cast<float *>(sG);
    for (int base = j0; base < j1; base += kTile) {
        const int j = base + tid;
        float4 sp_ = make_float4(1e18f, 0.f, 0.f, 0.f), sf_ = make_float4(1.f, 0.f, 0.f, 0.f);
        float4 st_ = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j < j1) {
            sp_ = src[j].p;
            sf_ = src[j].f;
            if (TORQUE) st_ = src[j].t;
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
        if (base != diag) {
#pragma unroll 2
            for (int k = 0; k < P; ++k) {
                const float4 a = sA[k], cc = sC[k], d = sD[k];
                const float4 e = TORQUE ? sE[k] : make_float4(0.f, 0.f, 0.f, 0.f);
                const float2 g = TORQUE ? sG[k] : zero2;
                const float2 zj = make_float2(cc.x, cc.y);
                float2 rx, ry, rz, rho2, r2;
                const bool close = pair_offsets_x2(txh, tyh, txl, tyl, tz2, zj, a, &sB[k], c, rx, ry, rz, rho2, r2);
                pair_velocity_x2_geo<TORQUE>(rx, ry, rz, rho2, r2, close, tz2, zj, make_float2(cc.z, cc.w),
                                             make_float2(d.x, d.y), make_float2(d.z, d.w), make_float2(e.x, e.y),
                                             make_float2(e.z, e.w), g, c, ux, uy, uz);
            }
        } else {
            for (int k = 0; k < P; ++k) {
                const float4 a = sA[k], b = sB[k], cc = sC[k], d = sD[k];
                const float4 e = TORQUE ? sE[k] : make_float4(0.f, 0.f, 0.f, 0.f);
                const float2 g = TORQUE ? sG[k] : zero2;
                const float2 rx = add2(sub2(txh, make_float2(a.x, a.y)), sub2(txl, make_float2(b.x, b.y)));
                const float2 ry = add2(sub2(tyh, make_float2(a.z, a.w)), sub2(tyl, make_float2(b.z, b.w)));
                float2 dx = zero2, dy = zero2, dz = zero2;
                pair_velocity_x2<TORQUE>(rx, ry, tz2, make_float2(cc.x, cc.y), make_float2(cc.z, cc.w),
                                         make_float2(d.x, d.y), make_float2(d.z, d.w), make_float2(e.x, e.y),
                                         make_float2(e.z, e.w), g, c, dx, dy, dz);
                if (k == pp) {  // source 2k + hh is this thread's own sphere
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
    if (live) {
        const size_t o = (size_t)blockIdx.y * 3 * nt;
        part[o + li] = (double)sx - (double)cx;
        part[o + nt + li] = (double)sy - (double)cy;
        part[o + 2 * nt + li] = (double)sz - (double)cz;
    }
}

// ------------------------------------------------------------------ symmetric tt pass
// Translation-translation product evaluating each unordered pair once (reciprocity M_ji = M_ij^T).
// The work is the upper triangle of (target block b, source tile t >= b) units of 128 x 128 spheres,
// taken in row-major order and cut into runs of equal length, one per CTA, so that every CTA has the
// same amount of work; a run is split at row ends into segments (b, t0, t1).  Per segment the CTA
// keeps the 128 targets of block b in registers; the diagonal tile (t = b) is done one-directionally
// with the self pair excluded; every other tile gives both u_i (target side, registers) and v_j
// (source side): each lane evaluates four source pairs (eight sources) per step, and their v_j are
// combined across the warp by a reduce-scatter (three exchange levels, then two butterfly levels;
// the order in which a lane takes the pairs and a swapped copy of the tile make it select-free), the
// four warps' sums are added at the end of the tile, and the tile's source sums go to
// src_part[col_start[t] + b].  Each segment's target sums go to tgt_part[segment].  The reduce
// kernel adds, for each sphere, its row's segment partials and its column's source partials in a
// fixed order.  The translation-translation forms load the next tile's sources while a tile is
// evaluated.  The work lists come from sym_schedule.h.
struct SymCta {
    int s0, s1, pad0, pad1;  // segments [s0, s1)
};
struct SymSeg {
    int b, t0, t1, pad;
};

// both halves of a float2 from the lane lane ^ m
__device__ __forceinline__ float2 shfl_xor2(float2 v, int m)
{
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}

// Periods of the pseudo-periodic mode for the float32 kernels: L = L_hi + L_lo, and 1 / L_hi.
struct PerLen {
    float xh, xl, yh, yl, ix, iy;
};
// Minimum image of an in-plane offset (positions folded into the unit cell: |d| < L).
__device__ __forceinline__ float min_image_f(float d, float Lh, float Ll, float inv)
{
    const float m = rintf(d * inv);
    return fmaf(-m, Ll, fmaf(-m, Lh, d));
}
__device__ __forceinline__ float2 min_image2(float2 d, float Lh, float Ll, float inv)
{
    return make_float2(min_image_f(d.x, Lh, Ll, inv), min_image_f(d.y, Lh, Ll, inv));
}
// d + n L for the image shift n in {-1, 0, 1}
__device__ __forceinline__ float2 shift2(float2 d, float n, float Lh, float Ll)
{
    return make_float2(fmaf(n, Ll, fmaf(n, Lh, d.x)), fmaf(n, Ll, fmaf(n, Lh, d.y)));
}

// RHS2: a second translation-translation right-hand side (src2: s_j P_j per sphere) evaluated with
// the same pair blocks; components 3..5 of the partials carry it.
// PER: pseudo-periodic boundaries (Appendix B): each pair's offset is taken at its minimum image and
// the block is summed over that image and its eight shifts by one period (reciprocity holds image by
// image: the reversed pair's image at -s is the transposed block); the sphere's own unshifted image
// is the self term of the reduce kernel.  Three images share one vote on the overlap branch, so that
// their blocks are straight-line code with three chains in flight: small cells have one warp per
// scheduler and wait for latencies (a step of 256 spheres 1.11 -> 0.93 ms; in order, so the same bits).
// BATCH: the tiles belong to many suspensions packed one after another (sinst: one record per
// suspension; a segment's pad field names its suspension, whose tiles are numbered from tile0);
// segments of suspensions with active[] == 0 are skipped.
template <int MINB, bool TORQUE, bool RHS2 = false, bool PER = false, bool BATCH = false>
__global__ void __launch_bounds__(kPairThreads, MINB) pair_f32x2_sym_kernel(const SrcF32 *__restrict__ src, int N,
                                                                             const SymCta *__restrict__ ctas,
                                                                             const SymSeg *__restrict__ segs,
                                                                             X2Consts c,
                                                                             const int *__restrict__ col_start,
                                                                             double *__restrict__ tgt_part,
                                                                             float *__restrict__ src_part,
                                                                             const float4 *__restrict__ src2 = nullptr,
                                                                             PerLen pl = PerLen{},
                                                                             const SymInst *__restrict__ sinst = nullptr,
                                                                             const int *__restrict__ active = nullptr,
                                                                             const double *__restrict__ stop = nullptr)
{
    if (!BATCH) after_may_start();
    const bool quit = !BATCH && stopped(stop);
    constexpr int P = kTile / 2;
    constexpr int NC = RHS2 ? 6 : 3;
    static_assert(!(PER && RHS2), "the two-right-hand-side form has no pseudo-periodic variant");
    static_assert(!(BATCH && (PER || RHS2)), "the batched form is the plain or the torque form");
    // G source pairs (2G sources) are evaluated per step and then reduce-scattered over the warp
    // (two pairs measured slower in every form).  Each source array holds the tile's pairs (2p, 2p+1) at [p]
    // and the same pairs swapped at [SW + p]; lanes with bit 2 set read the swapped copy, so that the element
    // each lane keeps in the reduce-scatter is always .x (SW puts the two copies in different banks for the 2G
    // lane groups)
    constexpr int G = 4;
    constexpr int SW = P + 4;
    __shared__ float4 sA[SW + P], sB[SW + P], sC[SW + P], sD[SW + P];
    __shared__ float4 sE[TORQUE ? SW + P : 1];
    __shared__ float4 sG[TORQUE ? SW + P : 1];  // (T_z, T_z', 6 z_j, 6 z_j')
    __shared__ float4 sZ[SW + P];                // (-2 z_j, -2 z_j', -4 z_j^2, -4 z_j'^2)
    __shared__ float4 sP[RHS2 ? SW + P : 1];
    __shared__ float2 sQ[RHS2 ? SW + P : 1];
    __shared__ float sv[4][NC][kTile];
    const SymCta cd = ctas[blockIdx.x];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float2 zero2 = make_float2(0.f, 0.f);
    const int pp = tid >> 1, hh = tid & 1;
    const bool bit4 = (lane >> 4) & 1, bit3 = (lane >> 3) & 1;
    // pk: the pair of a step this lane keeps in the reduce-scatter (it evaluates pairs in the order
    // h ^ pk, so v[0] is that pair and the pairs it sends come in the order its partners keep them);
    // swz: its copy of the source arrays
    const int pk = (2 * (int)bit4) ^ (int)bit3;
    const bool bsw = (lane >> 2) & 1;  // the lane reads the swapped copy
    const int swz = bsw ? SW : 0;
    float *fA = reinterpret_cast<float *>(sA);
    float *fB = reinterpret_cast<float *>(sB);
    float *fC = reinterpret_cast<float *>(sC);
    float *fD = reinterpret_cast<float *>(sD);
    float *fE = reinterpret_cast<float *>(sE);
    float *fG = reinterpret_cast<float *>(sG);
    float *fZ = reinterpret_cast<float *>(sZ);
    float *fP = reinterpret_cast<float *>(sP);
    float *fQ = reinterpret_cast<float *>(sQ);
    for (int sg = cd.s0; sg < cd.s1; ++sg) {
    const SymSeg seg = segs[sg];
    long long off = 0;
    int Ni = N, tb = 0;
    if (BATCH) {
        if (active && !active[seg.pad]) continue;  // the same for the whole CTA
        const SymInst si = sinst[seg.pad];
        off = si.off;
        Ni = si.N;
        tb = si.tile0;
    }
    const int li = (seg.b - tb) * kTile + tid;
    const long long i = off + li;
    float4 tp = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 tf = make_float4(1.f, 0.f, 0.f, 0.f);
    float4 th = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 tq = make_float4(0.f, 0.f, 0.f, 0.f);
    if (li < Ni) {
        tp = src[i].p;
        tf = src[i].f;
        if (TORQUE) th = src[i].t;
        if (RHS2) tq = src2[i];
    }
    const float2 txh = make_float2(tp.x, tp.x), tyh = make_float2(tp.y, tp.y);
    const float2 txl = make_float2(tp.z, tp.z), tyl = make_float2(tp.w, tp.w);
    const float2 tz2 = make_float2(tf.x, tf.x);
    const float2 Gx = make_float2(tf.y, tf.y), Gy = make_float2(tf.z, tf.z), Gz = make_float2(tf.w, tf.w);
    const float2 Hx = make_float2(th.x, th.x), Hy = make_float2(th.y, th.y), Hz = make_float2(th.z, th.z);
    const float2 Qx = make_float2(tq.x, tq.x), Qy = make_float2(tq.y, tq.y), Qz = make_float2(tq.z, tq.z);
    const float2 six_zi = make_float2(6.f * tf.x, 6.f * tf.x);
    float ks[NC], kc[NC];  // compensated per-tile sums of the target side
#pragma unroll
    for (int q = 0; q < NC; ++q) ks[q] = kc[q] = 0.f;
    // translation-translation forms: the next tile's sources are loaded into registers while the
    // current tile is evaluated (the load latency is hidden behind the pair work)
    constexpr bool PF = !TORQUE && !RHS2 && !PER;
    float4 nsp = make_float4(1e18f, 0.f, 0.f, 0.f), nsf = make_float4(1.f, 0.f, 0.f, 0.f);
    if (PF && (seg.t0 - tb) * kTile + tid < Ni) {
        const long long j0 = off + (seg.t0 - tb) * kTile + tid;
        nsp = src[j0].p;
        nsf = src[j0].f;
    }
    if (quit) return;  // after the loads above, beside which the word arrives
    for (int t = seg.t0; t < seg.t1; ++t) {
        const int lj = (t - tb) * kTile + tid;
        const long long j = off + lj;
        float4 sp_ = make_float4(1e18f, 0.f, 0.f, 0.f), sf_ = make_float4(1.f, 0.f, 0.f, 0.f);
        float4 st_ = make_float4(0.f, 0.f, 0.f, 0.f), sq_ = make_float4(0.f, 0.f, 0.f, 0.f);
        if (PF) {
            sp_ = nsp;
            sf_ = nsf;
        } else if (lj < Ni) {
            sp_ = src[j].p;
            sf_ = src[j].f;
            if (TORQUE) st_ = src[j].t;
            if (RHS2) sq_ = src2[j];
        }
#pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
            const int o4 = 4 * (cp * SW + pp) + (hh ^ cp), o2 = 2 * (cp * SW + pp) + (hh ^ cp);
            fA[o4] = sp_.x;
            fA[o4 + 2] = sp_.y;
            fB[o4] = sp_.z;
            fB[o4 + 2] = sp_.w;
            fC[o4] = sf_.x;
            fC[o4 + 2] = sf_.y;
            fD[o4] = sf_.z;
            fD[o4 + 2] = sf_.w;
            fZ[o4] = -2.f * sf_.x;
            fZ[o4 + 2] = -4.f * (sf_.x * sf_.x);
            if (TORQUE) {
                fE[o4] = st_.x;
                fE[o4 + 2] = st_.y;
                fG[o4] = st_.z;
                fG[o4 + 2] = 6.f * sf_.x;
            }
            if (RHS2) {
                fP[o4] = sq_.x;
                fP[o4 + 2] = sq_.y;
                fQ[o2] = sq_.z;
            }
        }
        __syncthreads();
        if (PF) {
            nsp = make_float4(1e18f, 0.f, 0.f, 0.f);
            nsf = make_float4(1.f, 0.f, 0.f, 0.f);
            if (t + 1 < seg.t1 && lj + kTile < Ni) {
                nsp = src[j + kTile].p;
                nsf = src[j + kTile].f;
            }
        }
        // a batched suspension's last tile is ragged: the loops stop after its last live source (the
        // padding sources carry zero force, so what they would add is an exact zero; the column
        // partial slots of padding sources then hold stale values, which no output reads)
        const int nsrc = BATCH ? min(kTile, Ni - (t - tb) * kTile) : kTile;
        float2 u[NC];
#pragma unroll
        for (int q = 0; q < NC; ++q) u[q] = zero2;
        if (t == seg.b) {
            const int kend = BATCH ? (nsrc + 1) >> 1 : P;
            for (int k = 0; k < kend; ++k) {
                const float4 a = sA[k], b = sB[k], cc = sC[k], d = sD[k];
                const float4 e = TORQUE ? sE[k] : make_float4(0.f, 0.f, 0.f, 0.f);
                const float2 g = TORQUE ? make_float2(sG[k].x, sG[k].y) : zero2;
                float2 rx0 = add2(sub2(txh, make_float2(a.x, a.y)), sub2(txl, make_float2(b.x, b.y)));
                float2 ry0 = add2(sub2(tyh, make_float2(a.z, a.w)), sub2(tyl, make_float2(b.z, b.w)));
                if constexpr (PER) {
                    rx0 = min_image2(rx0, pl.xh, pl.xl, pl.ix);
                    ry0 = min_image2(ry0, pl.yh, pl.yl, pl.iy);
                    const float2 zj = make_float2(cc.x, cc.y), rz = sub2(tz2, zj);
                    for (int sx = -1; sx <= 1; ++sx) {
                        const float2 rx = shift2(rx0, (float)sx, pl.xh, pl.xl);
                        float2 ry[3], rho2[3], r2[3];
                        bool near = false;
#pragma unroll
                        for (int q = 0; q < 3; ++q) {
                            ry[q] = shift2(ry0, (float)(q - 1), pl.yh, pl.yl);
                            rho2[q] = fma2(rx, rx, mul2(ry[q], ry[q]));
                            r2[q] = fma2(rz, rz, rho2[q]);
                            near = near || r2[q].x < c.four_a2 || r2[q].y < c.four_a2;
                        }
                        auto images = [&](bool close) {
#pragma unroll
                            for (int im = 0; im < 3; ++im) {
                                float2 dd[3] = {zero2, zero2, zero2};
                                pair_velocity_x2_geo<TORQUE>(rx, ry[im], rz, rho2[im], r2[im], close, tz2, zj,
                                                             make_float2(cc.z, cc.w), make_float2(d.x, d.y),
                                                             make_float2(d.z, d.w), make_float2(e.x, e.y),
                                                             make_float2(e.z, e.w), g, c, dd[0], dd[1], dd[2]);
                                // source 2k + hh is this thread's own sphere: its unshifted image is the self term
                                const bool self = k == pp && sx == 0 && im == 1;
#pragma unroll
                                for (int q = 0; q < 3; ++q) {
                                    if (self && hh == 0) dd[q].x = 0.f;
                                    if (self && hh == 1) dd[q].y = 0.f;
                                    u[q] = add2(u[q], dd[q]);
                                }
                            }
                        };
                        if (__any_sync(0xffffffffu, near))
                            images(true);
                        else
                            images(false);
                    }
                } else {
                    float2 dd[NC];
#pragma unroll
                    for (int q = 0; q < NC; ++q) dd[q] = zero2;
                    pair_velocity_x2<TORQUE>(rx0, ry0, tz2, make_float2(cc.x, cc.y), make_float2(cc.z, cc.w),
                                             make_float2(d.x, d.y), make_float2(d.z, d.w), make_float2(e.x, e.y),
                                             make_float2(e.z, e.w), g, c, dd[0], dd[1], dd[2]);
                    if (RHS2) {
                        const float4 pv = sP[k];
                        pair_velocity_x2<false>(rx0, ry0, tz2, make_float2(cc.x, cc.y), make_float2(pv.x, pv.y),
                                                make_float2(pv.z, pv.w), sQ[k], zero2, zero2, zero2, c, dd[3 % NC],
                                                dd[4 % NC], dd[5 % NC]);
                    }
                    if (k == pp) {  // source 2k + hh is this thread's own sphere
#pragma unroll
                        for (int q = 0; q < NC; ++q) {
                            if (hh == 0)
                                dd[q].x = 0.f;
                            else
                                dd[q].y = 0.f;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < NC; ++q) u[q] = add2(u[q], dd[q]);
                }
            }
        } else {
            const int kend = BATCH ? min(P, (nsrc + 2 * G - 1) / (2 * G) * G) : P;
            for (int k = 0; k < kend; k += G) {
                float2 v[G][NC];
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    const int kh = k + (h ^ pk) + swz;
                    const float4 a = sA[kh], cc = sC[kh], d = sD[kh];
                    const float4 e = TORQUE ? sE[kh] : make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 g4 = TORQUE ? sG[kh] : make_float4(0.f, 0.f, 0.f, 0.f);
                    const float2 g = make_float2(g4.x, g4.y), six_zj = make_float2(g4.z, g4.w);
                    const float4 zf = sZ[kh];
                    const float2 m2zj = make_float2(zf.x, zf.y), m4zj2 = make_float2(zf.z, zf.w);
                    const float4 pv = RHS2 ? sP[kh] : make_float4(0.f, 0.f, 0.f, 0.f);
                    const float2 pz = RHS2 ? sQ[kh] : zero2;
                    const float2 zj = make_float2(cc.x, cc.y);
                    if (!PER) {
                        float2 rx, ry, rz, rho2, r2;
                        const bool close =
                            pair_offsets_x2(txh, tyh, txl, tyl, tz2, zj, a, &sB[kh], c, rx, ry, rz, rho2, r2);
                        pair_sym_x2<TORQUE, RHS2>(rx, ry, rz, rho2, r2, close, tz2, zj, m2zj, m4zj2, six_zi, six_zj,
                                                  make_float2(cc.z, cc.w),
                                                  make_float2(d.x, d.y), make_float2(d.z, d.w), Gx, Gy, Gz,
                                                  make_float2(e.x, e.y), make_float2(e.z, e.w), g, Hx, Hy, Hz, c,
                                                  u[0], u[1], u[2], v[h][0], v[h][1], v[h][2],
                                                  make_float2(pv.x, pv.y), make_float2(pv.z, pv.w), pz, Qx, Qy, Qz,
                                                  RHS2 ? &u[3 % NC] : nullptr, RHS2 ? &v[h][3 % NC] : nullptr);
                    } else {
                        // minimum image from the full offsets, then the nine images summed both ways
                        const float4 bl = sB[kh];
                        const float2 rx0 = min_image2(add2(sub2(txh, make_float2(a.x, a.y)),
                                                           sub2(txl, make_float2(bl.x, bl.y))), pl.xh, pl.xl, pl.ix);
                        const float2 ry0 = min_image2(add2(sub2(tyh, make_float2(a.z, a.w)),
                                                           sub2(tyl, make_float2(bl.z, bl.w))), pl.yh, pl.yl, pl.iy);
                        const float2 rz = sub2(tz2, zj);
#pragma unroll
                        for (int q = 0; q < NC; ++q) v[h][q] = zero2;
                        for (int sx = -1; sx <= 1; ++sx) {
                            const float2 rx = shift2(rx0, (float)sx, pl.xh, pl.xl);
                            float2 ry[3], rho2[3], r2[3];
                            bool near = false;
#pragma unroll
                            for (int im = 0; im < 3; ++im) {
                                ry[im] = shift2(ry0, (float)(im - 1), pl.yh, pl.yl);
                                rho2[im] = fma2(rx, rx, mul2(ry[im], ry[im]));
                                r2[im] = fma2(rz, rz, rho2[im]);
                                near = near || r2[im].x < c.four_a2 || r2[im].y < c.four_a2;
                            }
                            auto images = [&](bool close) {
#pragma unroll
                                for (int im = 0; im < 3; ++im) {
                                    float2 vx, vy, vz;
                                    pair_sym_x2<TORQUE>(rx, ry[im], rz, rho2[im], r2[im], close, tz2, zj, m2zj, m4zj2, six_zi,
                                                        six_zj, make_float2(cc.z, cc.w), make_float2(d.x, d.y),
                                                        make_float2(d.z, d.w), Gx, Gy, Gz, make_float2(e.x, e.y),
                                                        make_float2(e.z, e.w), g, Hx, Hy, Hz, c, u[0], u[1], u[2], vx, vy, vz);
                                    v[h][0] = add2(v[h][0], vx);
                                    v[h][1] = add2(v[h][1], vy);
                                    v[h][2] = add2(v[h][2], vz);
                                }
                            };
                            if (__any_sync(0xffffffffu, near))
                                images(true);
                            else
                                images(false);
                        }
                    }
                }
                // reduce-scatter of the 2G sources 2k .. 2k + 2G - 1 over the warp.  G = 2: lane L ends
                // with the sum for source 2(k + pk) + bit3(L), stored by lanes 0, 8, 16, 24; G = 4:
                // with source 2(k + pk) + bit2(L), stored by lanes 0, 4, .., 28
#pragma unroll
                for (int q = 0; q < NC; ++q) {
                    const float2 a0 = add2(v[0][q], shfl_xor2(v[2][q], 16));
                    const float2 a1 = add2(v[1][q], shfl_xor2(v[3][q], 16));
                    const float2 x2 = add2(a0, shfl_xor2(a1, 8));
                    float w = x2.x + __shfl_xor_sync(0xffffffffu, x2.y, 4);
                    w += __shfl_xor_sync(0xffffffffu, w, 2);
                    w += __shfl_xor_sync(0xffffffffu, w, 1);
                    if ((lane & 3) == 0) sv[warp][q][2 * (k + pk) + bsw] = w;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            const float yv = (u[q].x + u[q].y) - kc[q];
            const float tv = ks[q] + yv;
            kc[q] = (tv - ks[q]) - yv;
            ks[q] = tv;
        }
        __syncthreads();
        if (t != seg.b) {
            float *o = src_part + (size_t)(col_start[t] + seg.b) * NC * kTile;
#pragma unroll
            for (int q = 0; q < NC; ++q) o[q * kTile + tid] = (sv[0][q][tid] + sv[1][q][tid]) + (sv[2][q][tid] + sv[3][q][tid]);
        }
        __syncthreads();
    }
    double *o = tgt_part + (size_t)sg * NC * kTile;
#pragma unroll
    for (int q = 0; q < NC; ++q) o[q * kTile + tid] = (double)ks[q] - (double)kc[q];
    }
}

// The pseudo-periodic pass of a small cell, one pair per lane.  A schedule of few one-tile runs leaves most of
// the chip idle while each of its warps works through 32 targets x 128 sources x 9 images (a cell of 256
// spheres: 3 CTAs, one warp per scheduler).  Here a cluster of eight CTAs takes a tile: CTA w and CTA w + 4 the
// targets [32 w, 32 w + 32), the first their sums, the second the velocities of the sources.  Its warps take
// parts that are independent in the sums of pair_f32x2_sym_kernel, so that the results are the same bits:
//   targets   a lane per target; four warps for the even sources and four for the odd ones (the halves of that
//             kernel's packed sums), in the lane's order there.  A warp forms the factors of every fourth
//             source's nine blocks, waits for its turn and adds them to the sums, which go from warp to warp
//             in shared memory.
//   sources   a lane per source; eight warps for four groups of 32 sources and two halves of the targets.  The
//             sum over the 32 targets runs through them in the order of that kernel's exchange between lanes (a
//             binary tree); the four CTAs' sums are added as the four warps' there.
// What bounds it: the instructions of 32 x 9 blocks (one direction, about 56 each) per scheduler.
template <bool TORQUE>
__global__ void __cluster_dims__(8) __launch_bounds__(256, TORQUE ? 1 : 2) pair_sym_lanes_kernel(
    const SrcF32 *__restrict__ src, int N, const SymCta *__restrict__ ctas, const SymSeg *__restrict__ segs, X2Consts c,
    const int *__restrict__ col_start, double *__restrict__ tgt_part, float *__restrict__ src_part, PerLen pl,
    const double *__restrict__ stop)
{
    after_may_start();
    const bool quit = stopped(stop);  // the same for the whole cluster
    __shared__ SrcF32 ss[kTile], st[32];
    __shared__ float us[2][3][32], sv[2][3][kTile];
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w = (int)cl.block_rank() & 3;
    const bool targets = cl.block_rank() < 4;
    const int sg = ctas[blockIdx.x / 8].s0;
    const int b = segs[sg].b, t = segs[sg].t0;
    const bool diag = b == t;  // the same in the whole cluster
    if (diag && !targets) return;
    const int nsrc = min(kTile, N - t * kTile);
    if (tid < kTile + 32) {
        const bool s = tid < kTile;
        const int j = s ? t * kTile + tid : b * kTile + 32 * w + (tid - kTile);
        SrcF32 v;
        v.p = make_float4(s ? 1e18f : 0.f, 0.f, 0.f, 0.f);
        v.f = make_float4(1.f, 0.f, 0.f, 0.f);
        v.t = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j < N) v = src[j];
        (s ? ss[tid] : st[tid - kTile]) = v;
    }
    __syncthreads();
    if (quit) return;
    // the nine images of target T and source S under one vote, so that their blocks are straight-line code with
    // nine chains in flight (three to a vote 54 us a product, nine 46, before warps took turns);
    // eval(image, rx, ry, rz, rho2, r2, close), image 4 the unshifted one
    auto images = [&](const SrcF32 &T, const SrcF32 &S, auto &&eval) {
        const float rx0 = min_image_f(add2(sub2(T.p.x, S.p.x), sub2(T.p.z, S.p.z)), pl.xh, pl.xl, pl.ix);
        const float ry0 = min_image_f(add2(sub2(T.p.y, S.p.y), sub2(T.p.w, S.p.w)), pl.yh, pl.yl, pl.iy);
        const float rz = sub2(T.f.x, S.f.x);
        float rx[3], ry[3], yy[3], rho2[9], r2[9];
        bool near = false;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            rx[s] = fmaf((float)(s - 1), pl.xl, fmaf((float)(s - 1), pl.xh, rx0));
            ry[s] = fmaf((float)(s - 1), pl.yl, fmaf((float)(s - 1), pl.yh, ry0));
            yy[s] = mul2(ry[s], ry[s]);
        }
#pragma unroll
        for (int s = 0; s < 9; ++s) {
            rho2[s] = fma2(rx[s / 3], rx[s / 3], yy[s % 3]);
            r2[s] = fma2(rz, rz, rho2[s]);
            near = near || r2[s] < c.four_a2;
        }
        if (__any_sync(0xffffffffu, near)) {
#pragma unroll
            for (int s = 0; s < 9; ++s) eval(s, rx[s / 3], ry[s % 3], rz, rho2[s], r2[s], true);
        } else {
#pragma unroll
            for (int s = 0; s < 9; ++s) eval(s, rx[s / 3], ry[s % 3], rz, rho2[s], r2[s], false);
        }
    };
    if (targets) {
        const int e = warp & 1, turn = warp >> 1;
        const SrcF32 T = st[lane];
        const int pk = diag ? 0 : (2 * ((lane >> 4) & 1)) ^ ((lane >> 3) & 1);
        const int K = diag ? ((nsrc + 1) / 2 + 3) / 4 * 4 : (nsrc + 7) / 8 * 4;  // at most kTile / 2
        float u[3] = {0.f, 0.f, 0.f};
        // turns: the 32 threads of the warp before arrive at one of barriers 1 .. 8 when they have added their
        // source, ours wait there
        for (int k = turn; k < K; k += 4) {
            const int j = 2 * (k ^ pk) + e;
            const SrcF32 S = ss[j];
            TTTerms<float> tt[9];
            TRTerms<float> tr[9];
            images(T, S, [&](int s, float rx, float ry, float rz, float rho2, float r2, bool close) {
                TTBlock<float> m;
                TRBlock<float> tb;
                pair_block_x2<TORQUE>(rx, ry, rz, rho2, r2, close, T.f.x, S.f.x, -2.f * S.f.x, -4.f * (S.f.x * S.f.x),
                                      6.f * T.f.x, 6.f * S.f.x, c, m, tb);
                tt[s] = tt_target_terms(m, S.f.y, S.f.z, S.f.w);
                if (TORQUE) tr[s] = tr_target_terms(m, tb, S.t.x, S.t.y, S.t.z);
            });
            float d[9][3];
            if (diag) {  // here every image's velocity is rounded before it is added, the self term's left out
                const bool self = j == 32 * w + lane;
#pragma unroll
                for (int s = 0; s < 9; ++s) {
                    d[s][0] = d[s][1] = d[s][2] = 0.f;
                    tt_target_add(tt[s], S.f.y, S.f.z, S.f.w, d[s][0], d[s][1], d[s][2]);
                    if (TORQUE) tr_target_add(tr[s], S.t.x, S.t.y, d[s][0], d[s][1], d[s][2]);
                    if (s == 4 && self) d[s][0] = d[s][1] = d[s][2] = 0.f;
                }
            }
            if (k > 0) {
                asm volatile("bar.sync %0, 64;" ::"r"(1 + 4 * e + turn) : "memory");
#pragma unroll
                for (int q = 0; q < 3; ++q) u[q] = us[e][q][lane];
            }
            if (diag) {
#pragma unroll
                for (int s = 0; s < 9; ++s)
#pragma unroll
                    for (int q = 0; q < 3; ++q) u[q] = add2(u[q], d[s][q]);
            } else {
#pragma unroll
                for (int s = 0; s < 9; ++s) {
                    tt_target_add(tt[s], S.f.y, S.f.z, S.f.w, u[0], u[1], u[2]);
                    if (TORQUE) tr_target_add(tr[s], S.t.x, S.t.y, u[0], u[1], u[2]);
                }
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) us[e][q][lane] = u[q];
            if (k + 1 < K) asm volatile("bar.arrive %0, 64;" ::"r"(1 + 4 * e + ((turn + 1) & 3)) : "memory");
        }
        __syncthreads();
        if (warp < 3) tgt_part[((size_t)sg * 3 + warp) * kTile + 32 * w + lane] = (double)add2(us[0][warp][lane], us[1][warp][lane]);
    } else {
        const int half = warp >> 2, j = 32 * (warp & 3) + lane;
        const SrcF32 S = ss[j];
        float tree[4][3], x[3];
        for (int n = 0; n < 16; ++n) {
            const SrcF32 T = st[__brev(16 * half + n) >> 27];
#pragma unroll
            for (int q = 0; q < 3; ++q) x[q] = 0.f;
            images(T, S, [&](int, float rx, float ry, float rz, float rho2, float r2, bool close) {
                TTBlock<float> m;
                TRBlock<float> tb;
                float v[3];
                pair_block_x2<TORQUE>(rx, ry, rz, rho2, r2, close, T.f.x, S.f.x, -2.f * S.f.x, -4.f * (S.f.x * S.f.x),
                                      6.f * T.f.x, 6.f * S.f.x, c, m, tb);
                tt_apply_source(m, T.f.y, T.f.z, T.f.w, v[0], v[1], v[2]);
                if (TORQUE) tr_apply_source(m, tb, T.t.x, T.t.y, T.t.z, v[0], v[1], v[2]);
#pragma unroll
                for (int q = 0; q < 3; ++q) x[q] = add2(x[q], v[q]);
            });
            // add the finished left subtrees that end here, keep the result as its level's left one
            bool kept = false;
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                if (!kept && ((n >> l) & 1)) {
#pragma unroll
                    for (int q = 0; q < 3; ++q) x[q] = add2(tree[l][q], x[q]);
                } else if (!kept) {
#pragma unroll
                    for (int q = 0; q < 3; ++q) tree[l][q] = x[q];
                    kept = true;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) sv[half][q][j] = x[q];
    }
    if (diag) return;
    cl.sync();  // the sums of the four CTAs are there
    if (!targets && tid < 96) {
        const int q = tid >> 5, j = 32 * w + lane;
        float x[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float *o = cl.map_shared_rank(&sv[0][0][0], 4 + r) + q * kTile + j;
            x[r] = add2(o[0], o[3 * kTile]);
        }
        src_part[((size_t)(col_start[t] + b) * 3 + q) * kTile + j] = add2(add2(x[0], x[1]), add2(x[2], x[3]));
    }
    cl.sync();  // no CTA leaves while another reads its sums
}

// Row partials of the targets plus column partials of the sources, fixed order, and the float64 self term
// from the spheres' coefficients (left out when self_term is 0, for all but one share of a shared
// product).  col_rows: the rows [r0, r1) of each column that the schedule wrote (null: all rows above the
// diagonal).  NC = 6: the partials also carry a second translation-translation right-hand side P,
// written to U2 with its own self term.
// BATCH: tiles of many suspensions (tile_inst: the suspension of each tile; sinst as in the pair
// kernel); the column of tile b holds the rows tile0 .. b - 1 of its suspension, summed in an order
// relative to tile0 so that a suspension's result does not depend on its companions.
// What bounds it: float64 instructions for the batched form (they were about 400 warp instructions a
// tile, most of them the self terms and the conversions of the compensated sums; now about 100), a chain
// of loads and additions for a single small suspension.
template <int NC, bool BATCH = false>
__global__ void __launch_bounds__(BATCH ? 384 : 768, BATCH ? 5 : 2) pair_sym_reduce_kernel(
    const double *tgt_part, const float *src_part, const int *__restrict__ row_seg,
    const int *__restrict__ col_start, int N, const double *__restrict__ F, const double *__restrict__ T, SelfCoefs sc,
    double *__restrict__ U, const double *__restrict__ P = nullptr, double *__restrict__ U2 = nullptr,
    const SymInst *__restrict__ sinst = nullptr, const int *__restrict__ tile_inst = nullptr,
    const int *__restrict__ active = nullptr, const int *__restrict__ col_rows = nullptr, int self_term = 1)
{
    // one CTA of 768 threads (384 batched) per 128-sphere tile, the longest columns first; thread (half, q, l):
    // component q of sphere l, rows of its column and segments of its row congruent to `half` modulo HALVES
    // (a batched suspension's columns are at most a few tiles long: one thread per (q, l) there, so
    // that twice as many tiles are resident at once)
    constexpr int HALVES = BATCH ? 1 : 6 / NC;
    __shared__ double s1[NC][kTile];
    __shared__ FloatSum f1[NC][kTile];
    const int nb = gridDim.x;
    const int b = BATCH ? (int)blockIdx.x : nb - 1 - (int)blockIdx.x;
    if (!BATCH) {
        after_may_start();
        wait_for_before();
    }
    long long off = 0;
    int Ni = N, tb = 0;
    if (BATCH) {
        const int inst = tile_inst[b];
        if (active && !active[inst]) return;  // the same for the whole CTA
        const SymInst si = sinst[inst];
        off = si.off;
        Ni = si.N;
        tb = si.tile0;
    }
    const int half = threadIdx.x / (NC * kTile);
    const int r = threadIdx.x - half * NC * kTile;
    const int q = r / kTile, l = r - q * kTile;
    // column of float32 partials: four independent compensated float32 sums per thread (GB300's
    // float64 rate would make a float64 add per partial the bottleneck; one chain per thread would
    // leave the column latency-bound), converted once and added in a fixed order
    // rows [r0, r1) of the column (a share of the triangle writes only some of them)
    const int r0 = BATCH ? tb : (col_rows ? col_rows[2 * b] : 0);
    const int r1 = BATCH ? b : (col_rows ? col_rows[2 * b + 1] : b);
    const float *col = src_part + (size_t)col_start[b] * NC * kTile + q * kTile + l;
    float cs[4] = {0.f, 0.f, 0.f, 0.f}, cc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int bb = r0 + half; bb < r1; bb += 4 * HALVES) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int row = bb + HALVES * u;
            if (row < r1) {
                const float yv = col[(size_t)row * NC * kTile] - cc[u];
                const float tv = cs[u] + yv;
                cc[u] = (tv - cs[u]) - yv;
                cs[u] = tv;
            }
        }
    }
    FloatSum f = join_sums(cs, cc);
    int k = row_seg[b] + half;
    const int k1 = row_seg[b + 1];
    double v = k < k1 ? tgt_part[((size_t)k * NC + q) * kTile + l] : 0.0;
#pragma unroll 4
    for (k += HALVES; k < k1; k += HALVES) v += tgt_part[((size_t)k * NC + q) * kTile + l];
    if (HALVES == 2) {
        if (half == 1) {
            s1[q][l] = v;
            f1[q][l] = f;
        }
        __syncthreads();
        if (half != 0) return;
        v += s1[q][l];
        f.add(f1[q][l]);
    }
    const int lb = (b - tb) * kTile + l;
    if (lb >= Ni) return;
    v += f.value();
    const long long i = off + lb;
    if (NC == 6 && q >= 3)
        U2[(q - 3) * (int64_t)N + i] = sc.velocity(i, q - 3, v, P, nullptr, N);
    else
        U[q * (int64_t)N + i] =
            BATCH || self_term ? sc.velocity(i, q, v, F, T, N) : sc.s[i] * sc.scale * v;
}

constexpr int kTtMinBlocks = 5;     // resident CTAs per SM of the translation-translation form (up to 102 registers:
                                    // four source pairs per step and the next tile's sources in flight fit in 96
                                    // with the polynomial coefficient form; 4 CTAs measured 2.6% slower)
constexpr int kFusedMinBlocks = 4;  // resident CTAs per SM of the form with torques
constexpr int kRhs2MinBlocks = 3;  // resident CTAs per SM of the two-right-hand-side form
// Resident CTAs per SM of the pseudo-periodic forms (the form with torques spills at 4; at 12000 spheres,
// one image per block against three: 1590 -> 1463 us, with torques 2236 -> 2079 us)
constexpr int kPerMinBlocks = 4, kPerFusedMinBlocks = 3;
// Where the schedule has at most two CTAs per SM, the forms compiled for two: occupancy buys nothing there
// and the registers keep the constants and more of a step in flight (a step of 1024 spheres 426 -> 411 us,
// pseudo-periodic 256 spheres 930 -> 905 us; with full waves they are 3% slower, 5.58 ms a product at 65536).
constexpr int kSmallMinBlocks = 2;
// Pseudo-periodic tiles that take pair_sym_lanes_kernel's cluster of eight CTAs: while these make at most three
// CTAs per SM (1280 spheres at 152 SMs).  A product in us, one CTA of packed arithmetic a tile -> a cluster, without
// / with torques: 256 spheres 79 -> 34 / 99 -> 37, 700 80 -> 44 / 101 -> 54, 1024 80 -> 46 / 101 -> 74,
// 1280 80 -> 70 / 101 -> 95, 1500 82 -> 79 / 103 -> 113.
constexpr int kLanesCtasPerSm = 3;

// Capacity of the schedule: at most kSymMaxCtaPerSm x SMs CTAs and that many plus nb segments.
constexpr int kSymMaxCtaPerSm = 64;

size_t sym_src_part_bytes(int64_t max_N)
{
    const int64_t nb = (max_N + kTile - 1) / kTile;
    return (size_t)(nb * (nb - 1) / 2) * 3 * kTile * sizeof(float);
}

// CTAs of any schedule up to max_N spheres: no more than the triangle has units.
static int64_t sym_max_ctas(int64_t max_N, int num_sms)
{
    const int64_t nb = (max_N + kTile - 1) / kTile;
    return std::min<int64_t>((int64_t)kSymMaxCtaPerSm * num_sms, nb * (nb + 1) / 2);
}

size_t sym_tgt_part_bytes(int64_t max_N, int num_sms)
{
    const int64_t nb = (max_N + kTile - 1) / kTile;
    return (size_t)(nb + sym_max_ctas(max_N, num_sms) + 1) * 3 * kTile * sizeof(double);
}

size_t sym_index_ints(int64_t max_N, int num_sms)
{
    const int64_t nb = (max_N + kTile - 1) / kTile;
    const int64_t maxcta = sym_max_ctas(max_N, num_sms);
    return (size_t)(4 * maxcta + 4 * (maxcta + nb + 1) + 4 * (nb + 1));
}

// Schedule of the symmetric pass for N, share `part` of `nparts` (built and copied to the device when
// they change): the whole triangle in ws.sym, a share in ws.sym_part.
static int sym_prepare(rpb_ctx *ctx, int N, const SymSched **out, int part = 0, int nparts = 1)
{
    Workspace &w = ctx->ws;
    SymSched &sc = nparts == 1 ? w.sym : w.sym_part;
    *out = &sc;
    if (sc.N == N && sc.part == part && sc.nparts == nparts) return RPB_OK;
    sc.N = -1;
    cudaStream_t st = ctx->stream;
    std::vector<int> cta4, seg4, row_seg, col_start, col_rows;
    int64_t u0, u1;
    sym_part_units(N, kTile, part, nparts, &u0, &u1);
    sym_schedule_range(N, ctx->num_sms, kTile, u0, u1, cta4, seg4, row_seg, col_start, col_rows);
    const size_t need = cta4.size() + seg4.size() + row_seg.size() + col_start.size() + col_rows.size();
    if (need > w.sym_index_ints || seg4.size() / 4 * 3 * kTile * sizeof(double) > w.sym_tgt_bytes) {
        set_error("internal: symmetric schedule larger than its scratch (N=%d)", N);
        return RPB_EINVAL;
    }
    std::vector<int> host(need);
    size_t o = 0;
    for (const std::vector<int> *v : {&cta4, &seg4, &row_seg, &col_start, &col_rows}) {
        std::copy(v->begin(), v->end(), host.begin() + o);
        o += v->size();
    }
    sc.index = w.sym_index + (nparts == 1 ? 0 : w.sym_index_ints);
    int rc;
    if ((rc = cuda_fail(cudaMemcpyAsync(sc.index, host.data(), need * sizeof(int), cudaMemcpyHostToDevice, st),
                        "symmetric schedule copy")))
        return rc;
    if ((rc = cuda_fail(cudaStreamSynchronize(st), "symmetric schedule copy"))) return rc;
    sc.N = N;
    sc.part = part;
    sc.nparts = nparts;
    sc.ncta = (int)(cta4.size() / 4);
    sc.nseg = (int)(seg4.size() / 4);
    sc.seg_off = (int)cta4.size();
    sc.row_off = sc.seg_off + (int)seg4.size();
    sc.col_off = sc.row_off + (int)row_seg.size();
    sc.rows_off = sc.col_off + (int)col_start.size();
    return RPB_OK;
}

int pair_prepare(rpb_ctx *ctx, int64_t N)
{
    const SymSched *sc;
    if (ctx->sym_enabled && N >= 2 * kTile && N <= ctx->max_N) return sym_prepare(ctx, (int)N, &sc);
    return RPB_OK;
}

// Symmetric product (float32 pairs), translation-translation or, with T, the fused product;
// requires ctx->ws.sym_* scratch.  With nparts > 1: share `part` of the triangle's pairs, the self
// terms with share 0 only (the shares add up to the product).
static int mobility_sym(rpb_ctx *ctx, int N, const double *pos, const double *F, const double *T, double *U,
                        bool packed = false, int part = 0, int nparts = 1)
{
    cudaStream_t st = ctx->stream;
    Workspace &w = ctx->ws;
    const SymSched *sc;
    int rc;
    if ((rc = sym_prepare(ctx, N, &sc, part, nparts))) return rc;
    const double a = ctx->p.a;
    SrcF32 *src = (SrcF32 *)w.src;
    const int pb = elem_threads(N, ctx->num_sms);
    const SelfCoefs self = self_coefs(ctx, N);
    if (!packed) pack_f32_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, 1, src, self);
    const SymCta *ctas = (const SymCta *)sc->index;
    const SymSeg *segs = (const SymSeg *)(sc->index + sc->seg_off);
    const X2Consts c = make_x2_consts(a);
    const int *cs = sc->index + sc->col_off;
    if (sc->ncta > 0) {
        if (T)
            pair_f32x2_sym_kernel<kFusedMinBlocks, true><<<sc->ncta, kPairThreads, 0, st>>>(src, N, ctas, segs, c, cs,
                                                                                            w.sym_tgt, w.sym_src);
        else if (sc->ncta <= kSmallMinBlocks * ctx->num_sms)
            pair_f32x2_sym_kernel<kSmallMinBlocks, false><<<sc->ncta, kPairThreads, 0, st>>>(
                src, N, ctas, segs, c, cs, w.sym_tgt, w.sym_src, nullptr, PerLen{}, nullptr, nullptr, ctx->stop);
        else
            pair_f32x2_sym_kernel<kTtMinBlocks, false><<<sc->ncta, kPairThreads, 0, st>>>(
                src, N, ctas, segs, c, cs, w.sym_tgt, w.sym_src, nullptr, PerLen{}, nullptr, nullptr, ctx->stop);
    }
    const cudaError_t e = launch_after(
        packed && N <= kAfterMaxN, pair_sym_reduce_kernel<3>, dim3((N + kTile - 1) / kTile), 6 * kTile, 0, st, w.sym_tgt, w.sym_src,
        sc->index + sc->row_off, cs, N, F, T, self, U, nullptr, nullptr, nullptr, nullptr, nullptr, sc->index + sc->rows_off,
        part == 0);
    count_launches((sc->ncta > 0 ? 2 : 1) + !packed);
    return cuda_fail(e == cudaSuccess ? cudaGetLastError() : e, "symmetric pair kernels");
}

// The symmetric product in pseudo-periodic mode: positions already folded into the unit cell
// (pos_w; the self terms use the heights of pos, which the fold leaves unchanged); shares as above.
static int mobility_sym_periodic(rpb_ctx *ctx, int N, const double *pos_w, const double *pos, const double *F,
                                 const double *T, double *U, bool packed = false, int part = 0, int nparts = 1)
{
    cudaStream_t st = ctx->stream;
    Workspace &w = ctx->ws;
    const SymSched *sc;
    int rc;
    if ((rc = sym_prepare(ctx, N, &sc, part, nparts))) return rc;
    const double a = ctx->p.a;
    SrcF32 *src = (SrcF32 *)w.src;
    const int pb = elem_threads(N, ctx->num_sms);
    const SelfCoefs self = self_coefs(ctx, N);
    if (!packed) pack_f32_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos_w, F, T, N, a, 1, src, self);
    const SymCta *ctas = (const SymCta *)sc->index;
    const SymSeg *segs = (const SymSeg *)(sc->index + sc->seg_off);
    const X2Consts c = make_x2_consts(a);
    const int *cs = sc->index + sc->col_off;
    PerLen pl;
    pl.xh = (float)ctx->Lx;
    pl.xl = (float)(ctx->Lx - (double)pl.xh);
    pl.yh = (float)ctx->Ly;
    pl.yl = (float)(ctx->Ly - (double)pl.yh);
    pl.ix = 1.f / pl.xh;
    pl.iy = 1.f / pl.yh;
    if (sc->ncta > 0) {
        const bool small = sc->ncta <= kSmallMinBlocks * ctx->num_sms;
        const bool lanes = 8 * sc->ncta <= kLanesCtasPerSm * ctx->num_sms;  // then a run is one tile
        auto run = [&](auto kernel) {
            kernel<<<sc->ncta, kPairThreads, 0, st>>>(src, N, ctas, segs, c, cs, w.sym_tgt, w.sym_src, nullptr, pl, nullptr,
                                                      nullptr, ctx->stop);
        };
        if (T && lanes)
            pair_sym_lanes_kernel<true><<<8 * sc->ncta, 256, 0, st>>>(src, N, ctas, segs, c, cs, w.sym_tgt, w.sym_src, pl,
                                                                      ctx->stop);
        else if (lanes)
            pair_sym_lanes_kernel<false><<<8 * sc->ncta, 256, 0, st>>>(src, N, ctas, segs, c, cs, w.sym_tgt, w.sym_src, pl,
                                                                       ctx->stop);
        else if (T && small)
            run(pair_f32x2_sym_kernel<kSmallMinBlocks, true, false, true>);
        else if (T)
            run(pair_f32x2_sym_kernel<kPerFusedMinBlocks, true, false, true>);
        else if (small)
            run(pair_f32x2_sym_kernel<kSmallMinBlocks, false, false, true>);
        else
            run(pair_f32x2_sym_kernel<kPerMinBlocks, false, false, true>);
    }
    const cudaError_t e = launch_after(
        packed && N <= kAfterMaxN, pair_sym_reduce_kernel<3>, dim3((N + kTile - 1) / kTile), 6 * kTile, 0, st, w.sym_tgt, w.sym_src,
        sc->index + sc->row_off, cs, N, F, T, self, U, nullptr, nullptr, nullptr, nullptr, nullptr, sc->index + sc->rows_off,
        part == 0);
    count_launches((sc->ncta > 0 ? 2 : 1) + !packed);
    return cuda_fail(e == cudaSuccess ? cudaGetLastError() : e, "periodic symmetric pair kernels");
}

// ------------------------------------------------------------------ batched symmetric pass
// Each suspension's rows of tiles are cut by a fixed rule (runs of at most kBatchSegTiles tiles), so
// that the partial sums a suspension's result is made of do not depend on the other suspensions; one
// CTA per run, longest runs first.
constexpr int kBatchSegTiles = 8;
constexpr size_t kBatchSymScratchLimit = (size_t)4 << 30;

void batch_sym_free(BatchSymPlan &pl)
{
    void *d[] = {pl.index, pl.sinst, pl.tgt, pl.srcp};
    for (void *x : d)
        if (x) cudaFree(x);
    pl = BatchSymPlan();
}

static int grow(void **ptr, size_t *cap, size_t need, const char *what)
{
    if (need <= *cap) return RPB_OK;
    if (*ptr) cudaFree(*ptr);
    *ptr = nullptr;
    *cap = 0;
    if (cudaMalloc(ptr, need) != cudaSuccess) {
        cudaGetLastError();
        *ptr = nullptr;
        set_error("cudaMalloc of %zu bytes (%s) failed", need, what);
        return RPB_ENOMEM;
    }
    *cap = need;
    return RPB_OK;
}

int batch_sym_plan(BatchSymPlan &pl, int B, const int64_t *N, cudaStream_t st, bool *ok, int seg_tiles)
{
    *ok = false;
    if (seg_tiles < 1) seg_tiles = kBatchSegTiles;
    std::vector<int64_t> sizes(N, N + B);
    if (pl.valid && sizes == pl.sizes && seg_tiles == pl.seg_tiles) {
        *ok = true;
        return RPB_OK;
    }
    pl.valid = false;
    BatchSchedule bs;
    batch_sym_schedule(B, N, kTile, seg_tiles, bs);
    std::vector<SymInst> si(B);
    for (int k = 0; k < B; ++k) si[k] = SymInst{(long long)bs.off[k], bs.n[k], bs.tile0[k]};
    const std::vector<int> &seg4 = bs.seg4, &row_seg = bs.row_seg, &col_start = bs.col_start,
                           &tile_inst = bs.tile_inst, &order = bs.cta_order;
    const int nseg = (int)(seg4.size() / 4);
    const int g = bs.ntiles;
    const size_t src_bytes = (size_t)bs.n_src_slots * 3 * kTile * sizeof(float);
    const size_t tgt_bytes = (size_t)nseg * 3 * kTile * sizeof(double);
    if (src_bytes + tgt_bytes > kBatchSymScratchLimit) return RPB_OK;  // one-way kernels instead
    std::vector<int> host;
    host.reserve(4 * nseg + seg4.size() + row_seg.size() + col_start.size() + tile_inst.size());
    for (int q : order) {
        host.push_back(q);
        host.push_back(q + 1);
        host.push_back(0);
        host.push_back(0);
    }
    const int seg_off = (int)host.size();
    host.insert(host.end(), seg4.begin(), seg4.end());
    const int row_off = (int)host.size();
    host.insert(host.end(), row_seg.begin(), row_seg.end());
    const int col_off = (int)host.size();
    host.insert(host.end(), col_start.begin(), col_start.end());
    const int inst_off = (int)host.size();
    host.insert(host.end(), tile_inst.begin(), tile_inst.end());
    int rc;
    size_t icap = pl.index_cap * sizeof(int), scap = (size_t)pl.sinst_cap * sizeof(SymInst);
    if ((rc = grow((void **)&pl.index, &icap, host.size() * sizeof(int), "batched symmetric schedule")) ||
        (rc = grow((void **)&pl.sinst, &scap, (size_t)B * sizeof(SymInst), "batched symmetric instances")) ||
        (rc = grow((void **)&pl.tgt, &pl.tgt_cap, tgt_bytes, "batched symmetric partials")) ||
        (rc = grow((void **)&pl.srcp, &pl.src_cap, std::max<size_t>(src_bytes, 16), "batched symmetric partials")))
        return rc;
    pl.index_cap = icap / sizeof(int);
    pl.sinst_cap = (int)(scap / sizeof(SymInst));
    if ((rc = cuda_fail(cudaMemcpyAsync(pl.index, host.data(), host.size() * sizeof(int), cudaMemcpyHostToDevice, st),
                        "batched symmetric schedule copy")) ||
        (rc = cuda_fail(cudaMemcpyAsync(pl.sinst, si.data(), (size_t)B * sizeof(SymInst), cudaMemcpyHostToDevice, st),
                        "batched symmetric instances copy")) ||
        (rc = cuda_fail(cudaStreamSynchronize(st), "batched symmetric plan")))
        return rc;
    pl.ncta = nseg;
    pl.nseg = nseg;
    pl.ntiles = g;
    pl.seg_off = seg_off;
    pl.row_off = row_off;
    pl.col_off = col_off;
    pl.inst_off = inst_off;
    pl.sizes = sizes;
    pl.seg_tiles = seg_tiles;
    pl.valid = true;
    *ok = true;
    return RPB_OK;
}

int batch_sym_apply(const BatchSymPlan &pl, cudaStream_t st, const SrcF32 *src, int64_t total, const double *F,
                    const double *T, double *U, const int *active, double a, const SelfCoefs &sc)
{
    const SymCta *ctas = (const SymCta *)pl.index;
    const SymSeg *segs = (const SymSeg *)(pl.index + pl.seg_off);
    const int *cs = pl.index + pl.col_off;
    const X2Consts c = make_x2_consts(a);
    const int n = (int)total;
    if (T)
        pair_f32x2_sym_kernel<kFusedMinBlocks, true, false, false, true><<<pl.ncta, kPairThreads, 0, st>>>(
            src, n, ctas, segs, c, cs, pl.tgt, pl.srcp, nullptr, PerLen{}, pl.sinst, active);
    else if (pl.tt_minb == 4)
        pair_f32x2_sym_kernel<4, false, false, false, true><<<pl.ncta, kPairThreads, 0, st>>>(
            src, n, ctas, segs, c, cs, pl.tgt, pl.srcp, nullptr, PerLen{}, pl.sinst, active);
    else
        pair_f32x2_sym_kernel<5, false, false, false, true><<<pl.ncta, kPairThreads, 0, st>>>(
            src, n, ctas, segs, c, cs, pl.tgt, pl.srcp, nullptr, PerLen{}, pl.sinst, active);
    pair_sym_reduce_kernel<3, true><<<pl.ntiles, 3 * kTile, 0, st>>>(
        pl.tgt, pl.srcp, pl.index + pl.row_off, cs, n, F, T, sc, U, nullptr, nullptr, pl.sinst, pl.index + pl.inst_off,
        active);
    count_launches(2);
    return cuda_fail(cudaGetLastError(), "batched symmetric kernels");
}

bool mobility_apply2_ok(const rpb_ctx *ctx, int64_t N)
{
    return !ctx->hook && ctx->sym_rhs2 && ctx->sym_enabled && ctx->p.wall && !(ctx->Lx > 0.0) && N >= 2 * kTile;
}

int mobility_apply2_impl(rpb_ctx *ctx, int64_t N64, const double *pos, const double *F, const double *T,
                         const double *P, double *U, double *U2)
{
    const int N = (int)N64;
    cudaStream_t st = ctx->stream;
    Workspace &w = ctx->ws;
    const SymSched *sc;
    int rc;
    if ((rc = sym_prepare(ctx, N, &sc))) return rc;
    if ((size_t)sc->nseg * 6 * kTile * sizeof(double) > w.sym_tgt_bytes ||
        sym_src_part_bytes(N) * 2 > w.sym_src_bytes) {
        set_error("internal: two-right-hand-side scratch too small (N=%d)", N);
        return RPB_EINVAL;
    }
    const double a = ctx->p.a;
    SrcF32 *src = (SrcF32 *)w.src;
    float4 *src2 = (float4 *)w.src2;
    const int pb = elem_threads(N, ctx->num_sms);
    const SelfCoefs self = self_coefs(ctx, N);
    pack_f32_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, 1, src, self);
    pack_rhs2_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, P, N, a, src2);
    const SymCta *ctas = (const SymCta *)sc->index;
    const SymSeg *segs = (const SymSeg *)(sc->index + sc->seg_off);
    const int *cs = sc->index + sc->col_off;
    pair_f32x2_sym_kernel<kRhs2MinBlocks, true, true><<<sc->ncta, kPairThreads, 0, st>>>(
        src, N, ctas, segs, make_x2_consts(a), cs, w.sym_tgt, w.sym_src, src2);
    pair_sym_reduce_kernel<6><<<(N + kTile - 1) / kTile, 6 * kTile, 0, st>>>(
        w.sym_tgt, w.sym_src, sc->index + sc->row_off, cs, N, F, T, self, U, P, U2, nullptr, nullptr, nullptr,
        sc->index + sc->rows_off);
    count_launches(4);
    return cuda_fail(cudaGetLastError(), "two-right-hand-side symmetric kernels");
}

template <bool TORQUE, bool WALL = true>
__global__ void __launch_bounds__(kPairThreads) pair_f64_kernel(const SrcF64 *__restrict__ src, int N, int chunk,
                                                                 PairConsts<double> c, double *__restrict__ part,
                                                                 int t0 = 0, int nt = -1)
{
    __shared__ double2 sp[kTile];
    __shared__ double2 sq[kTile];
    __shared__ double2 sr[kTile];
    __shared__ double2 ss[TORQUE ? kTile : 1];
    __shared__ double2 su[TORQUE ? kTile : 1];
    if (nt < 0) nt = N;
    const int tid = threadIdx.x;
    const int li = blockIdx.x * kPairThreads + tid;
    const int i = t0 + li;
    const bool live = li < nt && i < N;
    const int j0 = blockIdx.y * chunk;
    const int j1 = min(N, j0 + chunk);
    double2 tp = make_double2(0.0, 0.0);
    double tz = 1.0;
    if (live) {
        tp = src[i].p;
        tz = src[i].q.x;
    }
    double ux = 0.0, uy = 0.0, uz = 0.0;
    for (int base = j0; base < j1; base += kTile) {
        const int j = base + tid;
        if (j < j1) {
            sp[tid] = src[j].p;
            sq[tid] = src[j].q;
            sr[tid] = src[j].r;
            if (TORQUE) {
                ss[tid] = src[j].s;
                su[tid] = src[j].u;
            }
        }
        __syncthreads();
        const int cnt = min(kTile, j1 - base);
        const int self_k = i - base;  // this thread's own sphere is source self_k of the tile, if in [0, cnt)
        if (self_k < 0 || self_k >= cnt) {
#pragma unroll 2
            for (int k = 0; k < cnt; ++k) {
                const double2 p = sp[k], q = sq[k], r = sr[k];
                const double2 s = TORQUE ? ss[k] : make_double2(0.0, 0.0);
                const double2 u = TORQUE ? su[k] : make_double2(0.0, 0.0);
                pair_velocity_f64<TORQUE, WALL>(tp.x - p.x, tp.y - p.y, tz, q.x, q.y, r.x, r.y, s.x, s.y, u.x, c,
                                                    ux, uy, uz);
            }
        } else {
            for (int k = 0; k < cnt; ++k) {
                const double2 p = sp[k], q = sq[k], r = sr[k];
                const double2 s = TORQUE ? ss[k] : make_double2(0.0, 0.0);
                const double2 u = TORQUE ? su[k] : make_double2(0.0, 0.0);
                double dx = 0.0, dy = 0.0, dz = 0.0;
                pair_velocity_f64<TORQUE, WALL>(tp.x - p.x, tp.y - p.y, tz, q.x, q.y, r.x, r.y, s.x, s.y, u.x, c,
                                                    dx, dy, dz);
                if (k != self_k) {
                    ux += dx;
                    uy += dy;
                    uz += dz;
                }
            }
        }
        __syncthreads();
    }
    if (live) {
        const size_t o = (size_t)blockIdx.y * 3 * nt;
        part[o + li] = ux;
        part[o + nt + li] = uy;
        part[o + 2 * nt + li] = uz;
    }
}

// ------------------------------------------------------------------ pseudo-periodic boundaries
// Positions folded into the unit cell [0, Lx) x [0, Ly) (heights unchanged).
__global__ void wrap_kernel(const double *__restrict__ pos, int N, double Lx, double Ly, double *__restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double x = pos[i], y = pos[N + i];
    out[i] = x - Lx * floor(x / Lx);
    out[N + i] = y - Ly * floor(y / Ly);
    out[2 * N + i] = pos[2 * N + i];
}

// Appendix B: periodic in x and y; each source is taken at its minimum image and at the eight shifts of
// it by one period (the unit cell and its eight neighbour cells).  One-way kernels, for float64, products
// without forces or without the wall, and fewer than 256 spheres in float32.  The pack kernel has wrapped every position into the unit cell, so
// in-plane offsets lie in (-L, L) and the minimum-image correction is 0 or +-L.  The sphere's own
// unshifted image is the self term (added by the reduce kernel); its eight shifted images are pairs.
template <bool TORQUE, bool WALL>
__global__ void __launch_bounds__(kPairThreads) pair_periodic_f64_kernel(const SrcF64 *__restrict__ src, int N,
                                                                          int chunk, PairConsts<double> c, double Lx,
                                                                          double Ly, double *__restrict__ part)
{
    __shared__ SrcF64 ss[kTile];
    const int tid = threadIdx.x;
    const int i = blockIdx.x * kPairThreads + tid;
    const int j0 = blockIdx.y * chunk;
    const int j1 = min(N, j0 + chunk);
    double2 tp = make_double2(0.0, 0.0);
    double tz = 1.0;
    if (i < N) {
        tp = src[i].p;
        tz = src[i].q.x;
    }
    double ux = 0.0, uy = 0.0, uz = 0.0;
    for (int base = j0; base < j1; base += kTile) {
        if (base + tid < j1) ss[tid] = src[base + tid];
        __syncthreads();
        const int cnt = min(kTile, j1 - base);
        for (int k = 0; k < cnt; ++k) {
            const SrcF64 s = ss[k];
            double dx = tp.x - s.p.x, dy = tp.y - s.p.y;
            dx -= Lx * rint(dx / Lx);
            dy -= Ly * rint(dy / Ly);
            const bool self = base + k == i;
            for (int nx = -1; nx <= 1; ++nx)
                for (int ny = -1; ny <= 1; ++ny) {
                    if (self && nx == 0 && ny == 0) continue;
                    pair_velocity_f64<TORQUE, WALL>(dx + nx * Lx, dy + ny * Ly, tz, s.q.x, s.q.y, s.r.x, s.r.y,
                                                        s.s.x, s.s.y, s.u.x, c, ux, uy, uz);
                }
        }
        __syncthreads();
    }
    if (i < N) {
        const size_t o = (size_t)blockIdx.y * 3 * N;
        part[o + i] = ux;
        part[o + N + i] = uy;
        part[o + 2 * N + i] = uz;
    }
}

// Float32 version; the period is split L = L_hi + L_lo like the positions.
template <bool TORQUE, bool WALL>
__global__ void __launch_bounds__(kPairThreads) pair_periodic_f32_kernel(const SrcF32 *__restrict__ src, int N,
                                                                          int chunk, PairConsts<float> c, float Lxh,
                                                                          float Lxl, float Lyh, float Lyl,
                                                                          double *__restrict__ part)
{
    __shared__ SrcF32 ss[kTile];
    const int tid = threadIdx.x;
    const int i = blockIdx.x * kPairThreads + tid;
    const int j0 = blockIdx.y * chunk;
    const int j1 = min(N, j0 + chunk);
    float4 tp = make_float4(0.f, 0.f, 0.f, 0.f);
    float tz = 1.f;
    if (i < N) {
        tp = src[i].p;
        tz = src[i].f.x;
    }
    const float ix = 1.f / Lxh, iy = 1.f / Lyh;
    double sx = 0.0, sy = 0.0, sz = 0.0;
    for (int base = j0; base < j1; base += kTile) {
        if (base + tid < j1) ss[tid] = src[base + tid];
        __syncthreads();
        const int cnt = min(kTile, j1 - base);
        float ux = 0.f, uy = 0.f, uz = 0.f;
        for (int k = 0; k < cnt; ++k) {
            const SrcF32 s = ss[k];
            float dx = (tp.x - s.p.x) + (tp.z - s.p.z);
            float dy = (tp.y - s.p.y) + (tp.w - s.p.w);
            const float mx = rintf(dx * ix), my = rintf(dy * iy);
            dx = (dx - mx * Lxh) - mx * Lxl;
            dy = (dy - my * Lyh) - my * Lyl;
            const bool self = base + k == i;
            for (int nx = -1; nx <= 1; ++nx)
                for (int ny = -1; ny <= 1; ++ny) {
                    float ax = 0.f, ay = 0.f, az = 0.f;
                    pair_velocity_f32<TORQUE, WALL>((dx + nx * Lxh) + nx * Lxl, (dy + ny * Lyh) + ny * Lyl, tz, s.f.x,
                                                    s.f.y, s.f.z, s.f.w, s.t.x, s.t.y, s.t.z, c, ax, ay, az);
                    if (!(self && nx == 0 && ny == 0)) {
                        ux += ax;
                        uy += ay;
                        uz += az;
                    }
                }
        }
        sx += ux;
        sy += uy;
        sz += uz;
        __syncthreads();
    }
    if (i < N) {
        const size_t o = (size_t)blockIdx.y * 3 * N;
        part[o + i] = sx;
        part[o + N + i] = sy;
        part[o + 2 * N + i] = sz;
    }
}

// Sum the chunk partials in order, add the float64 self term, apply s_i / (8 pi eta).  Targets t0 ..
// t0 + nt - 1 (nt < 0: all N); U and the partials are indexed by i - t0, the partials with component
// stride nt, U with component stride ldu (ldu < 0: nt).
__global__ void pair_reduce_kernel(const double *__restrict__ part, int splits, int N, const double *__restrict__ pos,
                                   const double *__restrict__ F, const double *__restrict__ T, PairConsts<double> c,
                                   double a, double scale, double *__restrict__ U, int wall, int t0, int nt, int ldu,
                                   SelfCoefs sc)
{
    const int li = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = t0 + li;
    if (li >= nt || i >= N) return;
    double ux = 0.0, uy = 0.0, uz = 0.0;
    for (int s = 0; s < splits; ++s) {
        const size_t o = (size_t)s * 3 * nt;
        ux += part[o + li];
        uy += part[o + nt + li];
        uz += part[o + 2 * nt + li];
    }
    if (sc.s) {
        U[li] = sc.velocity(i, 0, ux, F, T, N);
        U[ldu + li] = sc.velocity(i, 1, uy, F, T, N);
        U[2 * ldu + li] = sc.velocity(i, 2, uz, F, T, N);
        return;
    }
    const double z = pos[2 * N + i];
    const double si = wall ? H0(z / a) : 1.0;
    const double zc = wall ? fmax(z, a) : z;
    const double Fx = F ? si * F[i] : 0.0, Fy = F ? si * F[N + i] : 0.0, Fz = F ? si * F[2 * N + i] : 0.0;
    const double Tx = T ? si * T[i] : 0.0, Ty = T ? si * T[N + i] : 0.0;
    if (wall)
        self_velocity<true, true>(zc, Fx, Fy, Fz, Tx, Ty, c, ux, uy, uz);
    else
        self_velocity<true, false>(zc, Fx, Fy, Fz, Tx, Ty, c, ux, uy, uz);
    const double k = si * scale;
    U[li] = k * ux;
    U[ldu + li] = k * uy;
    U[2 * ldu + li] = k * uz;
}

// The same sum with one warp per target, for products split into many source chunks (small float64
// products): lane l adds chunks l, l + 32, ... and a butterfly adds the lanes in a fixed order, so the
// float64 additions spread over many warps instead of one dependent chain per target; lane 0 adds the
// self term and writes.  Four targets per 128-thread block.
__global__ void __launch_bounds__(128) pair_reduce_warp_kernel(const double *__restrict__ part, int splits, int N,
                                                               const double *__restrict__ pos,
                                                               const double *__restrict__ F,
                                                               const double *__restrict__ T, PairConsts<double> c,
                                                               double a, double scale, double *__restrict__ U,
                                                               int wall, int t0, int nt, int ldu, SelfCoefs sc)
{
    const int lane = threadIdx.x & 31;
    const int li = blockIdx.x * 4 + (threadIdx.x >> 5);
    const int i = t0 + li;
    if (li >= nt || i >= N) return;  // the same for the whole warp
    double ux = 0.0, uy = 0.0, uz = 0.0;
    for (int s = lane; s < splits; s += 32) {
        const size_t o = (size_t)s * 3 * nt;
        ux += part[o + li];
        uy += part[o + nt + li];
        uz += part[o + 2 * nt + li];
    }
    for (int m = 16; m > 0; m >>= 1) {
        ux += __shfl_xor_sync(0xffffffffu, ux, m);
        uy += __shfl_xor_sync(0xffffffffu, uy, m);
        uz += __shfl_xor_sync(0xffffffffu, uz, m);
    }
    if (sc.s) {
        const int q = lane;  // every lane holds the sums
        if (q < 3) U[q * ldu + li] = sc.velocity(i, q, q == 0 ? ux : (q == 1 ? uy : uz), F, T, N);
        return;
    }
    if (lane != 0) return;
    const double z = pos[2 * N + i];
    const double si = wall ? H0(z / a) : 1.0;
    const double zc = wall ? fmax(z, a) : z;
    const double Fx = F ? si * F[i] : 0.0, Fy = F ? si * F[N + i] : 0.0, Fz = F ? si * F[2 * N + i] : 0.0;
    const double Tx = T ? si * T[i] : 0.0, Ty = T ? si * T[N + i] : 0.0;
    if (wall)
        self_velocity<true, true>(zc, Fx, Fy, Fz, Tx, Ty, c, ux, uy, uz);
    else
        self_velocity<true, false>(zc, Fx, Fy, Fz, Tx, Ty, c, ux, uy, uz);
    const double k = si * scale;
    U[li] = k * ux;
    U[ldu + li] = k * uy;
    U[2 * ldu + li] = k * uz;
}

// The same from float32 tile sums: per chunk of `per` tiles the compensated chain that pair_f32_kernel runs over
// them, then the chunks in order, so that the result does not depend on which kernel took the tiles.
// For products without the wall whose chunks make too few CTAs: two tiles per CTA leave 288 CTAs to 3001
// spheres, one makes 576; the pair kernel takes 18.1 us instead of 22.9, this one 6.9 instead of 5.5 and a
// Lanczos solve 920 us instead of 1053.
__global__ void __launch_bounds__(64) pair_reduce_tiles_kernel(const float *__restrict__ tile_sums, int tiles, int per,
                                                               int N, const double *__restrict__ F,
                                                               const double *__restrict__ T, SelfCoefs sc,
                                                               double *__restrict__ U)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, q = blockIdx.y;
    if (i >= N) return;
    const float *p = tile_sums + (size_t)q * N + i;
    double sum = 0.0;
    float s = 0.f, c = 0.f;
    for (int t0 = 0, left = per; t0 < tiles; t0 += 8) {
        float x[8];  // eight loads in flight
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = t0 + u < tiles ? p[(size_t)(t0 + u) * 3 * N] : 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (t0 + u >= tiles) break;
            const float y = x[u] - c, v = s + y;
            c = (v - s) - y;
            s = v;
            if (--left == 0 || t0 + u + 1 == tiles) {  // the end of a chunk
                sum += (double)s - (double)c;
                s = c = 0.f;
                left = per;
            }
        }
    }
    U[(size_t)q * N + i] = sc.velocity(i, q, sum, F, T, N);
}

// Chunk partials -> U (targets t0 .. t0 + nt - 1, nt < 0: all N; U's component stride ldu, ldu < 0:
// nt): a thread per target for few chunks (coalesced loads), a warp per target for many.  With the
// spheres' self coefficients in sc, or without (sc.s null) evaluating the self terms.
static void launch_pair_reduce(cudaStream_t st, const double *part, int splits, int N, const double *pos,
                               const double *F, const double *T, double a, double scale, double *U, int wall, int t0,
                               int nt, int ldu, const SelfCoefs &sc)
{
    if (nt < 0) nt = N;
    if (ldu < 0) ldu = nt;
    const PairConsts<double> c = make_consts<double>(a);
    if (splits >= 16) {
        pair_reduce_warp_kernel<<<(unsigned)((nt + 3) / 4), 128, 0, st>>>(part, splits, N, pos, F, T, c, a, scale, U,
                                                                          wall, t0, nt, ldu, sc);
    } else {
        // 64-target CTAs: the float64 self terms of a small product then spread over several SMs
        const int rb = 64;
        pair_reduce_kernel<<<(unsigned)((nt + rb - 1) / rb), rb, 0, st>>>(part, splits, N, pos, F, T, c, a, scale, U,
                                                                          wall, t0, nt, ldu, sc);
    }
}

void pair_grid(int64_t N, int num_sms, int precision, int slots, int *splits, int64_t *chunk)
{
    pair_grid_plan(N, num_sms, precision == RPB_FP64, slots, kTile, splits, chunk);
}

// Resident CTAs over the whole GPU of the float32 one-way kernels (translation only, with torques).
int pair_occupancy(rpb_ctx *ctx)
{
    int a = 0, b = 0;
    int rc;
    if ((rc = cuda_fail(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, pair_f32x2_kernel<false>, kPairThreads, 0),
                        "pair kernel occupancy")) ||
        (rc = cuda_fail(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, pair_f32x2_kernel<true>, kPairThreads, 0),
                        "pair kernel occupancy")))
        return rc;
    ctx->f32_slots[0] = std::max(1, a) * ctx->num_sms;
    ctx->f32_slots[1] = std::max(1, b) * ctx->num_sms;
    return RPB_OK;
}

size_t pair_partial_bytes(int64_t max_N, int num_sms)
{
    const int64_t tiles = (max_N + kTile - 1) / kTile;
    const int64_t f64 = (target_blocks(num_sms) + tiles + 1) * kTile;  // float64 splits x N bound
    const int64_t f32 = (int64_t)kMaxSplitsF32 * max_N;                 // float32 splits x N bound
    return (size_t)3 * sizeof(double) * (size_t)std::max(f64, f32);
}

// Rows t0 .. t1 - 1 of U = M_tt F + M_tr T (all N sources), written to U_rows with component stride
// ldu (ldu < 0: t1 - t0): the one-way kernels restricted to a range of targets (t0 a multiple of kTile).
int mobility_rows_impl(rpb_ctx *ctx, int64_t N64, const double *pos, const double *F, const double *T, int64_t t0,
                       int64_t t1, double *U_rows, int64_t ldu)
{
    const int N = (int)N64, nt = (int)(t1 - t0);
    cudaStream_t st = ctx->stream;
    const double a = ctx->p.a;
    const bool fp64 = ctx->p.precision == RPB_FP64;
    int splits;
    int64_t chunk;
    rows_grid_plan(nt, N64, ctx->num_sms, fp64, kTile, &splits, &chunk);
    if ((size_t)splits * 3 * nt * sizeof(double) > ctx->ws.partial_bytes) {
        set_error("internal: pair partial buffer too small for rows (nt=%d splits=%d)", nt, splits);
        return RPB_EINVAL;
    }
    double *part = (double *)ctx->ws.partial;
    const int pb = elem_threads(N, ctx->num_sms);
    const dim3 grid((unsigned)((nt + kPairThreads - 1) / kPairThreads), (unsigned)splits);
    const bool torque = T != nullptr;
    if (fp64) {
        SrcF64 *src = (SrcF64 *)ctx->ws.src;
        pack_f64_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, ctx->p.wall, src, no_self_coefs());
        const PairConsts<double> c = make_consts<double>(a);
        if (!ctx->p.wall) {
            if (torque)
                pair_f64_kernel<true, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part, (int)t0, nt);
            else
                pair_f64_kernel<false, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part, (int)t0, nt);
        } else if (torque) {
            pair_f64_kernel<true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part, (int)t0, nt);
        } else {
            pair_f64_kernel<false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part, (int)t0, nt);
        }
    } else {
        SrcF32 *src = (SrcF32 *)ctx->ws.src;
        pack_f32_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, 1, src, no_self_coefs());
        const X2Consts c = make_x2_consts(a);
        if (torque)
            pair_f32x2_kernel<true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part, (int)t0, nt);
        else
            pair_f32x2_kernel<false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part, (int)t0, nt);
    }
    launch_pair_reduce(st, part, splits, N, pos, F, T, a, 1.0 / (8.0 * kPi * ctx->p.eta), U_rows, ctx->p.wall,
                       (int)t0, nt, (int)ldu, no_self_coefs());
    count_launches(3);
    return cuda_fail(cudaGetLastError(), "row pair kernels");
}

static int mobility_direct(rpb_ctx *ctx, int64_t N64, const double *pos, const double *F, const double *T,
                           double *U, ProductMode mode = kPlain);

int mobility_apply_impl(rpb_ctx *ctx, int64_t N64, const double *pos, const double *F, const double *T, double *U,
                        ProductMode mode)
{
    if (ctx->hook && !ctx->in_hook) {  // the product is delegated (e.g. shared out among processes)
        ctx->in_hook = 1;
        const int rc = ctx->hook(ctx->hook_user, N64, pos, F, T, U);
        ctx->in_hook = 0;
        if (rc != RPB_OK && rpb_last_error()[0] == 0) set_error("product hook returned %d", rc);
        return rc;
    }
    return mobility_direct(ctx, N64, pos, F, T, U, mode);
}

// The product of a force on N spheres leaves early when ctx->stop tells it to.
bool product_stops(const rpb_ctx *ctx, int64_t N)
{
    if (ctx->p.precision == RPB_FP64) return mobility_sym64_ok(ctx, ctx->ws.vf);
    return ctx->p.wall ? ctx->sym_enabled && N >= 2 * kTile : !(ctx->Lx > 0.0);
}

// Rows [r0, r1) of share `part` of `nparts`: whole 128-row tiles, as equal as the tiles allow.
static void part_rows(int64_t N, int part, int nparts, int64_t *r0, int64_t *r1)
{
    const int64_t tiles = (N + kTile - 1) / kTile;
    const int64_t base = tiles / nparts, extra = tiles % nparts;
    const int64_t t0 = part * base + std::min<int64_t>(part, extra);
    const int64_t t1 = t0 + base + (part < extra ? 1 : 0);
    *r0 = std::min(N, t0 * kTile);
    *r1 = std::min(N, t1 * kTile);
}

int mobility_part_impl(rpb_ctx *ctx, int64_t N64, const double *pos, const double *F, const double *T, int part,
                       int nparts, double *U)
{
    if (nparts == 1) return mobility_direct(ctx, N64, pos, F, T, U);
    const int N = (int)N64;
    cudaStream_t st = ctx->stream;
    const bool sym = ctx->sym_enabled && ctx->p.wall && F && N >= 2 * kTile && (!T || ctx->sym_fused);
    if (sym && !(ctx->Lx > 0.0)) return mobility_sym(ctx, N, pos, F, T, U, false, part, nparts);
    if (sym && ctx->p.precision == RPB_FP32) {
        const int pb = elem_threads(N, ctx->num_sms);
        wrap_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, N, ctx->Lx, ctx->Ly, ctx->ws.pos_w);
        count_launches(1);
        return mobility_sym_periodic(ctx, N, ctx->ws.pos_w, pos, F, T, U, false, part, nparts);
    }
    int rc;
    if ((rc = cuda_fail(cudaMemsetAsync(U, 0, (size_t)3 * N * sizeof(double), st), "part product zero fill")))
        return rc;
    // the pseudo-periodic one-way kernels and the float32 ones without the wall take all targets:
    // share 0 holds the product
    if (ctx->Lx > 0.0 || (ctx->p.precision == RPB_FP32 && !ctx->p.wall))
        return part == 0 && (F || T) ? mobility_direct(ctx, N64, pos, F, T, U) : RPB_OK;
    if (!F && !T) return RPB_OK;
    int64_t r0, r1;
    part_rows(N64, part, nparts, &r0, &r1);
    if (r1 <= r0) return RPB_OK;
    return mobility_rows_impl(ctx, N64, pos, F, T, r0, r1, U + r0, N64);
}

static int mobility_direct(rpb_ctx *ctx, int64_t N64, const double *pos, const double *F, const double *T,
                           double *U, ProductMode mode)
{
    const int N = (int)N64;
    const bool packed = mode == kAgain;
    if (ctx->sym_enabled && ctx->p.wall && !(ctx->Lx > 0.0) && F && N >= 2 * kTile && (!T || ctx->sym_fused))
        return mobility_sym(ctx, N, pos, F, T, U, packed);
    if (mobility_sym64_ok(ctx, F)) return mobility_sym64(ctx, N, pos, F, T, U, mode);
    cudaStream_t st = ctx->stream;
    const double a = ctx->p.a;
    int splits;
    int64_t chunk;
    pair_grid(N64, ctx->num_sms, ctx->p.precision, ctx->f32_slots[T != nullptr ? 1 : 0], &splits, &chunk);
    if ((size_t)splits * 3 * N * sizeof(double) > ctx->ws.partial_bytes) {
        set_error("internal: pair partial buffer too small (N=%d splits=%d)", N, splits);
        return RPB_EINVAL;
    }
    double *part = (double *)ctx->ws.partial;
    const int pb = elem_threads(N, ctx->num_sms);
    const dim3 grid((unsigned)((N + kPairThreads - 1) / kPairThreads), (unsigned)splits);
    const bool torque = T != nullptr;
    const SelfCoefs self = self_coefs(ctx, N);
    if (ctx->Lx > 0.0) {  // pseudo-periodic: wrap into the unit cell, pack, nine shifts per source
        const double Lx = ctx->Lx, Ly = ctx->Ly;
        if (!packed) wrap_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, N, Lx, Ly, ctx->ws.pos_w);
        const double *pw = ctx->ws.pos_w;
        if (ctx->p.precision == RPB_FP32 && ctx->sym_enabled && ctx->p.wall && F && N >= 2 * kTile &&
            (!T || ctx->sym_fused)) {
            count_launches(!packed);
            return mobility_sym_periodic(ctx, N, pw, pos, F, T, U, packed);
        }
        if (ctx->p.precision == RPB_FP32) {
            SrcF32 *src = (SrcF32 *)ctx->ws.src;
            if (!packed) pack_f32_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pw, F, T, N, a, ctx->p.wall, src, self);
            const PairConsts<float> c = make_consts<float>(a);
            const float Lxh = (float)Lx, Lyh = (float)Ly;
            const float Lxl = (float)(Lx - (double)Lxh), Lyl = (float)(Ly - (double)Lyh);
            if (torque && ctx->p.wall)
                pair_periodic_f32_kernel<true, true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, Lxh, Lxl, Lyh, Lyl, part);
            else if (torque)
                pair_periodic_f32_kernel<true, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, Lxh, Lxl, Lyh, Lyl, part);
            else if (ctx->p.wall)
                pair_periodic_f32_kernel<false, true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, Lxh, Lxl, Lyh, Lyl, part);
            else
                pair_periodic_f32_kernel<false, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, Lxh, Lxl, Lyh, Lyl, part);
        } else {
            SrcF64 *src = (SrcF64 *)ctx->ws.src;
            if (!packed) pack_f64_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pw, F, T, N, a, ctx->p.wall, src, self);
            const PairConsts<double> c = make_consts<double>(a);
            if (torque && ctx->p.wall)
                pair_periodic_f64_kernel<true, true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, Lx, Ly, part);
            else if (torque)
                pair_periodic_f64_kernel<true, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, Lx, Ly, part);
            else if (ctx->p.wall)
                pair_periodic_f64_kernel<false, true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, Lx, Ly, part);
            else
                pair_periodic_f64_kernel<false, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, Lx, Ly, part);
        }
        launch_pair_reduce(st, part, splits, N, nullptr, F, T, a, 0.0, U, 0, 0, -1, -1, self);
        count_launches(packed ? 2 : 4);
        return cuda_fail(cudaGetLastError(), "periodic pair kernels");
    }
    if (ctx->p.precision == RPB_FP32) {
        SrcF32 *src = (SrcF32 *)ctx->ws.src;
        if (!packed) pack_f32_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, ctx->p.wall, src, self);
        if (!ctx->p.wall) {
            if (chunk == kTile) {
                const PairConsts<float> c = make_consts<float>(a);
                if (torque)
                    pair_f32_kernel<true, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part, ctx->stop);
                else
                    pair_f32_kernel<false, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part, ctx->stop);
            } else {
                const X2Consts c = make_x2_consts(a);
                auto run = [&](const dim3 &g, int len, double *chunks, float *tile_sums) {
                    if (torque)
                        pair_f32_free_kernel<true><<<g, 64, 0, st>>>(src, N, len, c, chunks, tile_sums, ctx->stop);
                    else
                        pair_f32_free_kernel<false><<<g, 64, 0, st>>>(src, N, len, c, chunks, tile_sums, ctx->stop);
                };
                // chunks that leave fewer CTAs than four per SM: a CTA per tile (their float32 sums need half
                // of the chunks' float64 ones per tile; one that finds no room takes the chunks)
                const int tiles = (int)grid.x, per = (int)(chunk / kTile);
                if ((int64_t)grid.x * grid.y < 4 * ctx->num_sms &&
                    (size_t)tiles * 3 * N * sizeof(float) <= ctx->ws.partial_bytes) {
                    float *sums = (float *)part;
                    run(dim3(grid.x, (unsigned)tiles), kTile, nullptr, sums);
                    pair_reduce_tiles_kernel<<<dim3((unsigned)((N + 63) / 64), 3), 64, 0, st>>>(sums, tiles, per, N,
                                                                                               F, T, self, U);
                    count_launches(packed ? 2 : 3);
                    return cuda_fail(cudaGetLastError(), "pair kernels");
                }
                run(grid, (int)chunk, part, nullptr);
            }
        } else if (ctx->fp32_variant == 1) {
            const X2Consts c = make_x2_consts(a);
            if (torque)
                pair_f32x2_kernel<true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
            else
                pair_f32x2_kernel<false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
        } else {
            const PairConsts<float> c = make_consts<float>(a);
            if (torque)
                pair_f32_kernel<true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
            else
                pair_f32_kernel<false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
        }
    } else {
        SrcF64 *src = (SrcF64 *)ctx->ws.src;
        if (!packed) pack_f64_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, ctx->p.wall, src, self);
        const PairConsts<double> c = make_consts<double>(a);
        if (!ctx->p.wall) {
            if (torque)
                pair_f64_kernel<true, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
            else
                pair_f64_kernel<false, false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
        } else if (torque) {
            pair_f64_kernel<true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
        } else {
            pair_f64_kernel<false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
        }
    }
    launch_pair_reduce(st, part, splits, N, nullptr, F, T, a, 0.0, U, 0, 0, -1, -1, self);
    count_launches(packed ? 2 : 3);
    return cuda_fail(cudaGetLastError(), "pair kernels");
}

// ------------------------------------------------------------------ forces (Sec. III)
// F_i = -weight z + sum_j f(|r_ij|) r_ij/|r_ij| + f_wall(z_i) z with f = -dU/dr of Eq. (soft_potential).
// Pairs are screened in float32 against a cutoff with a generous margin; the ones inside are
// evaluated in float64.
// PER: pseudo-periodic boundaries (Appendix B), minimum image in x (period Lx) and y (period Ly); the
// positions are then the ones folded into the unit cell.
// gate: when given, the kernel runs only if the cell-list pass declined the configuration.
template <bool PER>
__global__ void __launch_bounds__(128) forces_kernel(const double *__restrict__ pos, int N, double a, double weight,
                                                     double U0, double b, float cut2, double *__restrict__ F,
                                                     double Lx = 0.0, double Ly = 0.0,
                                                     const CellHeader *gate = nullptr)
{
    if (gate && !cell_overfull(gate)) return;
    __shared__ float4 sp[64];  // float32 copies of the tile's positions, for the screen only
    const int tid = threadIdx.x;
    const int i = blockIdx.x * 128 + tid;
    double xi = 0.0, yi = 0.0, zi = 0.0;
    if (i < N) {
        xi = pos[i];
        yi = pos[N + i];
        zi = pos[2 * N + i];
    }
    const float xf = (float)xi, yf = (float)yi, zf = (float)zi;
    const double f0 = U0 / b;
    double fx = 0.0, fy = 0.0, fz = 0.0;
    // Near pairs found by the float32 screen are queued per thread and evaluated in float64 together
    // after the screen (or when the queue cannot take two more), so a warp pays for the slowest lane's list
    // rather than for every lane's pairs one after another.  One place evaluates a full queue: with one after
    // each of the two sources the screen of a pseudo-periodic cell took twice as long (8193 spheres 823 -> 434 us,
    // 65536 6848 -> 3587; open, a column of 5000 spheres 1544 -> 1205).
    constexpr int kQ = 32;
    int queue[kQ];
    int nq = 0;
    auto flush = [&]() {
        for (int q = 0; q < nq; ++q) {
            const int jj = queue[q];
            double dx = xi - pos[jj], dy = yi - pos[N + jj];
            const double dz = zi - pos[2 * N + jj];
            if (PER) {
                dx -= Lx * rint(dx / Lx);
                dy -= Ly * rint(dy / Ly);
            }
            const double m = steric_pair_factor(dx * dx + dy * dy + dz * dz, 2.0 * a, f0, 1.0 / b);
            fx += m * dx;
            fy += m * dy;
            fz += m * dz;
        }
        nq = 0;
    };
    // the tile as 64 interleaved pairs: sp[p] = (x[2p], x[2p+1], y[2p], y[2p+1]); z in sp2, so that two
    // sources are screened per lane with packed float32x2 arithmetic
    __shared__ float2 sz[64];
    float *fxy = reinterpret_cast<float *>(sp);
    float *fz2 = reinterpret_cast<float *>(sz);
    const float2 X = make_float2(xf, xf), Y = make_float2(yf, yf), Z = make_float2(zf, zf);
    const float fLx = (float)Lx, fLy = (float)Ly;
    const float fiLx = PER ? 1.f / fLx : 0.f, fiLy = PER ? 1.f / fLy : 0.f;
    const int pp = tid >> 1, hh = tid & 1;
    for (int base = 0; base < N; base += 128) {
        const int j = base + tid;
        // slots past N hold a point far above the wall (never inside the screen, also after the
        // minimum-image fold of x and y); the queue test re-checks the index
        const bool in = j < N;
        fxy[4 * pp + hh] = in ? (float)pos[j] : 0.f;
        fxy[4 * pp + 2 + hh] = in ? (float)pos[N + j] : 0.f;
        fz2[2 * pp + hh] = in ? (float)pos[2 * N + j] : 1e18f;
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < 64; ++k) {
            const float4 p = sp[k];
            float2 dx = sub2(X, make_float2(p.x, p.y)), dy = sub2(Y, make_float2(p.z, p.w));
            const float2 dz = sub2(Z, sz[k]);
            if (PER) {
                dx.x -= fLx * rintf(dx.x * fiLx);
                dx.y -= fLx * rintf(dx.y * fiLx);
                dy.x -= fLy * rintf(dy.x * fiLy);
                dy.y -= fLy * rintf(dy.y * fiLy);
            }
            const float2 d2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
            if (d2.x < cut2 || d2.y < cut2) {  // rare: a near pair (or the sphere itself)
                const int j0 = base + 2 * k;
                if (d2.x < cut2 && j0 != i && j0 < N) queue[nq++] = j0;
                if (d2.y < cut2 && j0 + 1 != i && j0 + 1 < N) queue[nq++] = j0 + 1;
                if (nq >= kQ - 1) flush();
            }
        }
        __syncthreads();
    }
    flush();
    if (i < N) {
        fz += (zi < a ? f0 : f0 * exp(-(zi - a) / b)) - weight;
        F[i] = fx;
        F[N + i] = fy;
        F[2 * N + i] = fz;
    }
}

// Small suspensions: sixteen spheres per block, eight threads each, in one launch without cell lists.  The
// sources are screened in float32 against the same radius, kGroupChunk at a time; every thread marks its
// candidates in a bit mask, the eight threads of a sphere write theirs to its list one after another (a
// list holds a whole chunk, so it cannot overflow), and the list is evaluated in float64 by the eight in
// turn.  What bounds it: the float64 chain of the pairs (about 32 instructions each, 64 cycles a warp
// instruction whatever the active lanes): about 15 near pairs a sphere are two or three a thread here, where a
// thread per sphere took the whole list of the longest in its warp, after six short launches that built
// the cells (62 us a call from 64 to 4096 spheres; the pseudo-periodic all-pairs kernel 52 us at 256).  Twenty
// steps of 256 spheres: 7.75 -> 7.03 ms in float64, 23.1 -> 22.0 ms pseudo-periodic.
constexpr int kGroupTargets = 16, kGroupThreads = 8, kGroupChunk = 1024;
// Up to here; beyond, screening all pairs costs more than the cell lists (this kernel 41 us at 4096, 43 at 4300, 46
// at 4600, 56 at 5000, 67 at 6000, 100 at 8192; the cell lists 46 from 4097 to 5000, 49 at 8192).  Pseudo-periodic cells have no cell lists, and up to
// 40000 spheres the kernel of a thread per sphere is slower: 8193 434 us against 131, 16384 801 against 406, 32768
// 1704 against 1333, 40000 2104 against 1924, 65536 3587 against 4573 (with many near pairs a sphere far slower).
constexpr int64_t kGroupMaxN = 4096, kGroupMaxNPer = 40000;

template <bool PER>
__global__ void __launch_bounds__(kGroupTargets * kGroupThreads) forces_group_kernel(
    const double *__restrict__ pos, int N, double a, double weight, double f0, double b, double inv_b, float cut2,
    double *__restrict__ F, double Lx, double Ly)
{
    constexpr int kMask = kGroupChunk / kGroupThreads / 32;
    __shared__ float sx[kGroupChunk], sy[kGroupChunk], sz[kGroupChunk];
    __shared__ unsigned short list[kGroupTargets][kGroupChunk];
    const int tid = threadIdx.x, g = tid / kGroupThreads, p = tid % kGroupThreads;
    const int i = blockIdx.x * kGroupTargets + g, ic = min(i, N - 1);
    const double xi = pos[ic], yi = pos[N + ic], zi = pos[2 * N + ic];
    const float xf = (float)xi, yf = (float)yi, zf = (float)zi;
    const float fLx = (float)Lx, fLy = (float)Ly;
    const float fiLx = PER ? 1.f / fLx : 0.f, fiLy = PER ? 1.f / fLy : 0.f;
    const double two_a = a + a;
    double fx = 0.0, fy = 0.0, fz = 0.0;
    for (int base = 0; base < N; base += kGroupChunk) {
        const int n = min(kGroupChunk, N - base);
        for (int j = tid; j < n; j += kGroupTargets * kGroupThreads) {
            sx[j] = (float)pos[base + j];
            sy[j] = (float)pos[N + base + j];
            sz[j] = (float)pos[2 * N + base + j];
        }
        __syncthreads();
        unsigned mask[kMask];
        int cnt = 0;
#pragma unroll
        for (int w = 0; w < kMask; ++w) {
            unsigned m = 0;
            const int j0 = p + 32 * w * kGroupThreads;
            if (j0 - p < n) {
#pragma unroll 8
                for (int k = 0; k < 32; ++k) {
                    const int j = j0 + k * kGroupThreads;
                    float dx = xf - sx[j], dy = yf - sy[j];
                    const float dz = zf - sz[j];
                    if (PER) {
                        dx -= fLx * rintf(dx * fiLx);
                        dy -= fLy * rintf(dy * fiLy);
                    }
                    if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < cut2 && j < n && base + j != i) m |= 1u << k;
                }
            }
            mask[w] = m;
            cnt += __popc(m);
        }
        // places of this thread's candidates in its sphere's list
        int end = cnt;
        for (int o = 1; o < kGroupThreads; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, end, o, kGroupThreads);
            if (p >= o) end += v;
        }
        const int total = __shfl_sync(0xffffffffu, end, kGroupThreads - 1, kGroupThreads);
        int at = end - cnt;
#pragma unroll
        for (int w = 0; w < kMask; ++w)
            for (unsigned m = mask[w]; m; m &= m - 1)
                list[g][at++] = (unsigned short)(p + (32 * w + __ffs(m) - 1) * kGroupThreads);
        __syncwarp();
        for (int e = p; e < total; e += kGroupThreads) {
            const int j = base + list[g][e];
            double dx = xi - pos[j], dy = yi - pos[N + j];
            const double dz = zi - pos[2 * N + j];
            if (PER) {
                dx -= Lx * rint(dx / Lx);
                dy -= Ly * rint(dy / Ly);
            }
            const double m = steric_pair_factor(dx * dx + dy * dy + dz * dz, two_a, f0, inv_b);
            fx += m * dx;
            fy += m * dy;
            fz += m * dz;
        }
        __syncthreads();  // the tile and the lists are written again
    }
    for (int o = kGroupThreads / 2; o > 0; o >>= 1) {
        fx += __shfl_xor_sync(0xffffffffu, fx, o);
        fy += __shfl_xor_sync(0xffffffffu, fy, o);
        fz += __shfl_xor_sync(0xffffffffu, fz, o);
    }
    if (p == 0 && i < N) {
        F[i] = fx;
        F[N + i] = fy;
        F[2 * N + i] = fz + wall_force(zi, a, weight, f0, b, inv_b);
    }
}

int forces_impl(rpb_ctx *ctx, int64_t N, const double *pos, const rpb_force_params *fp, double *F)
{
    const double a = ctx->p.a;
    const double r_cut = 2.0 * a + kForceCutoffB * fp->b;
    const double rcm = r_cut * 1.01 + 0.01 * a;
    const float cut2 = (float)(rcm * rcm);
    const double f0 = fp->U0 / fp->b, inv_b = 1.0 / fp->b;
    const int n = (int)N;
    const unsigned groups = (unsigned)((N + kGroupTargets - 1) / kGroupTargets);
    cudaStream_t st = ctx->stream;
    if (ctx->Lx > 0.0) {
        const int pb = elem_threads(N, ctx->num_sms);
        wrap_kernel<<<(unsigned)((N + pb - 1) / pb), pb, 0, st>>>(pos, n, ctx->Lx, ctx->Ly, ctx->ws.pos_w);
        if (N <= kGroupMaxNPer)
            forces_group_kernel<true><<<groups, kGroupTargets * kGroupThreads, 0, st>>>(
                ctx->ws.pos_w, n, a, fp->weight, f0, fp->b, inv_b, cut2, F, ctx->Lx, ctx->Ly);
        else
            forces_kernel<true><<<(unsigned)((N + 127) / 128), 128, 0, st>>>(ctx->ws.pos_w, n, a, fp->weight, fp->U0,
                                                                             fp->b, cut2, F, ctx->Lx, ctx->Ly);
        count_launches(2);
        return cuda_fail(cudaGetLastError(), "forces kernel");
    }
    if (N <= kGroupMaxN) {
        forces_group_kernel<false><<<groups, kGroupTargets * kGroupThreads, 0, st>>>(pos, n, a, fp->weight, f0, fp->b,
                                                                                     inv_b, cut2, F, 0.0, 0.0);
        count_launches(1);
        return cuda_fail(cudaGetLastError(), "forces kernel");
    }
    // buckets of cells of side = the screen radius, then the bucket force pass; the all-pairs kernel
    // runs instead when a bucket holds more than kCellMaxSorted spheres (it checks the flag itself)
    const CellLists L = cell_lists(ctx->ws.cells, ctx->max_N);
    int rc;
    if ((rc = cell_forces<OneSuspension>(st, L, pos, N, a, fp->weight, fp->U0, fp->b, rcm, 0.0, nullptr, nullptr, F)))
        return rc;
    forces_kernel<false><<<(unsigned)((N + 127) / 128), 128, 0, st>>>(pos, n, a, fp->weight, fp->U0, fp->b, cut2, F,
                                                                      0.0, 0.0, L.hdr);
    count_launches(1);
    return cuda_fail(cudaGetLastError(), "forces kernels");
}

}  // namespace rpb

// ------------------------------------------------------------------ allocation-free product
// rpb_mobility_apply_noalloc: the same pack / pair / reduce kernels as rpb_mobility_apply, with their
// scratch (packed sources, then the per-chunk partial sums) in a fixed array of the library's device
// image instead of a context's cudaMalloc'd workspace.  The array is created with the module on
// every device that loads the library and lives until the process exits.
#include <cuda.h>

#include <mutex>

namespace rpb {

constexpr int64_t kNoAllocSrcBytes = (int64_t)RPB_NOALLOC_MAX_N * (int64_t)sizeof(SrcF64);
constexpr int64_t kNoAllocPartialElems = (int64_t)16 * 3 * RPB_NOALLOC_MAX_N;  // 16 chunks at the maximum N
constexpr int64_t kNoAllocBytes = kNoAllocSrcBytes + kNoAllocPartialElems * (int64_t)sizeof(double);
static_assert(kNoAllocSrcBytes % 256 == 0, "partials must start 256-byte aligned");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 64;
static std::mutex g_noalloc_mu;
// Per device: the context the address was looked up in (its process-unique id), the address, the SM
// count.  A context destroyed and created again (cudaDeviceReset, or a primary context released and
// retained anew) loads the module again, and the array may then live elsewhere: the id tells.
struct NoAllocSlot {
    unsigned long long ctx_id;
    void *ptr;
    int sms;
};
static NoAllocSlot g_noalloc[kNoAllocMaxDevices];

typedef CUresult (*CtxGetCurrentFn)(CUcontext *);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long *);

// Process-unique id of the calling thread's current CUDA context (driver entry points through the
// runtime, so the library needs no link against the driver library).  Called with g_noalloc_mu held.
static int current_ctx_id(unsigned long long *id)
{
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    int rc;
    if (!get_current || !get_id) {
        void *f0 = nullptr, *f1 = nullptr;
        cudaDriverEntryPointQueryResult q0 = cudaDriverEntryPointSymbolNotFound, q1 = q0;
        if ((rc = cuda_fail(cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f0, 12000, cudaEnableDefault, &q0),
                            "cudaGetDriverEntryPointByVersion(cuCtxGetCurrent)")))
            return rc;
        if ((rc = cuda_fail(cudaGetDriverEntryPointByVersion("cuCtxGetId", &f1, 12000, cudaEnableDefault, &q1),
                            "cudaGetDriverEntryPointByVersion(cuCtxGetId)")))
            return rc;
        if (q0 != cudaDriverEntryPointSuccess || q1 != cudaDriverEntryPointSuccess || !f0 || !f1) {
            set_error("the CUDA driver offers no cuCtxGetCurrent / cuCtxGetId");
            return RPB_ECUDA;
        }
        get_current = (CtxGetCurrentFn)f0;
        get_id = (CtxGetIdFn)f1;
    }
    CUcontext c = nullptr;
    if (get_current(&c) != CUDA_SUCCESS || !c) {
        set_error("no current CUDA context");
        return RPB_ECUDA;
    }
    if (get_id(c, id) != CUDA_SUCCESS) {
        set_error("cuCtxGetId failed");
        return RPB_ECUDA;
    }
    return RPB_OK;
}

// Device address of the scratch array in the current context (looked up once per device and
// context).  The lookup is refused while `st` is being captured into a graph: it runs host-side
// runtime calls that have no place in a capture.
static int noalloc_setup(cudaStream_t st, void **ptr, int *sms)
{
    int dev = 0;
    int rc;
    if ((rc = cuda_fail(cudaGetDevice(&dev), "cudaGetDevice"))) return rc;
    if (dev < 0 || dev >= kNoAllocMaxDevices) {
        set_error("device ordinal %d outside [0, %d)", dev, kNoAllocMaxDevices);
        return RPB_EINVAL;
    }
    // (a runtime call on the stream: it also makes the device's context current if nothing has yet)
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if ((rc = cuda_fail(cudaStreamIsCapturing(st, &cs), "cudaStreamIsCapturing"))) return rc;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);  // also guards the driver entry points' first lookup
    unsigned long long id = 0;
    if ((rc = current_ctx_id(&id))) return rc;
    NoAllocSlot &sl = g_noalloc[dev];
    if (!sl.ptr || sl.ctx_id != id) {
        if (cs != cudaStreamCaptureStatusNone) {
            set_error("rpb_mobility_apply_noalloc: the first call on a device (or after its context was "
                      "recreated) must not be made while the stream is being captured");
            return RPB_EINVAL;
        }
        void *p = nullptr;
        if ((rc = cuda_fail(cudaGetSymbolAddress(&p, g_noalloc_scratch), "cudaGetSymbolAddress(scratch)"))) return rc;
        int n = 0;
        if ((rc = cuda_fail(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev), "SM count"))) return rc;
        sl.ctx_id = id;
        sl.ptr = p;
        sl.sms = n;
    }
    *ptr = sl.ptr;
    *sms = sl.sms;
    return RPB_OK;
}

}  // namespace rpb

extern "C" int rpb_mobility_apply_noalloc(int64_t N64, const double *pos, const double *F, const double *T, double *U,
                                          const rpb_params *p, void *stream)
{
    using namespace rpb;
    if (!p || !(p->a > 0.0) || !(p->eta > 0.0) || (p->precision != RPB_FP64 && p->precision != RPB_FP32) ||
        p->wall != 1) {
        set_error("rpb_mobility_apply_noalloc: missing or bad parameters (wall must be 1)");
        return RPB_EINVAL;
    }
    if (N64 <= 0 || N64 > RPB_NOALLOC_MAX_N) {
        set_error("rpb_mobility_apply_noalloc: N=%lld outside [1, %d] (the size of its fixed scratch)", (long long)N64,
                  RPB_NOALLOC_MAX_N);
        return RPB_EINVAL;
    }
    const void *ptrs[] = {pos, F, T, U};
    for (const void *q : ptrs)
        if (q && ((uintptr_t)q & 7u)) {
            set_error("rpb_mobility_apply_noalloc: pointer not 8-byte aligned");
            return RPB_EINVAL;
        }
    if (!pos || !U) {
        set_error("rpb_mobility_apply_noalloc: pos and U must not be null");
        return RPB_EINVAL;
    }
    if (U == pos || U == F || U == T) {
        set_error("rpb_mobility_apply_noalloc: U aliases an input");
        return RPB_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int N = (int)N64;
    if (!F && !T) return cuda_fail(cudaMemsetAsync(U, 0, 3 * N64 * sizeof(double), st), "memset U");
    void *base = nullptr;
    int sms = 0;
    int rc;
    if ((rc = noalloc_setup(st, &base, &sms))) return rc;
    int splits;
    int64_t chunk;
    noalloc_grid_plan(N64, sms, p->precision == RPB_FP64, kTile, kNoAllocPartialElems, &splits, &chunk);
    double *part = (double *)((unsigned char *)base + kNoAllocSrcBytes);
    const int pb = elem_threads(N, sms);
    const dim3 grid((unsigned)((N + kPairThreads - 1) / kPairThreads), (unsigned)splits);
    const double a = p->a;
    if (p->precision == RPB_FP32) {
        SrcF32 *src = (SrcF32 *)base;
        pack_f32_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, 1, src, no_self_coefs());
        const PairConsts<float> c = make_consts<float>(a);
        if (T)
            pair_f32_kernel<true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
        else
            pair_f32_kernel<false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
    } else {
        SrcF64 *src = (SrcF64 *)base;
        pack_f64_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, 1, src, no_self_coefs());
        const PairConsts<double> c = make_consts<double>(a);
        if (T)
            pair_f64_kernel<true><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
        else
            pair_f64_kernel<false><<<grid, kPairThreads, 0, st>>>(src, N, (int)chunk, c, part);
    }
    launch_pair_reduce(st, part, splits, N, pos, F, T, a, 1.0 / (8.0 * kPi * p->eta), U, 1, 0, -1, -1, no_self_coefs());
    count_launches(3);
    return cuda_fail(cudaGetLastError(), "rpb_mobility_apply_noalloc kernels");
}
