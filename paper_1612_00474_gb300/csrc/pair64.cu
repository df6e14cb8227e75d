// pair64.cu -- float64 product U = M_tt F + M_tr T evaluating each unordered pair once (Sec. II.B's mobility
// is reciprocal, M_ji = M_ij^T).
//
// What bounds it: the float64 pipe, 2 multiply-adds per clock and SM, so a warp instruction takes 64 cycles
// of its scheduler and everything else (shared memory, shuffles, integer work) is free beside it.  The
// kernel is laid out for the fewest float64 instructions per pair: both directions of a pair from one
// evaluation of its geometry and coefficients (82 instructions and two reciprocal square roots against
// 2 x 66 and four one-way); a warp's 32 targets meet the 32 sources of a tile in 32 rotations, lane l taking
// source (l + q) mod 32, and the source sums travel around the warp with the rotation, so that adding a
// pair to them costs nothing beyond its multiply-adds (a reduction over the lanes would cost 3 or more
// additions a pair); the comparisons that pick the overlap branch are made on the bit patterns.
// The four warps of a CTA take eight rotations each of the same unit, so that a unit's float64 chain is
// short; small products split a unit over several CTAs as well (sym64_plan.h).
// A product of 4096 spheres: 2.55 ms with the one-way kernel, 1.25 ms with this one; a product of 64 spheres
// 41 -> 21 us.
// A Lanczos solve makes its products at the same positions: the first one stores every pair's block (64 bytes,
// 0.54 GB at 4096 spheres) and the others read them: 18 instructions a pair, 0.27 ms a product.  An AB step
// of 4096 spheres took 30.2 ms one-way, 15.4 ms with every pair evaluated once per product, 6.9 ms with the
// blocks; 20 steps of 256 spheres 6.2 -> 5.5 ms.  (Float32 pairs are evaluated faster than HBM would
// deliver their blocks.)
#include "pair_math.cuh"
#include "sym64_plan.h"

namespace rpb {

// a < b for non-negative doubles, on the bit patterns (off the float64 pipe)
__device__ __forceinline__ bool less_bits(double a, double b)
{
    return __double_as_longlong(a) < __double_as_longlong(b);
}

struct Vec3 {
    double x, y, z;
};

// Constants of the pair in the radius, as kernel parameters: a float64 multiply-add reads one operand from
// the constant bank, so they take no registers and are not formed again in the loop.
struct Sym64Consts {
    double four_a2, two_3_a2, two_a2, m_two_a2, near_c1, m_near_r, near_c2, near_tr, m_near_tr_r;
    double m2_3_a2, two_3_a4, m10_3_a4, c140_3_a4, c20_a4, m4_a2, m8_3_a4, c20_3_a4, m20_3_a4, m10_a2;
};

inline Sym64Consts make_sym64_consts(double a)
{
    const double a2 = a * a, a4 = a2 * a2;
    Sym64Consts c;
    c.four_a2 = 4.0 * a2;
    c.two_3_a2 = 2.0 * a2 / 3.0;
    c.two_a2 = 2.0 * a2;
    c.m_two_a2 = -2.0 * a2;
    c.near_c1 = 4.0 / (3.0 * a);
    c.m_near_r = -9.0 / (32.0 * a);
    c.near_c2 = 1.0 / (8.0 * a2);
    c.near_tr = 1.0 / (2.0 * a2 * a);
    c.m_near_tr_r = -3.0 / (8.0 * a);
    c.m2_3_a2 = -2.0 * a2 / 3.0;
    c.two_3_a4 = 2.0 * a4 / 3.0;
    c.m10_3_a4 = -10.0 * a4 / 3.0;
    c.c140_3_a4 = 140.0 * a4 / 3.0;
    c.c20_a4 = 20.0 * a4;
    c.m4_a2 = -4.0 * a2;
    c.m8_3_a4 = -8.0 * a4 / 3.0;
    c.c20_3_a4 = 20.0 * a4 / 3.0;
    c.m20_3_a4 = -20.0 * a4 / 3.0;
    c.m10_a2 = -10.0 * a2;
    return c;
}

// Translation block of a pair in units of 1/(8 pi eta): u_i += M F_j, v_j += M^T G_i.  Eight numbers, since
// its in-plane part is symmetric.
struct Block64 {
    double xx, xy, yy, xz, yz, zx, zy, zz;
};

__device__ __forceinline__ void block_apply(const Block64 &m, const Vec3 &F, const Vec3 &G, Vec3 &u, Vec3 &v)
{
    u.x = fma(m.xx, F.x, fma(m.xy, F.y, fma(m.xz, F.z, u.x)));
    u.y = fma(m.xy, F.x, fma(m.yy, F.y, fma(m.yz, F.z, u.y)));
    u.z = fma(m.zx, F.x, fma(m.zy, F.y, fma(m.zz, F.z, u.z)));
    v.x = fma(m.xx, G.x, fma(m.xy, G.y, fma(m.zx, G.z, v.x)));
    v.y = fma(m.xy, G.x, fma(m.yy, G.y, fma(m.zy, G.z, v.y)));
    v.z = fma(m.xz, G.x, fma(m.yz, G.y, fma(m.zz, G.z, v.z)));
}

// One pair, both directions: u += M_ij (F, T) (the target's velocity from the source's load) and
// v += M_ji (G, H) (the source's from the target's); the block and its transpose as in pair_sym_x2.
// zj2 = 2 z_j, m4zj2 = -4 z_j^2.  KEEP: the translation part by its block, returned in m (five
// instructions more than applying the coefficients).
template <bool TORQUE, bool WALL, bool KEEP>
__device__ __forceinline__ void pair_sym64(double rx, double ry, double zi, double zj, double zj2, double m4zj2,
                                           const Vec3 &F, const Vec3 &G, const Vec3 &T, const Vec3 &H,
                                           const Sym64Consts &c, Vec3 &u, Vec3 &v, Block64 &m)
{
    const double rz = zi - zj;
    const double rho2 = fma(rx, rx, ry * ry);
    const double r2 = fma(rz, rz, rho2);
    const double ir = rsqrt_pos(r2);
    const double ir2 = ir * ir, ir3 = ir * ir2;
    double Rz = 0.0, Z = 0.0, w0 = 0.0;  // w0 = 1/|R|
    if (WALL) {
        Rz = zi + zj;
        Z = Rz * Rz;
        w0 = rsqrt_pos(rho2 + Z);
    }
    double c1mu = fma(c.two_3_a2, ir3, WALL ? ir - w0 : ir);
    double c2 = fma(c.m_two_a2, ir3 * ir2, ir3);
    double ct = ir3;
    const bool near = less_bits(r2, c.four_a2);
    if (__any_sync(0xffffffffu, near)) {
        if (near) {  // overlap; a distance whose square is not a normal number is a coincident pair
            const bool apart = __double2hiint(r2) >= 0x00100000;
            const double r = apart ? r2 * ir : 0.0;
            c1mu = fma(c.near_c1, fma(c.m_near_r, r, 1.0), -w0);
            c2 = apart ? c.near_c2 * ir : 0.0;
            ct = c.near_tr * fma(c.m_near_tr_r, r, 1.0);
        }
    }
    double u3 = 0.0, u5 = 0.0, u5Rz = 0.0, u7Rz = 0.0, cF = c1mu, cFE = c1mu, B3 = 0.0, C3 = 0.0, D3 = 0.0;
    if (WALL) {
        const double s = w0 * w0, sZ = s * Z;
        u3 = s * w0;
        u5 = u3 * s;
        const double p = fma(-zj2, zi, c.m2_3_a2);
        const double q = fma(c.two_a2, Z, c.two_3_a4);
        const double XA = fma(s, fma(sZ, c.m10_3_a4, q), p);
        // 2 X_B = -6 p + s (-10 q + (140/3) a^4 sZ), as -20 a^2 Z - (20/3) a^4 = -10 q
        const double XB2 = fma(s, fma(sZ, c.c140_3_a4, -10.0 * q), -6.0 * p);
        const double Eh = fma(s, fma(sZ, c.c20_a4, fma(c.m4_a2, Z, c.m8_3_a4)), m4zj2);
        const double b2 = u5 * XB2;
        const double T2 = u3 * zj2;
        u5Rz = u5 * Rz;
        u7Rz = u5Rz * s;
        cF = fma(u3, XA, c1mu);
        cFE = fma(u3, Eh, cF);
        B3 = fma(0.5, b2, -u3);
        D3 = fma(u7Rz, c.m20_3_a4, T2);
        C3 = fma(-Rz, b2, fma(u7Rz, c.c20_3_a4, T2));
    }
    if (KEEP) {
        const double a = WALL ? c2 + B3 : c2;
        const double ax = a * rx, ay = a * ry, cz = c2 * rz;
        m.xx = fma(ax, rx, cF);
        m.xy = ax * ry;
        m.yy = fma(ay, ry, cF);
        if (WALL) {
            const double bz = B3 * Rz, e = cz + bz;
            const double p = e + C3, q = e + D3;
            m.xz = rx * p;
            m.yz = ry * p;
            m.zx = rx * q;
            m.zy = ry * q;
            m.zz = fma(cz, rz, fma(Rz, bz + (C3 + D3), cFE));
        } else {
            m.xz = m.zx = rx * cz;
            m.yz = m.zy = ry * cz;
            m.zz = fma(cz, rz, cFE);
        }
        block_apply(m, F, G, u, v);
    } else {
        const double pF = fma(rx, F.x, ry * F.y), pG = fma(rx, G.x, ry * G.y);
        const double kF = c2 * fma(rz, F.z, pF), kG = c2 * fma(rz, G.z, pG);
        double kk = kF, zF = kF * rz;
        if (WALL) {
            const double w = fma(Rz, F.z, pF);
            const double ke = fma(B3, w, C3 * F.z);
            kk = kF + ke;
            zF = fma(kF, rz, fma(ke, Rz, fma(D3, w, u.z)));
        } else {
            zF += u.z;
        }
        u.x = fma(cF, F.x, fma(kk, rx, u.x));
        u.y = fma(cF, F.y, fma(kk, ry, u.y));
        u.z = fma(cFE, F.z, zF);
        kk = kG;
        double zG = kG * rz;
        if (WALL) {
            const double w = fma(Rz, G.z, pG);
            const double ke = fma(B3, w, D3 * G.z);
            kk = kG + ke;
            zG = fma(kG, rz, fma(ke, Rz, fma(C3, w, v.z)));
        } else {
            zG += v.z;
        }
        v.x = fma(cF, G.x, fma(kk, rx, v.x));
        v.y = fma(cF, G.y, fma(kk, ry, v.y));
        v.z = fma(cFE, G.z, zG);
    }
    if (TORQUE && WALL) {
        const double dcp = ct - u3;
        const double dz = dcp * rz;
        const double m2t = fma(u5Rz, c.two_a2, dz), m2s = fma(u5Rz, c.two_a2, -dz);
        const double w10 = c.m10_a2 * u7Rz;
        const double u56 = 6.0 * u5;
        const double kt = fma(zi, u56, w10), ks = fma(zj, u56, w10);
        const double d2 = fma(c.m_two_a2, u5, dcp);
        const double zt = fma(-Rz, kt, d2), zs = fma(-Rz, ks, d2);
        const double a = fma(T.x, ry, -(T.y * rx)), b = fma(H.x, ry, -(H.y * rx));
        const double dT = dcp * T.z, dH = dcp * H.z, ka = kt * a, kb = ks * b;
        u.x = fma(T.y, m2t, fma(-dT, ry, fma(-ka, rx, u.x)));
        u.y = fma(-T.x, m2t, fma(dT, rx, fma(-ka, ry, u.y)));
        u.z = fma(a, zt, u.z);
        v.x = fma(H.y, m2s, fma(dH, ry, fma(-kb, rx, v.x)));
        v.y = fma(-H.x, m2s, fma(-dH, rx, fma(-kb, ry, v.y)));
        v.z = fma(-b, zs, v.z);
    } else if (TORQUE) {  // c_t T x r, and the reversed pair with -r
        const double tx = ct * rx, ty = ct * ry, tz = ct * rz;
        u.x = fma(T.y, tz, fma(-T.z, ty, u.x));
        u.y = fma(T.z, tx, fma(-T.x, tz, u.y));
        u.z = fma(T.x, ty, fma(-T.y, tx, u.z));
        v.x = fma(-H.y, tz, fma(H.z, ty, v.x));
        v.y = fma(-H.z, tx, fma(H.x, tz, v.y));
        v.z = fma(-H.x, ty, fma(H.y, tx, v.z));
    }
}

// Blocks of unit (b, t), rotation q: eight rows of 32 lanes each.
__device__ __forceinline__ double *block_rows(double *blocks, int b, int t, int q)
{
    return blocks + (((int64_t)t * (t + 1) / 2 + b) * 32 + q) * (8 * 32);
}

constexpr int kSym64Warps = 4;

// How a product gets its pairs: evaluated, evaluated and their blocks stored, or read from those blocks.
enum PairSource { kEvaluate, kStore, kRead };

// Grid (runs, qs).  tgt_part[(run qs + s)][3][32]: the row sums of the run; src_part[slot][3][32]: the
// source sums of each of its units off the diagonal.  Lanes past the last sphere repeat it with no load.
// PAIRS == kRead: 18 float64 instructions a pair instead of about 95, and 64 bytes read, which HBM delivers in a
// third of the time that those 18 take; the next rotation's blocks are loaded while one is applied.
template <bool TORQUE, bool WALL, PairSource PAIRS>
__global__ void __launch_bounds__(32 * kSym64Warps) pair_sym64_kernel(const SrcF64 *__restrict__ src, int N, Sym64Plan pl,
                                                                       Sym64Consts c, double *__restrict__ tgt_part,
                                                                       double *__restrict__ src_part,
                                                                       double *__restrict__ blocks,
                                                                       const double *__restrict__ stop)
{
    after_may_start();
    const bool quit = stop && *stop != 0.0;  // see stopped() in pair.cu
    static_assert(!(TORQUE && PAIRS == kRead), "the blocks are the translation part");
    constexpr int NS = TORQUE ? 11 : 8;
    // 2 z_j, -4 z_j^2, x, y, z~, F, T of the source tile
    __shared__ double sm[2][NS][kTile64];
    __shared__ double sv[kSym64Warps][3][kTile64];
    __shared__ double dv[3][kTile64];      // the diagonal unit's source sums: they belong to the row too
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s = blockIdx.y, parts = kSym64Warps * pl.qs, part = kSym64Warps * s + warp;
    const int b = sym64_row_of(pl, blockIdx.x);
    const int t0 = b + (int)(blockIdx.x - sym64_row_run(pl, b)) * pl.L;
    const int t1 = min(pl.nb, t0 + pl.L);
    const Vec3 zero = {0.0, 0.0, 0.0};
    double xi, yi, zi;
    Vec3 G = zero, H = zero, u = zero;
    {
        const int i = b * kTile64 + lane;
        const SrcF64 r = src[min(i, N - 1)];
        xi = r.p.x;
        yi = r.p.y;
        zi = r.q.x;
        if (i < N) {
            G = Vec3{r.q.y, r.r.x, r.r.y};
            if (TORQUE) H = Vec3{r.s.x, r.s.y, r.u.x};
        }
    }
    if (tid < 96) dv[tid >> 5][lane] = 0.0;
    for (int t = t0; t < t1; ++t) {
        double(*S)[kTile64] = sm[t & 1];
        const bool diag = t == b;
        // off the diagonal rotations 0 .. 31; on it 1 .. 16 meet every pair, those of rotation 16 twice
        const int q0 = diag ? 1 + 16 * part / parts : 32 * part / parts;
        const int q1 = diag ? 1 + 16 * (part + 1) / parts : 32 * (part + 1) / parts;
        Block64 m, next;
        auto load = [&](int q, Block64 &x) {
            const double *p = block_rows(blocks, b, t, q) + lane;
            x = Block64{__ldcs(p),       __ldcs(p + 32),  __ldcs(p + 64),  __ldcs(p + 96),
                        __ldcs(p + 128), __ldcs(p + 160), __ldcs(p + 192), __ldcs(p + 224)};
        };
        if (PAIRS == kRead && q0 < q1) load(q0, next);
        // components warp, warp + 4, .. of the tile's sources (record: x y z~ Fx Fy Fz Tx Ty Tz)
        const int j = t * kTile64 + lane;
        const double *rec = reinterpret_cast<const double *>(src + min(j, N - 1));
        for (int k = warp + (PAIRS == kRead ? 3 : 0); k < NS - 2; k += kSym64Warps)
            S[k + 2][lane] = k < 3 || j < N ? rec[k] : 0.0;
        if (PAIRS != kRead && WALL && warp == 3) {
            const double z2 = 2.0 * rec[2];
            S[0][lane] = z2;
            S[1][lane] = -(z2 * z2);
        }
        __syncthreads();
        if (quit) return;
        Vec3 v = zero;
#pragma unroll 1
        for (int q = q0; q < q1; ++q) {
            const int k = (lane + q) & 31;
            Vec3 F = {S[5][k], S[6][k], S[7][k]}, T = zero, Gq = G, Hq = H;
            if (TORQUE) T = Vec3{S[8 % NS][k], S[9 % NS][k], S[10 % NS][k]};
            if (diag && q == 16 && lane >= 16) F = T = Gq = Hq = zero;
            if (PAIRS == kRead) {
                m = next;
                if (q + 1 < q1) load(q + 1, next);
                block_apply(m, F, Gq, u, v);
            } else {
                pair_sym64<TORQUE, WALL, PAIRS == kStore>(xi - S[2][k], yi - S[3][k], zi, S[4][k], S[0][k], S[1][k], F, Gq,
                                                          T, Hq, c, u, v, m);
                if (PAIRS == kStore) {
                    double *p = block_rows(blocks, b, t, q) + lane;
                    const double x[8] = {m.xx, m.xy, m.yy, m.xz, m.yz, m.zx, m.zy, m.zz};
#pragma unroll
                    for (int e = 0; e < 8; ++e) p[32 * e] = x[e];
                }
            }
            // the sums move with their sources to the lane that takes them next
            const int from = (lane + 1) & 31;
            v.x = __shfl_sync(0xffffffffu, v.x, from);
            v.y = __shfl_sync(0xffffffffu, v.y, from);
            v.z = __shfl_sync(0xffffffffu, v.z, from);
        }
        const int k = (lane + q1) & 31;
        sv[warp][0][k] = v.x;
        sv[warp][1][k] = v.y;
        sv[warp][2][k] = v.z;
        __syncthreads();
        if (tid < 96) {
            const int q = tid >> 5;
            const double x = (sv[0][q][lane] + sv[1][q][lane]) + (sv[2][q][lane] + sv[3][q][lane]);
            if (diag)
                dv[q][lane] = x;
            else
                src_part[sym64_col_slot(pl, b, t, s) * 96 + tid] = x;
        }
    }
    __syncthreads();  // the last unit's sums have been read
    sv[warp][0][lane] = u.x;
    sv[warp][1][lane] = u.y;
    sv[warp][2][lane] = u.z;
    __syncthreads();
    if (tid < 96) {
        const int q = tid >> 5;
        tgt_part[((int64_t)blockIdx.x * pl.qs + s) * 96 + tid] =
            ((sv[0][q][lane] + sv[1][q][lane]) + (sv[2][q][lane] + sv[3][q][lane])) + dv[q][lane];
    }
}

// One CTA per tile: the tile's row and column partials in a fixed order, eight threads per sum, and the
// self term.
constexpr int kRed64Groups = 8;
constexpr int kRed64Threads = 96 * kRed64Groups;

__global__ void __launch_bounds__(kRed64Threads) pair_sym64_reduce_kernel(
    const double *tgt_part, const double *src_part, Sym64Plan pl, int N,
    const double *__restrict__ F, const double *__restrict__ T, SelfCoefs sc, double *__restrict__ U)
{
    __shared__ double sum[kRed64Groups][96];
    const int b = pl.nb - 1 - (int)blockIdx.x;  // the longest columns first
    const int tid = threadIdx.x;
    const int g = tid / 96, e = tid - 96 * g;
    const int64_t r0 = sym64_row_run(pl, b) * pl.qs;
    const int nr = (int)((pl.nb - b + pl.L - 1) / pl.L) * pl.qs, nc = b * pl.qs;
    const double *row = tgt_part + r0 * 96 + e, *col = src_part + sym64_col_slot(pl, 0, b, 0) * 96 + e;
    after_may_start();
    wait_for_before();
    double x[2] = {0.0, 0.0};
#pragma unroll 4
    for (int k = g; k < nr; k += kRed64Groups) x[0] += row[(int64_t)k * 96];
#pragma unroll 4
    for (int k = g; k < nc; k += kRed64Groups) x[1] += col[(int64_t)k * 96];
    sum[g][e] = x[0] + x[1];
    __syncthreads();
    const int i = b * kTile64 + (tid & 31);
    if (tid < 96 && i < N) {
        double s = 0.0;
        for (int k = 0; k < kRed64Groups; ++k) s += sum[k][tid];
        U[(int64_t)(tid >> 5) * N + i] = sc.velocity(i, tid >> 5, s, F, T, N);
    }
}

bool mobility_sym64_ok(const rpb_ctx *ctx, const double *F)
{
    return ctx->ws.sym64 != nullptr && F != nullptr && !(ctx->Lx > 0.0);
}

// Room for the blocks of a solve of N spheres where the context's scratch has none: asked for by the first solve that
// can read them (a context that makes products only, or pseudo-periodic or hooked ones, takes none), kept, and
// enlarged for a larger one.  What is not granted is not asked for again: those solves evaluate their pairs.
void blocks64_prepare(rpb_ctx *ctx, int64_t N)
{
    Workspace &w = ctx->ws;
    if (ctx->hook || !mobility_sym64_ok(ctx, w.vf) || N <= w.blocks64_N || N >= w.blocks64_refused) return;
    // another thread may be capturing; this one does so only where the solve is refused
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(ctx->stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return;
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
    size_t avail = 0, total = 0;
    int64_t room = 0;
    if (cudaMemGetInfo(&avail, &total) == cudaSuccess)
        room = blocks64_room(N, w.blocks64_N, ctx->max_N, (int64_t)avail, (int64_t)total);
    if (room > 0) {
        if (w.blocks64) {  // kernels that read the old ones have ended
            cudaStreamSynchronize(ctx->stream);
            cudaFree(w.blocks64);
        }
        w.blocks64 = nullptr;
        w.blocks64_N = 0;
        if (cudaMalloc(&w.blocks64, (size_t)blocks64_bytes(room)) == cudaSuccess)
            w.blocks64_N = room;
        else
            w.blocks64 = nullptr;
    }
    if (N > w.blocks64_N) w.blocks64_refused = N;
    cudaGetLastError();
    cudaThreadExchangeStreamCaptureMode(&mode);
}

int mobility_sym64(rpb_ctx *ctx, int N, const double *pos, const double *F, const double *T, double *U, ProductMode mode)
{
    cudaStream_t st = ctx->stream;
    const double a = ctx->p.a;
    const SelfCoefs self = self_coefs(ctx, N);
    const Sym64Consts c64 = make_sym64_consts(a);
    const Sym64Plan pl = sym64_plan(N, ctx->num_sms);
    double *tgt = ctx->ws.sym64, *col = tgt + sym64_tgt_elems(ctx->ws.sym64_N, ctx->num_sms);
    double *blocks = N <= ctx->ws.blocks64_N ? ctx->ws.blocks64 : nullptr;
    SrcF64 *src = (SrcF64 *)ctx->ws.src;
    const int pb = elem_threads(N, ctx->num_sms);
    if (mode != kAgain)
        pack_f64_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, ctx->p.wall, src, self);
    const dim3 grid((unsigned)pl.runs, (unsigned)pl.qs);
    auto run = [&](auto kernel) { kernel<<<grid, 32 * kSym64Warps, 0, st>>>(src, N, pl, c64, tgt, col, blocks, ctx->stop); };
    const PairSource pairs = !blocks || mode == kPlain ? kEvaluate : (mode == kKeep ? kStore : kRead);
    if (pairs == kRead)
        run(pair_sym64_kernel<false, true, kRead>);
    else if (ctx->p.wall && T)
        pairs == kStore ? run(pair_sym64_kernel<true, true, kStore>) : run(pair_sym64_kernel<true, true, kEvaluate>);
    else if (ctx->p.wall)
        pairs == kStore ? run(pair_sym64_kernel<false, true, kStore>) : run(pair_sym64_kernel<false, true, kEvaluate>);
    else if (T)
        pairs == kStore ? run(pair_sym64_kernel<true, false, kStore>) : run(pair_sym64_kernel<true, false, kEvaluate>);
    else
        pairs == kStore ? run(pair_sym64_kernel<false, false, kStore>) : run(pair_sym64_kernel<false, false, kEvaluate>);
    const cudaError_t e = launch_after(mode == kAgain && N <= kAfterMaxN, pair_sym64_reduce_kernel, dim3(pl.nb), kRed64Threads, 0, st, tgt, col, pl, N,
                                       F, T, self, U);
    count_launches(mode == kAgain ? 2 : 3);
    return cuda_fail(e == cudaSuccess ? cudaGetLastError() : e, "float64 symmetric pair kernels");
}

}  // namespace rpb
