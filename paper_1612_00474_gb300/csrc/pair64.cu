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
// An AB step of 4096 spheres, eleven products: 30.2 ms with the one-way kernel, 15.6 ms with this one
// (1.36 ms a product, 8.1e-11 s per ordered pair); a product of 64 spheres 41 -> 21 us; 20 steps of 256
// spheres 16.8 -> 13.2 ms.
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

// One pair, both directions: u += M_ij (F, T) (the target's velocity from the source's load) and
// v += M_ji (G, H) (the source's from the target's); the block and its transpose as in pair_sym_x2.
template <bool TORQUE, bool WALL>
__device__ __forceinline__ void pair_sym64(double rx, double ry, double zi, double zj, const Vec3 &F, const Vec3 &G,
                                           const Vec3 &T, const Vec3 &H, const Sym64Consts &c, Vec3 &u, Vec3 &v)
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
    const double pF = fma(rx, F.x, ry * F.y), pG = fma(rx, G.x, ry * G.y);
    const double kF = c2 * fma(rz, F.z, pF), kG = c2 * fma(rz, G.z, pG);
    if (!WALL) {
        u.x = fma(c1mu, F.x, fma(kF, rx, u.x));
        u.y = fma(c1mu, F.y, fma(kF, ry, u.y));
        u.z = fma(c1mu, F.z, fma(kF, rz, u.z));
        v.x = fma(c1mu, G.x, fma(kG, rx, v.x));
        v.y = fma(c1mu, G.y, fma(kG, ry, v.y));
        v.z = fma(c1mu, G.z, fma(kG, rz, v.z));
        if (TORQUE) {  // c_t T x r, and the reversed pair with -r
            const double tx = ct * rx, ty = ct * ry, tz = ct * rz;
            u.x = fma(T.y, tz, fma(-T.z, ty, u.x));
            u.y = fma(T.z, tx, fma(-T.x, tz, u.y));
            u.z = fma(T.x, ty, fma(-T.y, tx, u.z));
            v.x = fma(-H.y, tz, fma(H.z, ty, v.x));
            v.y = fma(-H.z, tx, fma(H.x, tz, v.y));
            v.z = fma(-H.x, ty, fma(H.y, tx, v.z));
        }
        return;
    }
    const double s = w0 * w0, u3 = s * w0, u5 = u3 * s, sZ = s * Z;
    const double zj2 = zj + zj;
    const double p = fma(-zj2, zi, c.m2_3_a2);
    const double q = fma(c.two_a2, Z, c.two_3_a4);
    const double XA = fma(s, fma(sZ, c.m10_3_a4, q), p);
    // 2 X_B = -6 p + s (-10 q + (140/3) a^4 sZ), as -20 a^2 Z - (20/3) a^4 = -10 q
    const double XB2 = fma(s, fma(sZ, c.c140_3_a4, -10.0 * q), -6.0 * p);
    const double Eh = fma(s, fma(sZ, c.c20_a4, fma(c.m4_a2, Z, c.m8_3_a4)), -(zj2 * zj2));
    const double b2 = u5 * XB2;
    const double T2 = u3 * zj2;
    const double u5Rz = u5 * Rz, u7Rz = u5Rz * s;
    const double cF = fma(u3, XA, c1mu);
    const double cFE = fma(u3, Eh, cF);
    const double B3 = fma(0.5, b2, -u3);
    const double D3 = fma(u7Rz, c.m20_3_a4, T2);
    const double C3 = fma(-Rz, b2, fma(u7Rz, c.c20_3_a4, T2));
    {
        const double w = fma(Rz, F.z, pF);
        const double ke = fma(B3, w, C3 * F.z);
        const double kk = kF + ke;
        u.x = fma(cF, F.x, fma(kk, rx, u.x));
        u.y = fma(cF, F.y, fma(kk, ry, u.y));
        u.z = fma(cFE, F.z, fma(kF, rz, fma(ke, Rz, fma(D3, w, u.z))));
    }
    {
        const double w = fma(Rz, G.z, pG);
        const double ke = fma(B3, w, D3 * G.z);
        const double kk = kG + ke;
        v.x = fma(cF, G.x, fma(kk, rx, v.x));
        v.y = fma(cF, G.y, fma(kk, ry, v.y));
        v.z = fma(cFE, G.z, fma(kG, rz, fma(ke, Rz, fma(C3, w, v.z))));
    }
    if (TORQUE) {
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
    }
}

constexpr int kSym64Warps = 4;

// Grid (runs, qs).  tgt_part[(run qs + s)][3][32]: the row sums of the run; src_part[slot][3][32]: the
// source sums of each of its units off the diagonal.  Lanes past the last sphere repeat it with no load.
template <bool TORQUE, bool WALL>
__global__ void __launch_bounds__(32 * kSym64Warps) pair_sym64_kernel(const SrcF64 *__restrict__ src, int N, Sym64Plan pl,
                                                                       Sym64Consts c, double *__restrict__ tgt_part,
                                                                       double *__restrict__ src_part)
{
    constexpr int NS = TORQUE ? 9 : 6;
    __shared__ double sm[2][NS][kTile64];  // x, y, z~, F, T of the source tile
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
        // components warp, warp + 4, .. of the tile's sources (record: x y z~ Fx Fy Fz Tx Ty Tz)
        const int j = t * kTile64 + lane;
        const double *rec = reinterpret_cast<const double *>(src + min(j, N - 1));
        for (int k = warp; k < NS; k += kSym64Warps) S[k][lane] = k < 3 || j < N ? rec[k] : 0.0;
        __syncthreads();
        const bool diag = t == b;
        // off the diagonal rotations 0 .. 31; on it 1 .. 16 meet every pair, those of rotation 16 twice
        const int q0 = diag ? 1 + 16 * part / parts : 32 * part / parts;
        const int q1 = diag ? 1 + 16 * (part + 1) / parts : 32 * (part + 1) / parts;
        Vec3 v = zero;
#pragma unroll 1
        for (int q = q0; q < q1; ++q) {
            const int k = (lane + q) & 31;
            Vec3 F = {S[3][k], S[4][k], S[5][k]}, T = zero, Gq = G, Hq = H;
            if (TORQUE) T = Vec3{S[6 % NS][k], S[7 % NS][k], S[8 % NS][k]};
            if (diag && q == 16 && lane >= 16) F = T = Gq = Hq = zero;
            pair_sym64<TORQUE, WALL>(xi - S[0][k], yi - S[1][k], zi, S[2][k], F, Gq, T, Hq, c, u, v);
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
    const double *__restrict__ tgt_part, const double *__restrict__ src_part, Sym64Plan pl, int N,
    const double *__restrict__ F, const double *__restrict__ T, SelfCoefs sc, double *__restrict__ U)
{
    __shared__ double sum[kRed64Groups][96];
    const int b = pl.nb - 1 - (int)blockIdx.x;  // the longest columns first
    const int tid = threadIdx.x;
    const int g = tid / 96, e = tid - 96 * g;
    const int64_t r0 = sym64_row_run(pl, b) * pl.qs;
    const int nr = (int)((pl.nb - b + pl.L - 1) / pl.L) * pl.qs, nc = b * pl.qs;
    const double *row = tgt_part + r0 * 96 + e, *col = src_part + sym64_col_slot(pl, 0, b, 0) * 96 + e;
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

int mobility_sym64(rpb_ctx *ctx, int N, const double *pos, const double *F, const double *T, double *U, bool packed)
{
    cudaStream_t st = ctx->stream;
    const double a = ctx->p.a;
    const SelfCoefs self = self_coefs(ctx, N);
    const Sym64Consts c64 = make_sym64_consts(a);
    const Sym64Plan pl = sym64_plan(N, ctx->num_sms);
    double *tgt = ctx->ws.sym64, *col = tgt + sym64_tgt_elems(ctx->ws.sym64_N, ctx->num_sms);
    SrcF64 *src = (SrcF64 *)ctx->ws.src;
    const int pb = elem_threads(N, ctx->num_sms);
    if (!packed) pack_f64_kernel<<<(N + pb - 1) / pb, pb, 0, st>>>(pos, F, T, N, a, ctx->p.wall, src, self);
    const dim3 grid((unsigned)pl.runs, (unsigned)pl.qs);
    const int nt = 32 * kSym64Warps;
    if (ctx->p.wall && T)
        pair_sym64_kernel<true, true><<<grid, nt, 0, st>>>(src, N, pl, c64, tgt, col);
    else if (ctx->p.wall)
        pair_sym64_kernel<false, true><<<grid, nt, 0, st>>>(src, N, pl, c64, tgt, col);
    else if (T)
        pair_sym64_kernel<true, false><<<grid, nt, 0, st>>>(src, N, pl, c64, tgt, col);
    else
        pair_sym64_kernel<false, false><<<grid, nt, 0, st>>>(src, N, pl, c64, tgt, col);
    pair_sym64_reduce_kernel<<<pl.nb, kRed64Threads, 0, st>>>(tgt, col, pl, N, F, T, self, U);
    count_launches(packed ? 2 : 3);
    return cuda_fail(cudaGetLastError(), "float64 symmetric pair kernels");
}

}  // namespace rpb
