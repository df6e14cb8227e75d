// lanczos_math.cuh -- tridiagonal step of the Lanczos square root shared by the single and batched
// kernels: y_k = |W| T_{k+1}^{1/2} e_1 for the tridiagonal T_{k+1}, the error estimate eps_k and the
// stopping decision (Sec. II.C).  128 threads per Krylov space evaluate a rational
// approximation of the square root, one node per thread; a T that is not positive definite takes the
// eigen-decomposition, one warp.
#pragma once

#include <cfloat>

#include "rpb_internal.cuh"
#include "sqrt_nodes.h"

namespace rpb {

constexpr int kMaxIter = 64;      // largest supported Lanczos dimension

// Layout of the small state block (doubles).
struct LzLayout {
    int M;
    size_t alpha, beta, y, yprev, c1, c2, coef, status, total;
    explicit LzLayout(int max_iter) : M(max_iter)
    {
        size_t o = 0;
        alpha = o; o += M + 1;
        beta = o; o += M + 1;
        y = o; o += M + 1;
        yprev = o; o += M + 1;
        c1 = o; o += M + 1;
        c2 = o; o += M + 1;
        coef = o; o += M + 1;
        status = o; o += 8;
        total = o;
    }
};
// status words
enum { ST_EPS = 0, ST_INV_BETA = 1, ST_NW = 2, ST_INV_NW = 3, ST_STOP = 4, ST_BREAK = 5 };

// Symmetric tridiagonal eigen-decomposition by the implicit QL method with a Wilkinson-type shift
// (Bowdler, Martin, Reinsch & Wilkinson), then y = |W| Q sqrt(max(Lambda, 0)) Q^T e_1.
// Called by one full warp: every lane runs the (identical) scalar recurrence on private copies of d
// and e and applies the rotations to its own rows (lane, lane + 32) of Q, so no lane reads another's
// data until the end.  alpha, beta: the entries of T (k + 1 and k of them); q0, sl: shared scratch
// (kMaxIter doubles each).  Lane i returns entries i and i + 32 of y in y0, y1.
static __device__ __noinline__ void tridiag_sqrt_ql(const double *alpha, const double *beta, int k, double nW, double *q0,
                                             double *sl, double *y_out0, double *y_out1)
{
    const int lane = threadIdx.x & 31;
    const int n = k + 1;
    double d[kMaxIter], e[kMaxIter], z0[kMaxIter], z1[kMaxIter];
    for (int i = 0; i < n; ++i) {
        d[i] = alpha[i];
        e[i] = (i < k) ? beta[i] : 0.0;
        z0[i] = (i == lane) ? 1.0 : 0.0;
        z1[i] = (i == lane + 32) ? 1.0 : 0.0;
    }
    for (int l = 0; l < n; ++l) {
        for (int iter = 0; iter < 100; ++iter) {
            int m = l;
            for (; m < n - 1; ++m) {
                const double dd = fabs(d[m]) + fabs(d[m + 1]);
                if (fabs(e[m]) <= DBL_EPSILON * dd) break;
            }
            if (m == l) break;
            double g = (d[l + 1] - d[l]) / (2.0 * e[l]);
            // |g| <= |d| / (2 DBL_EPSILON |d|) here (e[l] passed the test above), so g^2 + 1 cannot
            // overflow and the square root needs no hypot
            double r = sqrt(fma(g, g, 1.0));
            g = d[m] - d[l] + e[l] / (g + copysign(r, g));
            double s = 1.0, c = 1.0, p = 0.0;
            bool restart = false;
            for (int i = m - 1; i >= l; --i) {
                const double f = s * e[i];
                const double bb = c * e[i];
                // Givens rotation from one reciprocal square root (the entries of T are of the order
                // of the mobility, far from the float64 overflow and underflow limits)
                const double r2 = fma(f, f, g * g);
                if (r2 == 0.0) {
                    e[i + 1] = 0.0;
                    d[i + 1] -= p;
                    e[m] = 0.0;
                    restart = true;
                    break;
                }
                const double ir = rsqrt(r2);
                e[i + 1] = r2 * ir;
                s = f * ir;
                c = g * ir;
                g = d[i + 1] - p;
                r = (d[i] - g) * s + 2.0 * c * bb;
                p = s * r;
                d[i + 1] = g + p;
                g = c * r - bb;
                const double a0 = z0[i + 1];
                z0[i + 1] = s * z0[i] + c * a0;
                z0[i] = c * z0[i] - s * a0;
                if (n > 32) {  // rows lane + 32 exist only beyond 32 dimensions (float64 costs per warp instruction)
                    const double a1 = z1[i + 1];
                    z1[i + 1] = s * z1[i] + c * a1;
                    z1[i] = c * z1[i] - s * a1;
                }
            }
            if (restart) continue;
            d[l] -= p;
            e[l] = g;
            e[m] = 0.0;
        }
    }
    if (lane == 0)
        for (int j = 0; j < n; ++j) q0[j] = z0[j];
    // the eigenvalues are the same in every lane: lane j takes the square root of the j-th
    if (lane < n) sl[lane] = sqrt(fmax(d[lane], 0.0));
    if (lane + 32 < n) sl[lane + 32] = sqrt(fmax(d[lane + 32], 0.0));
    __syncwarp();
    double y0 = 0.0, y1 = 0.0;
    for (int j = 0; j < n; ++j) {
        const double cj = sl[j] * q0[j];
        y0 = fma(z0[j], cj, y0);
        if (n > 32) y1 = fma(z1[j], cj, y1);
    }
    *y_out0 = y0 * nW;
    *y_out1 = y1 * nW;
}

constexpr int kTailThreads = kSqrtNodes;  // one node per thread
constexpr int kTailRows = 16;             // entries of y summed over the nodes at a time
struct TailShared {
    double al[kMaxIter], be[kMaxIter], b2[kMaxIter];  // the entries of T, beta^2
    double y[kMaxIter], yprev[kMaxIter];
    double q0[kMaxIter], sl[kMaxIter];                // eigen-decomposition
    double z[kTailRows][kSqrtNodes + 8];              // the nodes' terms (padded: the sums read 8 columns of
                                                      // four rows at a time)
};

// Largest of the lanes' non-negative values: the bit patterns of non-negative doubles order as integers,
// so this leaves the float64 pipe alone.
__device__ __forceinline__ double warp_max_pos(double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long q = __shfl_xor_sync(0xffffffffu, b, o);
        b = q > b ? q : b;
    }
    return __longlong_as_double((long long)b);
}

// Barrier 1 among the kTailThreads threads of a tridiagonal step (their block may have more), and the
// or of a predicate over them.
__device__ __forceinline__ void tail_sync()
{
    asm volatile("bar.sync 1, %0;" ::"n"(kTailThreads) : "memory");
}
__device__ __forceinline__ bool tail_any(bool p)
{
    unsigned r;
    asm volatile("{\n\t.reg .pred a, b;\n\tsetp.ne.u32 a, %1, 0;\n\tbar.red.or.pred b, 1, %2, a;\n\t"
                 "selp.u32 %0, 1, 0, b;\n\t}"
                 : "=r"(r)
                 : "r"((unsigned)p), "n"(kTailThreads)
                 : "memory");
    return r != 0;
}

// The tridiagonal step of one Krylov space by kTailThreads threads (tid: 0 .. kTailThreads - 1), in three parts.
// lanczos_tail_load fetches what is known before iteration k's projections: the nodes (kSqrtNodes shifts, then as
// many weights, sqrt_nodes.h), the entries of T_k, the last y and |W|.
struct TailRegs {
    double s, w, nW;
};
__device__ __forceinline__ TailRegs lanczos_tail_load(const double *__restrict__ lz, const LzLayout &L, int k,
                                                      const double *__restrict__ nodes, TailShared &sh, int tid)
{
    if (tid < k) {
        const double b = lz[L.beta + tid];
        sh.al[tid] = lz[L.alpha + tid];
        sh.be[tid] = b;
        sh.b2[tid] = b * b;
        sh.yprev[tid] = lz[L.yprev + tid];
    }
    if (tid == k) sh.be[k] = sh.b2[k] = sh.yprev[k] = 0.0;
    return TailRegs{nodes[tid], nodes[kSqrtNodes + tid], lz[L.status + ST_NW]};
}

// lanczos_tail_y: with alpha_k, stores alpha_k and y; thread 0 returns eps and the largest entry of T.
//
// With T = tridiag(beta, alpha, beta) scaled by M, the power of four above its Gershgorin bound (its square
// root is exact and costs nothing), y = |W| T^{1/2} e_1 ~ |W| sqrt(M) sum_j w_j T (T + M s_j)^{-1} e_1.  Thread j solves its shifted system by eliminating from
// the last row up: c_i = alpha_i - beta_i^2 / d_{i+1}, d_i = c_i + s; then x_0 = 1/d_0,
// x_{i+1} = -(beta_i / d_{i+1}) x_i, and (T x)_0 = c_0 x_0, (T x)_i = -s x_i, with no cancellation.
// Everything is backward stable for a positive definite T (relative errors of a few 1e-16 in y, against
// 1e-15 to 1e-13 of an eigen-decomposition); a pivot that is not positive (or not finite) in some
// thread shows a T that is not, and the block takes the eigen-decomposition instead, whose negative
// eigenvalues (rounding of a semi-definite mobility) are clamped to 0.
//
// What bounds it: the float64 chain of one elimination, about 7 instructions per row and thread, each
// 64 cycles of a scheduler whatever the active lanes.  The eigen-decomposition is a chain of about
// 1.7 k^2 / 2 rotations of 28 such instructions on one warp: 48 us per launch on average over the
// iterations of a converging solve of 8 dimensions and 164 us over one of 19; with the nodes a
// 3001-sphere free-space solve (18 iterations, float32 pairs) went from 3251 to 1211 us and a step of 4096
// spheres from 1103 to 1004 us.
struct TailResult {
    double eps, tnorm;
};
__device__ __forceinline__ TailResult lanczos_tail_y(double *__restrict__ lz, const LzLayout &L, int k, double alpha_k,
                                                     const TailRegs &reg, TailShared &sh, int tid)
{
    const int lane = tid & 31;
    const int n = k + 1;
    const double sj = reg.s, wj = reg.w, nW = reg.nW;
    TailResult res = {-1.0, 0.0};
    if (tid == 0) sh.al[k] = alpha_k;
    tail_sync();
    // Gershgorin bound and largest entry (every warp, over the entries lane and lane + 32)
    double mb = 0.0, mt = 0.0;
    for (int i = lane; i < n; i += 32) {
        const double a = fabs(sh.al[i]), b = fabs(sh.be[i]);
        mb = fmax(mb, a + b + (i > 0 ? fabs(sh.be[i - 1]) : 0.0));
        mt = fmax(mt, fmax(a, b));
    }
    // M = 4^e >= the bound, sqrt(M) = 2^e (a bound that is not a plain positive number fails the pivots' test)
    const double bound = warp_max_pos(mb);
    const int e4 = plain_pos(bound) ? ((__double2hiint(bound) >> 20) - 1023 + 2) >> 1 : 0;
    const double M = __hiloint2double((1023 + 2 * e4) << 20, 0), rootM = __hiloint2double((1023 + e4) << 20, 0);
    res.tnorm = warp_max_pos(mt);
    const double s = M * sj;
    double r[kMaxIter];
    double c = sh.al[k];
    double d = c + s;
    bool ok = plain_pos(d) && plain_pos(bound);
    double ri = rcp_pos(d);
    r[k] = ri;
    for (int i = k - 1; i >= 0; --i) {
        c = fma(-sh.b2[i], ri, sh.al[i]);
        d = c + s;
        ok = ok && plain_pos(d);
        ri = rcp_pos(d);
        r[i] = ri;
    }
    if (tail_any(!ok)) {
        if (tid >= 32) return res;  // (no barrier follows for the first warp on this path)
        double y0, y1;
        tridiag_sqrt_ql(sh.al, sh.be, k, nW, sh.q0, sh.sl, &y0, &y1);
        if (lane < n) sh.y[lane] = y0;
        if (lane + 32 < n) sh.y[lane + 32] = y1;
        __syncwarp();
    } else {
        const double scale = rootM * nW;
        const double x0 = wj * ri;
        double z = -(s * x0);
        for (int base = 0; base < n; base += kTailRows) {
            const int m = min(kTailRows, n - base);
            for (int i = 0; i < m; ++i) {
                if (base + i > 0) z = -(sh.be[base + i - 1] * r[base + i]) * z;
                sh.z[i][tid] = base + i > 0 ? z : c * x0;
            }
            tail_sync();
            // eight threads per entry, 16 for up to eight entries: 16 or 8 nodes each, then the butterfly
            // levels (a fixed order)
            const int lg = n <= 8 ? 4 : 3, row = tid >> lg, p = tid & ((1 << lg) - 1);
            double v = 0.0;
            if (row < m)
                for (int u = p; u < kSqrtNodes; u += 1 << lg) v += sh.z[row][u];
            if (lg == 4) v += __shfl_xor_sync(0xffffffffu, v, 8);
            for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (p == 0 && row < m) sh.y[base + row] = v * scale;
            tail_sync();
        }
        if (tid >= 32) return res;
    }
    // eps_k = |y - (yprev, 0)| / |yprev|: lanes 0 .. 15 sum the numerator, 16 .. 31 the denominator
    const bool upper = lane >= 16;
    double sq = 0.0;
    for (int i = lane & 15; i < n; i += 16) {
        const double p = sh.yprev[i];
        const double d = upper ? p : sh.y[i] - p;
        sq = fma(d, d, sq);
    }
    for (int i = lane; i < n; i += 32) lz[L.y + i] = lz[L.yprev + i] = sh.y[i];
    for (int o = 8; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    const double den = __shfl_sync(0xffffffffu, sq, 16);
    const double num = sq;  // in lane 0
    if (lane == 0) {
        lz[L.alpha + k] = alpha_k;
        if (k >= 1 && den > 0.0) {
            const double q = plain_pos(den) ? num * rcp_pos(den) : num / den;
            res.eps = plain_pos(q) ? q * rsqrt_pos(q) : sqrt(q);
        }
    }
    return res;
}

// lanczos_tail_stop, by one thread: with beta_k, stores it and the stopping decision (*hs: also there, null:
// nowhere); returns whether the iteration stops.
__device__ __forceinline__ bool lanczos_tail_stop(double *__restrict__ lz, const LzLayout &L, int k, double tol,
                                                  double beta_k, const TailResult &r, double nW, double *hs)
{
    double *status = lz + L.status;
    lz[L.beta + k] = beta_k;
    const bool brk = beta_k <= 1e-14 * fmax(r.tnorm, beta_k);
    const bool stop = brk || (tol > 0.0 && k >= 1 && r.eps <= tol);
    status[ST_EPS] = r.eps;
    status[ST_BREAK] = brk ? 1.0 : 0.0;
    status[ST_STOP] = stop ? 1.0 : 0.0;
    status[ST_INV_BETA] = brk ? 0.0 : (plain_pos(beta_k) ? rcp_pos(beta_k) : 1.0 / beta_k);
    if (hs) {
        hs[ST_EPS] = r.eps;
        hs[ST_NW] = nW;
        hs[ST_STOP] = stop ? 1.0 : 0.0;
    }
    return stop;
}

}  // namespace rpb
