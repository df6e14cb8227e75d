// gs.cuh -- device side of the Gram-Schmidt steps of the Lanczos iteration (classical Gram-Schmidt
// applied twice, Sec. II.C), on blocks of kGsThreads threads that each own a chunk of spheres.
//
// What bounds them: float64 instructions (64 cycles of a scheduler per warp instruction), not memory.  A
// thread keeps its rows of w in registers; dot products are taken eight basis vectors at a time, so
// that summing them over a warp costs nine additions for the eight (a reduce-scatter over the lanes)
// instead of forty.
#pragma once

#include "lanczos_math.cuh"

namespace rpb {

constexpr int kGsThreads = 256;
constexpr int kGsWarps = kGsThreads / 32;
constexpr int kGsChunk = 256;                              // spheres of a chunk at most
constexpr int kGsRows = 3 * kGsChunk / kGsThreads;         // rows (sphere, component) of a thread

// Barrier 2 among a block's first kGsThreads threads (a block may have others beside them).
__device__ __forceinline__ void gs_sync()
{
    asm volatile("bar.sync 2, %0;" ::"n"(kGsThreads) : "memory");
}

// Rows of a chunk: components x, y, z of `cnt` spheres at offsets base + c stride + i.
struct GsSpan {
    int64_t base, stride;
    int cnt;
};

// Offsets of this thread's rows (component-major in the chunk); -1 past the end.  Returns the number of rows that
// some lane of the warp has: the loops over the rows run to it, since a float64 instruction costs the same
// with no lane active.
__device__ __forceinline__ int gs_rows(const GsSpan &s, int64_t (&row)[kGsRows])
{
#pragma unroll
    for (int u = 0; u < kGsRows; ++u) {
        const int r = threadIdx.x + u * kGsThreads;
        const int c = r < s.cnt ? 0 : (r < 2 * s.cnt ? 1 : 2);
        row[u] = r < 3 * s.cnt ? s.base + c * s.stride + (r - c * s.cnt) : -1;
    }
    const int left = 3 * s.cnt - (int)(threadIdx.x & ~31u);
    return left <= 0 ? 0 : min(kGsRows, (left + kGsThreads - 1) / kGsThreads);
}
// Warps of the block that have rows.
__device__ __forceinline__ int gs_warps(const GsSpan &s)
{
    return min(kGsWarps, (3 * s.cnt + 31) / 32);
}

// Sums over the warp of eight values per lane: lane l returns the sum of v[l >> 2] (a fixed order).
__device__ __forceinline__ double warp_sum8(double (&v)[8])
{
    const int lane = threadIdx.x & 31;
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    double a[4], b[2];
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = (b4 ? v[q + 4] : v[q]) + __shfl_xor_sync(0xffffffffu, b4 ? v[q] : v[q + 4], 16);
#pragma unroll
    for (int q = 0; q < 2; ++q) b[q] = (b3 ? a[q + 2] : a[q]) + __shfl_xor_sync(0xffffffffu, b3 ? a[q] : a[q + 2], 8);
    double s = (b2 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, b2 ? b[0] : b[1], 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    return s + __shfl_xor_sync(0xffffffffu, s, 1);
}

// Sum over the block of one value per thread, in the first warp's threads; sh: kGsWarps doubles.
__device__ __forceinline__ double gs_block_sum(double v, int nu, int nw, double *sh)
{
    const int lane = threadIdx.x & 31;
    if (nu > 0) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sh[threadIdx.x >> 5] = v;
    }
    gs_sync();
    double s = 0.0;
    if (threadIdx.x < 32) {
        s = lane < nw ? sh[lane] : 0.0;
        for (int o = kGsWarps / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        s = __shfl_sync(0xffffffffu, s, 0);  // the first kGsWarps lanes hold the sum
    }
    return s;
}

template <int NU>
__device__ __forceinline__ void gs_dots_rows(const double *__restrict__ V, size_t ld, int nvec,
                                             const int64_t (&row)[kGsRows], const double (&w)[kGsRows], double *sh)
{
    const int lane = threadIdx.x & 31;
    for (int j0 = 0; j0 < nvec; j0 += 8) {
        double acc[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            acc[q] = 0.0;
            if (j0 + q < nvec) {
                const double *v = V + (size_t)(j0 + q) * ld;
#pragma unroll
                for (int u = 0; u < NU; ++u)
                    if (row[u] >= 0) acc[q] = fma(v[row[u]], w[u], acc[q]);
            }
        }
        const double s = warp_sum8(acc);
        if ((lane & 3) == 0) sh[j0 + (lane >> 2)] = s;
    }
}

// The block's part of <V_j, w>, j < nvec: thread j < nvec returns it (nvec <= kGsThreads).
// sh: kGsWarps x (kMaxIter + 8) doubles; nu, nw: gs_rows, gs_warps.
__device__ __forceinline__ double gs_dots(const double *__restrict__ V, size_t ld, int nvec, const int64_t (&row)[kGsRows],
                                          int nu, int nw, const double (&w)[kGsRows], double (*sh)[kMaxIter + 8])
{
    static_assert(kGsRows == 3, "one case per number of rows");
    double *mine = sh[threadIdx.x >> 5];
    if (nu == 1)
        gs_dots_rows<1>(V, ld, nvec, row, w, mine);
    else if (nu == 2)
        gs_dots_rows<2>(V, ld, nvec, row, w, mine);
    else if (nu == 3)
        gs_dots_rows<3>(V, ld, nvec, row, w, mine);
    gs_sync();
    double s = 0.0;
    if (threadIdx.x < nvec)
        for (int k = 0; k < nw; ++k) s += sh[k][threadIdx.x];
    return s;
}

template <int NU>
__device__ __forceinline__ void gs_project_rows(const double *__restrict__ V, size_t ld, int nvec,
                                                const int64_t (&row)[kGsRows], const double *coef, double (&w)[kGsRows])
{
#pragma unroll 4
    for (int j = 0; j < nvec; ++j) {
        const double *v = V + (size_t)j * ld;
        const double m = -coef[j];
#pragma unroll
        for (int u = 0; u < NU; ++u)
            if (row[u] >= 0) w[u] = fma(m, v[row[u]], w[u]);
    }
}

// w -= sum_j coef_j V_j
__device__ __forceinline__ void gs_project(const double *__restrict__ V, size_t ld, int nvec, const int64_t (&row)[kGsRows],
                                           int nu, const double *coef, double (&w)[kGsRows])
{
    if (nu == 1)
        gs_project_rows<1>(V, ld, nvec, row, coef, w);
    else if (nu == 2)
        gs_project_rows<2>(V, ld, nvec, row, coef, w);
    else if (nu == 3)
        gs_project_rows<3>(V, ld, nvec, row, coef, w);
}

// coef_j = sum of n partials red[j rs + k], j < nvec, by one warp per vector in a fixed order; ends with a
// block barrier.
__device__ __forceinline__ void gs_coefs(const double *__restrict__ red, size_t rs, int n, int nvec, double *coef)
{
    const int lane = threadIdx.x & 31;
    for (int j = threadIdx.x >> 5; j < nvec; j += kGsWarps) {
        double s = 0.0;
        for (int k = lane; k < n; k += 32) s += red[(size_t)j * rs + k];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) coef[j] = s;
    }
    gs_sync();
}

}  // namespace rpb
