// cells.cuh -- the steric forces of Sec. III by cell lists, for one suspension (pair.cu) or a packed batch of
// them (batch.cu).
//
// Square cells of side h = the screen radius on an unbounded grid, hashed into G x G buckets by their coordinates
// modulo G (G ~ sqrt(N), a power of two in [64, kCellGrid]; far-away cells that share a bucket only add
// candidates, which the distance screen rejects); heights are not binned.  In a batch every suspension's cells
// are shifted by a hash of its number, and candidates of another suspension are rejected by their index.
// Spheres are put into bucket order by a counting sort and then by index within the bucket, so that every force
// is summed in a fixed order that depends on the sphere's own suspension only.
#pragma once

#include <type_traits>

#include "pair_math.cuh"

namespace rpb {

struct OneSuspension {};  // the template argument that stands for no batch

__device__ __forceinline__ void cell_coords(double x, double y, double inv_h, int &cx, int &cy)
{
    // clamped so that the conversion is defined for any input (non-finite positions land in one cell)
    const double fx = floor(fmin(fmax(x * inv_h, -1e9), 1e9)), fy = floor(fmin(fmax(y * inv_h, -1e9), 1e9));
    cx = fx == fx ? (int)fx : 0;
    cy = fy == fy ? (int)fy : 0;
}
// the cell of a sphere of suspension k of a batch
__device__ __forceinline__ void cell_shift(int k, int &cx, int &cy)
{
    cx += (int)(((unsigned)k * 0x9e3779b1u) >> 16);
    cy += (int)(((unsigned)k * 0x85ebca77u) >> 16);
}
// G x G buckets, G a power of two
__device__ __forceinline__ int cell_bucket(int cx, int cy, int G)
{
    return (cy & (G - 1)) * G + (cx & (G - 1));
}

// cellof[i] = (bucket, place among the spheres counted into it, in any order)
template <bool BATCH>
__global__ void __launch_bounds__(256) cell_count_kernel(const double *__restrict__ pos, int64_t N, double inv_h, int G,
                                                         const int *__restrict__ inst_of, int *__restrict__ count,
                                                         int2 *__restrict__ cellof)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    int cx, cy;
    cell_coords(pos[i], pos[N + i], inv_h, cx, cy);
    if (BATCH) cell_shift(inst_of[i], cx, cy);
    const int c = cell_bucket(cx, cy, G);
    cellof[i] = make_int2(c, atomicAdd(&count[c], 1));
}

// Exclusive scan of the nb = G^2 counts, 4096 buckets a block: a block adds up all counts before its own first
// (from L2) and scans its own.  One block over all 65536 buckets took 40 us at 65536 spheres, of 182 for the forces.
static __global__ void __launch_bounds__(1024) cell_scan_kernel(const int *__restrict__ count, int nb, int *__restrict__ start)
{
    __shared__ int wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int4 *in4 = reinterpret_cast<const int4 *>(count);
    auto block_sum = [&](int v) {  // over all threads, for all of them
        v = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0) wsum[warp] = v;
        __syncthreads();
        const int s = __reduce_add_sync(0xffffffffu, wsum[lane]);
        __syncthreads();
        return s;
    };
    int before = 0;
    const int first = blockIdx.x * 1024;
#pragma unroll 4
    for (int k = tid; k < first; k += 1024) {
        const int4 q = in4[k];
        before += (q.x + q.y) + (q.z + q.w);
    }
    before = block_sum(before);
    const int4 q = in4[first + tid];
    const int s = (q.x + q.y) + (q.z + q.w);
    int inc = s;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    const int warps = __reduce_add_sync(0xffffffffu, lane < warp ? wsum[lane] : 0);
    int4 o;
    o.x = before + warps + inc - s;
    o.y = o.x + q.x;
    o.z = o.y + q.y;
    o.w = o.z + q.z;
    reinterpret_cast<int4 *>(start)[first + tid] = o;
    if (4 * (first + tid + 1) == nb) start[nb] = o.w + q.w;
}

static __global__ void __launch_bounds__(256) cell_place_kernel(int64_t N, const int2 *__restrict__ cellof,
                                                                const int *__restrict__ start, int *__restrict__ any)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int2 c = cellof[i];
    any[start[c.x] + c.y] = (int)i;
}

// Spheres by index within their buckets, a thread per sphere (a thread per bucket, sorting in place, took 14 us
// at 65536 spheres against 4): its place is the number of smaller indices in the bucket.  Outside batches a
// bucket of more than kCellMaxSorted spheres is left to the all-pairs kernel.  The force of the wall and the
// weight are put into Fz here, where a warp has 32 spheres.
template <bool BATCH>
__global__ void __launch_bounds__(256) cell_order_kernel(const double *__restrict__ pos, int64_t N,
                                                         const int2 *__restrict__ cellof, const int *__restrict__ start,
                                                         const int *__restrict__ any,
                                                         float4 *__restrict__ posf, double *__restrict__ posd,
                                                         CellHeader *__restrict__ hdr, double a, double weight,
                                                         double f0, double b, double inv_b, double *__restrict__ Fz)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int c = cellof[i].x, a0 = start[c], a1 = start[c + 1];
    if (!BATCH && a1 - a0 > kCellMaxSorted) {
        hdr->overfull = 1;  // every writer stores the same value
        return;
    }
    int k = a0;
#pragma unroll 4
    for (int m = a0; m < a1; ++m) k += any[m] < (int)i;
    const double x = pos[i], y = pos[N + i], z = pos[2 * N + i];
    posf[k] = make_float4((float)x, (float)y, (float)z, __int_as_float((int)i));
    posd[k] = x;
    posd[N + k] = y;
    posd[2 * N + k] = z;
    Fz[i] = wall_force(z, a, weight, f0, b, inv_b);
}

// Force pass over the buckets, kCellLanes threads per sphere in bucket order (neighbouring groups search the same
// buckets): the three rows of three cells are up to six runs of consecutive places; candidates are screened in
// float32, the group's hits go to its list in order and are evaluated in float64, one of kCellLanes by each
// thread.  What bounds it is the float64 of the pairs (32 warp instructions of 64 cycles each; the pipe is busy
// for 76% of its time): a thread per sphere paid for the longest list of 32 and left four warps on some schedulers
// and three on others.  65536 spheres: this kernel 111 -> 86 us, the forces 182 -> 119 (8 threads a sphere 121,
// 2 128, 1 173); 8193: 78 -> 49.
// In a batch, pairs farther apart than 2a + kFarB b (near2), whose repulsion is below e^-kFarB U0/b (~2e-9 U0/b),
// take it in float32 from the list's other end (IEEE square root and division, expf: a relative error of a few 1e-6 on
// a term that small is below 1e-14 U0/b) and are summed in float32 before their total joins the float64 sum.
constexpr double kFarB = 20.0;
constexpr int kCellLanes = 4, kCellList = 64;

template <class Inst>
__global__ void __launch_bounds__(128) forces_cell_kernel(int64_t N, double two_a, double f0, double inv_b, float cut2,
                                                          float near2, int G, const CellHeader *__restrict__ hdr,
                                                          const int *__restrict__ start, const int2 *__restrict__ cellof,
                                                          const float4 *__restrict__ posf, const double *__restrict__ posd,
                                                          const Inst *__restrict__ inst,
                                                          const int *__restrict__ inst_of, double *__restrict__ F)
{
    constexpr bool BATCH = !std::is_same<Inst, OneSuspension>::value;
    __shared__ int list[128 / kCellLanes][kCellList];
    if (!BATCH && cell_overfull(hdr)) return;
    const int tid = threadIdx.x, p = tid % kCellLanes, g = tid / kCellLanes;
    const int64_t k = (int64_t)blockIdx.x * (128 / kCellLanes) + g;
    if (k >= N) return;  // whole groups
    const unsigned group = ((1u << kCellLanes) - 1) << (tid & 31 & ~(kCellLanes - 1));
    const float4 own = posf[k];
    const float xf = own.x, yf = own.y, zf = own.z;
    const double xi = posd[k], yi = posd[N + k], zi = posd[2 * N + k];
    const int i = __float_as_int(own.w), c = cellof[i].x;
    const int cx = c & (G - 1), cy = c / G;
    unsigned off = 0, Ni = 0;
    if constexpr (BATCH) {
        const int q = inst_of[i];
        off = (unsigned)inst[q].off;
        Ni = (unsigned)inst[q].N;
    }
    double fx = 0.0, fy = 0.0, fz = 0.0;
    float gx = 0.f, gy = 0.f, gz = 0.f;  // far pairs
    int nn = 0, nf = 0;  // near pairs at list[0 .. nn), far pairs at list[kCellList - nf .. kCellList)
    auto flush = [&]() {
        __syncwarp(group);
        for (int e = p; e < nn; e += kCellLanes) {
            const int m = list[g][e];
            const double dx = xi - posd[m], dy = yi - posd[N + m], dz = zi - posd[2 * N + m];
            const double s = steric_pair_factor(dx * dx + dy * dy + dz * dz, two_a, f0, inv_b);
            fx += s * dx;
            fy += s * dy;
            fz += s * dz;
        }
        if (BATCH) {
            const float f0f = (float)f0, inv_bf = (float)inv_b, two_af = (float)two_a;
            for (int e = kCellList - 1 - p; e >= kCellList - nf; e -= kCellLanes) {
                const int m = list[g][e];
                const float dx = (float)(xi - posd[m]), dy = (float)(yi - posd[N + m]), dz = (float)(zi - posd[2 * N + m]);
                const float r = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
                const float s = f0f * expf((two_af - r) * inv_bf) / r;
                gx = fmaf(s, dx, gx);
                gy = fmaf(s, dy, gy);
                gz = fmaf(s, dz, gz);
            }
        }
        __syncwarp(group);  // the list is written again
        nn = nf = 0;
    };
    const unsigned below = group & ((1u << (tid & 31)) - 1);
    auto search = [&](int m0, int m1) {
        for (int mb = m0; mb < m1; mb += kCellLanes) {
            const int m = mb + p;
            float d2 = INFINITY;
            if (m < m1 && m != k) {
                const float4 q = posf[m];
                const float ex = xf - q.x, ey = yf - q.y, ez = zf - q.z;
                d2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
                if (BATCH && (unsigned)__float_as_int(q.w) - off >= Ni) d2 = INFINITY;
            }
            const bool near = d2 < (BATCH ? near2 : cut2);
            const unsigned hit = __ballot_sync(group, near);
            if (near) list[g][nn + __popc(hit & below)] = m;
            nn += __popc(hit);
            if (BATCH) {
                const bool far = !near && d2 < cut2;
                const unsigned hf = __ballot_sync(group, far);
                if (far) list[g][kCellList - 1 - nf - __popc(hf & below)] = m;
                nf += __popc(hf);
            }
            if (nn + nf > kCellList - kCellLanes) flush();
        }
    };
    const int x0 = (cx - 1) & (G - 1);
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
        const int *row = start + ((cy + dy) & (G - 1)) * G;
        search(row[x0], row[min(x0 + 3, G)]);
        if (x0 + 3 > G) search(row[0], row[x0 + 3 - G]);
    }
    flush();
#pragma unroll
    for (int o = kCellLanes / 2; o > 0; o >>= 1) {
        fx += __shfl_xor_sync(group, fx, o);
        fy += __shfl_xor_sync(group, fy, o);
        fz += __shfl_xor_sync(group, fz, o);
        if (BATCH) {
            gx += __shfl_xor_sync(group, gx, o);
            gy += __shfl_xor_sync(group, gy, o);
            gz += __shfl_xor_sync(group, gz, o);
        }
    }
    if (p == 0) {
        if (BATCH) {
            fx += (double)gx;
            fy += (double)gy;
            fz += (double)gz;
        }
        F[i] = fx;
        F[N + i] = fy;
        F[2 * N + i] += fz;
    }
}

// The whole pass; cut and near are the screen radii (near only for a batch), N the spheres of all suspensions.
template <class Inst>
inline int cell_forces(cudaStream_t st, const CellLists &L, const double *pos, int64_t N, double a, double weight, double U0,
                       double b, double cut, double near, const Inst *inst, const int *inst_of, double *F)
{
    constexpr bool BATCH = !std::is_same<Inst, OneSuspension>::value;
    const double inv_h = 1.0 / cut;
    const int G = cell_grid(N), nb = G * G;
    const unsigned blocks = (unsigned)((N + 255) / 256);
    int rc;
    // the header (overfull flag) and the bucket counts are contiguous: one clear
    if ((rc = cuda_fail(cudaMemsetAsync(L.hdr, 0, sizeof(CellHeader) + sizeof(int) * (size_t)nb, st), "clear cell counts")))
        return rc;
    cell_count_kernel<BATCH><<<blocks, 256, 0, st>>>(pos, N, inv_h, G, inst_of, L.count, L.cellof);
    cell_scan_kernel<<<nb / 4096, 1024, 0, st>>>(L.count, nb, L.start);
    cell_place_kernel<<<blocks, 256, 0, st>>>(N, L.cellof, L.start, L.any);
    const double f0 = U0 / b, inv_b = 1.0 / b;
    cell_order_kernel<BATCH><<<blocks, 256, 0, st>>>(pos, N, L.cellof, L.start, L.any, L.posf, L.posd, L.hdr, a, weight, f0,
                                                     b, inv_b, F + 2 * N);
    constexpr int per = 128 / kCellLanes;
    forces_cell_kernel<Inst><<<(unsigned)((N + per - 1) / per), 128, 0, st>>>(
        N, 2.0 * a, f0, inv_b, (float)(cut * cut), (float)(near * near), G, L.hdr, L.start, L.cellof, L.posf, L.posd, inst,
        inst_of, F);
    count_launches(5);
    return cuda_fail(cudaGetLastError(), "force kernels");
}

}  // namespace rpb
