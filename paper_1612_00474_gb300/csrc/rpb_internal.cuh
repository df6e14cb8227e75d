// rpb_internal.cuh -- shared declarations of the CUDA translation units (not part of the ABI).
#pragma once

#include <utility>

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/rpb.h"

namespace rpb {

constexpr int kTile = 128;        // sources staged per shared-memory tile = targets per block
constexpr int kPairThreads = 128; // threads per pair-kernel block (one target each)
constexpr double kPi = 3.14159265358979323846;

// Packed source records, built once per product from the float64 SoA inputs.
// s_j = H0(z_j / a) is folded into F and T; z is the clamped height max(z, a) (Appendix A).
struct alignas(16) SrcF32 {
    float4 p;  // x_hi, y_hi, x_lo, y_lo   (x = x_hi + x_lo exactly to ~2^-48 relative)
    float4 f;  // z~, s Fx, s Fy, s Fz
    float4 t;  // s Tx, s Ty, s Tz, 0
};
struct alignas(16) SrcF64 {
    double2 p;  // x, y
    double2 q;  // z~, s Fx
    double2 r;  // s Fy, s Fz
    double2 s;  // s Tx, s Ty
    double2 u;  // s Tz, 0
};

#ifdef __CUDACC__
// 1/sqrt(x) for a positive normal x: the hardware's approximation (relative error measured at 2^-20.0), then one
// third-order step of the binomial series, y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2 (Householder's
// iteration): it leaves 5 e^3/16 = 2^-58.7, below rounding.  The approximation has zeros in its lower 32 bits, so its
// square is exact and e is rounded once: within 0.53 ulp.  (With e from x y, rounded, it was 0.98 ulp, and the
// float64 products of 500 spheres had 3.7e-16 of error where the library's root had given 3.4e-16.)
__device__ __forceinline__ double rsqrt_pos(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y * y, 1.0);
    return fma(e * y, fma(e, 0.375, 0.5), y);
}

// 1/d for a positive normal d: the hardware's approximation (relative error measured at 2^-19.9) and one
// third-order step of Householder's iteration, y (1 + e + e^2) with e = 1 - d y: within 0.52 ulp.
__device__ __forceinline__ double rcp_pos(double d)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// Positive and normal, below 2^1000: on the exponent bits (false for NaN).
__device__ __forceinline__ bool plain_pos(double v)
{
    return (unsigned)(__double2hiint(v) - 0x00100000) < 0x7e600000u;
}

// sqrt(x) and 1/sqrt(x) of a sum of squares: a square root and a division are about 25 float64 instructions,
// the reciprocal root 5 and the root 4 more (one Newton step: within 0.51 ulp while its residual is a normal number).
__device__ __forceinline__ void root_and_inverse(double x, double *root, double *inverse)
{
    if (plain_pos(x)) {
        const double y = rsqrt_pos(x), r = x * y;
        *inverse = y;
        *root = __double2hiint(x) >= 0x04000000 ? fma(fma(-r, r, x), 0.5 * y, r) : sqrt(x);  // from 2^-959 on
    } else {
        *root = sqrt(x);
        *inverse = 1.0 / *root;
    }
}
#endif

// Geometry constants of the pair formula, in units where velocities carry 1/(8 pi eta).
template <typename R>
struct PairConsts {
    R two_a;        // 2a
    R two_a2;       // 2a^2
    R two_3_a2;     // 2a^2/3
    R a2;           // a^2
    R near_c1;      // 4/(3a)          (mu0 in units of 1/(8 pi eta))
    R near_r;       // 9/(32a)
    R near_c2;      // 1/(8 a^2)
    R near_tr;      // 1/(2 a^3)
    R near_tr_r;    // 3/(8a)
    R four_a2;      // 4a^2 (overlap test on r^2)
};

template <typename R>
inline PairConsts<R> make_consts(double a)
{
    PairConsts<R> c;
    c.two_a = (R)(2.0 * a);
    c.two_a2 = (R)(2.0 * a * a);
    c.two_3_a2 = (R)(2.0 * a * a / 3.0);
    c.a2 = (R)(a * a);
    c.near_c1 = (R)(4.0 / (3.0 * a));
    c.near_r = (R)(9.0 / (32.0 * a));
    c.near_c2 = (R)(1.0 / (8.0 * a * a));
    c.near_tr = (R)(1.0 / (2.0 * a * a * a));
    c.near_tr_r = (R)(3.0 / (8.0 * a));
    c.four_a2 = (R)(4.0 * a * a);
    return c;
}

// Pair forces beyond 2a + kForceCutoffB b are left out: there the soft repulsion is below
// e^{-40} U0/b ~ 4e-18 U0/b, far under the float64 rounding of any force it would be added to.
constexpr double kForceCutoffB = 40.0;

// Cell lists of the force pass (cells.cuh): header, then the arrays in one allocation.
constexpr int kCellGrid = 1024;     // at most kCellGrid x kCellGrid buckets (cells hashed modulo G)
constexpr int kCellMaxSorted = 512;  // a fuller cell hands the force pass to the all-pairs kernel
struct CellHeader {
    int overfull, pad[15];  // 64 bytes, followed by the bucket counts
};
__device__ __forceinline__ bool cell_overfull(const CellHeader *h)
{
    return *(volatile const int *)&h->overfull != 0;
}
struct CellLists {
    CellHeader *hdr;
    int *count, *start;  // G^2 and G^2 + 1 entries
    float4 *posf;        // in bucket order: float32 copies (x, y, z, index bits)
    double *posd;        // ... the positions (SoA)
    int2 *cellof;
    int *any;
};
inline int cell_grid(int64_t N)
{
    int G = 64;
    while (G < kCellGrid && (int64_t)2 * G * G < N) G *= 2;  // about 5 spheres a cell: at least one bucket for 2
    return G;
}
inline size_t cell_lists_bytes(int64_t max_N)
{
    const size_t nb = (size_t)cell_grid(max_N) * cell_grid(max_N);
    return sizeof(CellHeader) + sizeof(int) * (2 * nb + 4) +
           (sizeof(float4) + 3 * sizeof(double) + sizeof(int2) + sizeof(int)) * (size_t)max_N;
}
// Lists for up to max_N spheres at base (256-byte aligned); count, start and posf begin on 16-byte boundaries.
inline CellLists cell_lists(void *base, int64_t max_N)
{
    const size_t nb = (size_t)cell_grid(max_N) * cell_grid(max_N);
    CellLists L;
    L.hdr = (CellHeader *)base;
    L.count = (int *)(L.hdr + 1);
    L.start = L.count + nb;
    L.posf = (float4 *)(L.start + nb + 4);
    L.posd = (double *)(L.posf + max_N);
    L.cellof = (int2 *)(L.posd + 3 * max_N);
    L.any = (int *)(L.cellof + max_N);
    return L;
}

// One suspension of a batch in the symmetric pass: its first sphere in the packed layout, its size and
// its first tile in the batch's tile numbering.
struct SymInst {
    long long off;
    int N;
    int tile0;
};

// Symmetric pass over a batch of suspensions (float32): schedule and scratch, built by
// batch_sym_plan and owned by the batch context.
struct BatchSymPlan {
    int *index = nullptr;         // device: CTA table, segment table, row_seg, col_start, tile_inst
    size_t index_cap = 0;         // ints
    SymInst *sinst = nullptr;     // device, one per suspension
    int sinst_cap = 0;
    double *tgt = nullptr;        // segment partials, 3 x 128 doubles each
    size_t tgt_cap = 0;           // bytes
    float *srcp = nullptr;        // column partials, 3 x 128 floats each
    size_t src_cap = 0;           // bytes
    int ncta = 0, nseg = 0, ntiles = 0, seg_off = 0, row_off = 0, col_off = 0, inst_off = 0;
    bool valid = false;
    std::vector<int64_t> sizes;   // the suspension sizes the plan was built for
    int seg_tiles = 0;            // ... and the run length of its row cut
    int tt_minb = 5;              // resident CTAs per SM of the translation-translation kernel (4 or 5)
};

// A schedule of the symmetric pass on the device (sym_schedule_range): the CTA table and segment table
// (4 ints each), row_seg, col_start and col_rows at the given offsets of `index`, for share `part` of
// `nparts` equal shares of the triangle of N spheres.
struct SymSched {
    int *index = nullptr;
    int N = -1, part = 0, nparts = 1;
    int ncta = 0, nseg = 0, seg_off = 0, row_off = 0, col_off = 0, rows_off = 0;
};

// Scratch owned by a context.
struct Workspace {
    void *slab = nullptr;         // the allocation of the arrays down to vec_g, of sym64, of small blocks64 and of the
                                  // SideSpace
    void *src = nullptr;          // packed sources, max_N records (SrcF64 size)
    void *partial = nullptr;      // pair-kernel partial sums
    size_t partial_bytes = 0;
    double *V = nullptr;          // Lanczos basis, (max_iter + 1) x 3 max_N
    double *w = nullptr;          // Lanczos work vector, 3 max_N
    double *vf = nullptr;         // load of the next Lanczos product (the Krylov vector, scaled by the preconditioner)
    double *red = nullptr;        // reduction partials
    size_t red_elems = 0;
    double *lz = nullptr;         // Lanczos small state (alpha, beta, y, y_prev, coefficients, status)
    double *pos_a = nullptr;      // displaced positions (RFD), 3 max_N
    double *pos_b = nullptr;
    double *pos_w = nullptr;      // positions folded into the unit cell (pseudo-periodic mode), 3 max_N
    void *cells = nullptr;        // cell lists of the force pass (cell_lists_bytes)
    double *selfc = nullptr;      // self coefficients of the packed positions (SelfCoefs), 4 max_N
    double *vec_a = nullptr;      // 3 max_N scratch vectors for the AB step
    double *vec_b = nullptr;
    double *vec_c = nullptr;
    double *vec_d = nullptr;
    double *vec_e = nullptr;
    double *vec_f = nullptr;
    double *vec_g = nullptr;
    double *host_status = nullptr; // pinned host copy of the Lanczos status word
    double *pc = nullptr;          // block-diagonal preconditioner D^{-1/2} (3 max_N), rpb_set_preconditioner
    // symmetric translation-translation pass (float32 contexts): schedules, row and column partials
    int *sym_index = nullptr;      // room for two schedules of sym_index_ints each (sym.index, sym_part.index)
    size_t sym_index_ints = 0;
    double *sym_tgt = nullptr;
    size_t sym_tgt_bytes = 0;
    float *sym_src = nullptr;
    size_t sym_src_bytes = 0;
    void *src2 = nullptr;          // second right-hand side of the two-RHS symmetric pass (float4 per sphere)
    double *sym64 = nullptr;       // float64 contexts: row and column partials of the symmetric pass (pair64.cu)
    int64_t sym64_N = 0;           // ... sized for this many spheres
    double *blocks64 = nullptr;    // the pairs' translation blocks at a Lanczos solve's positions (blocks64_prepare)
    int64_t blocks64_N = 0;                // ... sized for this many spheres
    int64_t blocks64_refused = INT64_MAX;  // ... no room for this many or more
    bool blocks64_small = false;           // ... part of the slab
    SymSched sym;       // the whole triangle
    SymSched sym_part;  // one share of it (rpb_mobility_apply_part)
};

// What one product writes besides its result, for products on the side stream (a step's drift beside its Lanczos
// iterations, a drift's second product beside its first): the fields of Workspace of the same names, for up to
// max_N spheres.
struct SideSpace {
    int64_t max_N = 0, sym64_N = 0;
    void *src = nullptr, *partial = nullptr;
    size_t partial_bytes = 0, sym_tgt_bytes = 0, sym_src_bytes = 0;
    double *selfc = nullptr, *w = nullptr, *pos_w = nullptr, *sym64 = nullptr, *sym_tgt = nullptr;
    float *sym_src = nullptr;
};

// Programmatic dependent launch along the chain of a Lanczos iteration, product -> reduce -> cluster kernel: a kernel
// launched by launch_after() may start while the one before it runs, once every CTA of that one has passed
// after_may_start(), and waits in wait_for_before() until it is complete and its writes are visible, before it
// reads or writes any global memory.  What the one before writes is no `const __restrict__` parameter of such a
// kernel: that would promise that nothing changes it while the kernel runs, and allow its loads ahead of the wait.
// Every kernel launched this way waits, so completion is transitive along the chain; started otherwise,
// wait_for_before() returns at once.  Products of a solve after the first, of at most kAfterMaxN spheres, the range of
// the cluster kernel: there a kernel's launch is a good part of its time, and waiting CTAs take no room that running ones
// need.  A float32 step of 4096 spheres 747 -> 698 us, a float64 one of 256 358 -> 316, twenty replayed ones 5.18 ->
// 4.85 ms, a solve of 3001 spheres 436 -> 403 us.  Host-driven solves without / with, float64: 300 spheres 330 / 311 us,
// 800 472 / 450, 2000 1175 / 1153, 4096 3554 / 3535; float32: 300 390 / 368, 4096 606 / 589.  The line is no crossing:
// with the reduce kernels of larger solves launched early too, float32 solves of 4500 and 8192 spheres take 778 and
// 1251 us instead of 800 and 1270, float64 ones of 4500 4331 instead of 4354.
constexpr int64_t kAfterMaxN = 4096;
#ifdef __CUDACC__
__device__ __forceinline__ void after_may_start()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_before()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... P, typename... A>
inline cudaError_t launch_after(bool early, void (*kernel)(P...), dim3 grid, unsigned threads, unsigned cluster, cudaStream_t st,
                                A... args)
{
    if (!early && !cluster) {  // half the host time of the call below
        kernel<<<grid, threads, 0, st>>>(static_cast<P>(args)...);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    if (early) {
        at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster) {
        at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        at[cfg.numAttrs].val.clusterDim.x = cluster;
        at[cfg.numAttrs].val.clusterDim.y = at[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    cfg.attrs = at;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#endif

// Threads per block of an elementwise kernel over n items: single warps while they leave room on the SMs (a
// float64 warp instruction takes 64 cycles of its scheduler, so a small vector is spread over all of
// them), 256 beyond.
inline int elem_threads(int64_t n, int num_sms)
{
    return n <= 32 * 8 * (int64_t)num_sms ? 32 : 256;
}

constexpr int kRunMaxIter = 64;  // = kMaxIter of the Lanczos state

// Device state of a graph-replayed run (rpb_run): the step index the noise is drawn with, whether the
// coming step is a first (Euler-Maruyama) step, the Lanczos dimension m of the latest step and the
// iteration it is at, and counters of the steps that did not converge and of the iterations run in the
// loop node (all but each step's first).
struct RunState {
    unsigned int step;
    int first;
    int m;
    int left;  // steps left in the run
    int k;
    int pad;
    unsigned long long unconv;
    unsigned long long loops;
};
struct RunCtx;  // run.cu

// Capture of the Lanczos iterations into a CUDA graph (rpb_run): the iterations after the first are the
// body of a loop (WHILE) node captured on `body`; the last kernel of an iteration sets its condition on
// the device from the stopping test, and records m and the iteration in state.
struct LzGraph {
    cudaStream_t body = nullptr;
    RunState *state = nullptr;
    int body_launches = 0;  // kernels captured into the loop's body
};

}  // namespace rpb

struct rpb_ctx {
    rpb_params p;
    int64_t max_N;
    int max_iter;
    cudaStream_t stream;
    int device;
    int num_sms;
    int fp32_variant;  // float32 pair kernel: 1 = packed float32x2 (default), 0 = scalar; env RPB_FP32_PAIR
    int sym_enabled;   // float32 translation-translation products use the symmetric pass; env RPB_FP32_SYM=0 off
    int sym_fused;     // products with torques also use the symmetric pass; env RPB_FP32_SYM_FUSED=0 off
    int sym_rhs2;      // a step's fused product and first Lanczos product share one pass; env RPB_FP32_SYM_RHS2=0 off
    double Lx = 0.0, Ly = 0.0;  // pseudo-periodic periods (0: unbounded in-plane), rpb_set_periodic
    int precond = 0;            // Lanczos preconditioner (RPB_PRECOND_*), rpb_set_preconditioner
    int f32_slots[2] = {0, 0};  // resident CTAs of the float32 one-way pair kernels (tt, with torques)
    rpb::Workspace ws;
    rpb::RunCtx *run = nullptr; // streams and device state of graph-replayed runs (rpb_run), made on first use
    rpb_product_hook hook = nullptr;  // products delegated to the caller (rpb_set_product_hook)
    void *hook_user = nullptr;
    int in_hook = 0;                  // inside the hook: products are computed here
    int gs_cluster = 8;               // blocks of the Lanczos cluster kernel at most (lanczos_setup)
    rpb::SideSpace side;              // scratch, stream and events of a step's drift beside its Lanczos solve
    cudaStream_t side_stream = nullptr;
    bool in_side = false;             // a SideScope lives
    cudaEvent_t side_fork = nullptr, side_join = nullptr;
    cudaEvent_t lz_ev = nullptr;      // host-driven Lanczos: an iteration's status has been written
    const double *stop = nullptr;     // set while a Lanczos solve enqueues a product it may discard: the stop word
};

namespace rpb {

// Error reporting (thread-local message).
void set_error(const char *fmt, ...);
// Count kernel launches enqueued by the library (reported by rpb_launch_count).
void count_launches(int n);
int cuda_fail(cudaError_t e, const char *what);

// While it lives, the context's products use the side scratch and its stream (host state only: the kernels
// enqueued meanwhile keep the pointers they were given).
struct SideScope {
    rpb_ctx *c;
    cudaStream_t stream;
    explicit SideScope(rpb_ctx *ctx) : c(ctx), stream(ctx->stream)
    {
        swap();
        c->stream = c->side_stream;
        c->in_side = true;
    }
    ~SideScope()
    {
        swap();
        c->stream = stream;
        c->in_side = false;
    }
    void swap()
    {
        Workspace &w = c->ws;
        SideSpace &q = c->side;
        std::swap(w.src, q.src);
        std::swap(w.partial, q.partial);
        std::swap(w.partial_bytes, q.partial_bytes);
        std::swap(w.selfc, q.selfc);
        std::swap(w.w, q.w);
        std::swap(w.pos_w, q.pos_w);
        std::swap(w.sym64, q.sym64);
        std::swap(w.sym64_N, q.sym64_N);
        std::swap(w.sym_tgt, q.sym_tgt);
        std::swap(w.sym_tgt_bytes, q.sym_tgt_bytes);
        std::swap(w.sym_src, q.sym_src);
        std::swap(w.sym_src_bytes, q.sym_src_bytes);
    }
};

int side_fork(rpb_ctx *ctx, int64_t N);
int side_join(rpb_ctx *ctx);

// Pair product: U = M_tt F + M_tr T with the context's precision.  F or T may be null.
// All pointers device, SoA float64.  Enqueued on ctx->stream.  mode (a Lanczos solve makes many products at the
// same positions): kPlain; kKeep, a first one that leaves what the others can use (the packed positions, and
// in float64 the pairs' blocks, pair64.cu); kAgain, another one at those positions, with no product of the
// context in between: the packed sources hold s F already (F is still read for the self terms; T null).
enum ProductMode { kPlain, kKeep, kAgain };
bool product_stops(const rpb_ctx *ctx, int64_t N);
int mobility_apply_impl(rpb_ctx *ctx, int64_t N, const double *pos, const double *F, const double *T,
                        double *U, ProductMode mode = kPlain);
// Rows t0 .. t1 - 1 of the product (component stride ldu, ldu < 0: t1 - t0), one-way kernels over a
// target range.
int mobility_rows_impl(rpb_ctx *ctx, int64_t N, const double *pos, const double *F, const double *T, int64_t t0,
                       int64_t t1, double *U_rows, int64_t ldu = -1);
// Share `part` of `nparts` of the product (rpb_mobility_apply_part); never goes through the product hook.
int mobility_part_impl(rpb_ctx *ctx, int64_t N, const double *pos, const double *F, const double *T, int part,
                       int nparts, double *U);
// The float64 product with each unordered pair evaluated once (pair64.cu): whether it can be taken (a
// float64 context with its scratch, forces given, no periodic images), and the product.
bool mobility_sym64_ok(const rpb_ctx *ctx, const double *F);
int mobility_sym64(rpb_ctx *ctx, int N, const double *pos, const double *F, const double *T, double *U, ProductMode mode);
void blocks64_prepare(rpb_ctx *ctx, int64_t N);
// Whether mobility_apply2_impl can take this product (float32 symmetric pass with two right-hand sides).
bool mobility_apply2_ok(const rpb_ctx *ctx, int64_t N);
// U = M_tt F + M_tr T and U2 = M_tt P in one symmetric pass (F, T, P non-null).
int mobility_apply2_impl(rpb_ctx *ctx, int64_t N, const double *pos, const double *F, const double *T,
                         const double *P, double *U, double *U2);

// Packed source records from float64 SoA inputs (pair.cu), and the spheres' self coefficients where
// sc.s is given; also used by the batched path.
struct SelfCoefs;
__global__ void pack_f32_kernel(const double *__restrict__ pos, const double *__restrict__ F,
                                const double *__restrict__ T, int N, double a, int wall, SrcF32 *__restrict__ out,
                                SelfCoefs sc);
__global__ void pack_f64_kernel(const double *__restrict__ pos, const double *__restrict__ F,
                                const double *__restrict__ T, int N, double a, int wall, SrcF64 *__restrict__ out,
                                SelfCoefs sc);

// Number of column splits and chunk length the pair kernel uses for N targets.
// slots: resident CTAs of the float32 kernel over the GPU (0: unknown, fixed rule).
void pair_grid(int64_t N, int num_sms, int precision, int slots, int *splits, int64_t *chunk);
int pair_occupancy(rpb_ctx *ctx);
size_t pair_partial_bytes(int64_t max_N, int num_sms);
size_t sym_src_part_bytes(int64_t max_N);
size_t sym_tgt_part_bytes(int64_t max_N, int num_sms);
size_t sym_index_ints(int64_t max_N, int num_sms);

int forces_impl(rpb_ctx *ctx, int64_t N, const double *pos, const rpb_force_params *fp, double *F);

// Build (or keep, when the sizes are unchanged) the batched symmetric plan for B suspensions of sizes N
// packed one after another; grows the plan's scratch (not inside a stream capture).  Returns RPB_OK,
// or an error; *ok is false when the plan would need more than the scratch limit (the caller then uses
// the one-way kernels).
// seg_tiles: the run length of every suspension's row cut (the results depend on it, not on the
// companions).
int batch_sym_plan(BatchSymPlan &pl, int B, const int64_t *N, cudaStream_t st, bool *ok, int seg_tiles);
void batch_sym_free(BatchSymPlan &pl);
// U_b = M_tt F_b (+ M_tr T_b) for every suspension of the plan, from packed float32 sources; active
// masks suspensions (null: all).
int batch_sym_apply(const BatchSymPlan &pl, cudaStream_t st, const SrcF32 *src, int64_t total, const double *F,
                    const double *T, double *U, const int *active, double a, const SelfCoefs &sc);
// d_step (optional): a device word to read the step index from instead of `step` (graph replays).
int philox_impl(rpb_ctx *ctx, int64_t N, uint64_t seed, uint32_t step, uint32_t stream_id, uint32_t instance,
                double *out, const unsigned int *d_step = nullptr);
// Open a conditional node after the work captured so far on `st` and start capturing its body on
// `body`; an IF node runs its body when `h` was set non-zero, a WHILE node as long as it is.
int graph_begin_cond(cudaStream_t st, cudaStream_t body, cudaGraphConditionalHandle h,
                     cudaGraphConditionalNodeType type);
// Adds a WHILE node (its handle created with the default value 1) after the capture dependencies of
// st and begins capturing its body on `body`; the body ends with graph_loop_tail_kernel.
int graph_begin_loop(cudaStream_t st, cudaStream_t body, cudaGraphConditionalHandle *h);
// *left = n (before the loop's graph is launched)
__global__ void graph_loop_init_kernel(int *left, int n);
// End of one pass of a loop body: --*left, and the loop runs again while *left > 0.
__global__ void graph_loop_tail_kernel(int *left, cudaGraphConditionalHandle h);
// Host-side preparation a product at this N needs (the symmetric pass's schedule), done before a
// stream capture so that the captured products find it in place.
int pair_prepare(rpb_ctx *ctx, int64_t N);
// packed: the positions are packed already (a product at these positions was the last one)
int lanczos_impl(rpb_ctx *ctx, int64_t N, const double *pos, const double *W, double *g, double tol, int max_iter,
                 bool packed, int *iters_out, double *err_out, int *converged_out, LzGraph *gr = nullptr);
// The two halves of lanczos_impl: v_0 = W/|W| into ws.V and, times the preconditioner, into ws.vf (packed:
// into the packed sources too); then the iterations.  first_done: the product M vf is already in ws.w.
int lanczos_init(rpb_ctx *ctx, int64_t N, const double *W, bool packed, LzGraph *gr);
// With ctx->precond set: P = D^{-1/2} at these positions into ws.pc (D: diagonal of the self blocks),
// so that the iteration runs on P M P and returns g = D^{1/2} y.
int lanczos_precond_prepare(rpb_ctx *ctx, int64_t N, const double *pos);
// gr: inside a stream capture, the iterations after the first in a loop node (see LzGraph); the host
// outputs are then not written (the noise W of a step is never 0).
int lanczos_run(rpb_ctx *ctx, int64_t N, const double *pos, double *g, double tol, int max_iter, bool first_done,
                bool packed, int *iters_out, double *err_out, int *converged_out, LzGraph *gr = nullptr);
int lanczos_setup(rpb_ctx *ctx);
int rfd_impl(rpb_ctx *ctx, int64_t N, const double *pos, const double *Wt, double delta, double *drift,
             int one_sided = 0);
// d_first (optional): a device word that, when non-zero, makes the update a first step (graph replays).
int ab_update_impl(rpb_ctx *ctx, int64_t N, double *pos, double *U_prev, const double *Un, const double *g,
                   const double *drift, double dt, double noise_scale, int first, const int *d_first = nullptr);

// Arguments of a time step (rpb_step, rpb_run), and the step itself (api.cu; see there).
int check_step_args(rpb_ctx *ctx, int64_t N, const double *pos, const double *U_prev, int64_t step, double dt,
                    double delta, int max_iter, const rpb_force_params *fp, const rpb_step_options *opts);
int step_impl(rpb_ctx *ctx, int64_t N, double *pos, double *U_prev, uint32_t step, uint64_t seed, double dt,
              double delta, double tol, int max_iter, const rpb_force_params *fp, int scheme, int rfd,
              rpb_step_stats *stats, LzGraph *gr);
// Streams and device state of graph-replayed runs (run.cu), released by rpb_destroy.
void run_free(rpb_ctx *ctx);

// Copy the nodes and weights of the square root (sqrt_nodes.h: all shifts, then all weights) to the
// device; the copies are complete or staged when it returns.
int upload_sqrt_nodes(double *nodes, cudaStream_t st);
// Sizes of the Lanczos small-state block (doubles) for max_iter; the square root's nodes follow the
// state (at LzLayout::total).
size_t lanczos_state_elems(int max_iter);
int lanczos_upload(double *lz, int max_iter, cudaStream_t st);  // the nodes into a state block
size_t lanczos_red_elems(int64_t max_N, int max_iter);

}  // namespace rpb
