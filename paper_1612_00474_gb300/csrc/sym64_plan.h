// sym64_plan.h -- work split of the float64 symmetric pass (host and device logic without CUDA calls, so
// that the tests can compile and check it on the CPU).
//
// The spheres are in tiles of 32 and the work is the upper triangle of (target tile b, source tile
// t >= b) units; row b is cut into runs of at most L tiles, one CTA each, numbered row by row.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define RPB_HD __host__ __device__
#else
#define RPB_HD
#endif

namespace rpb {

constexpr int kTile64 = 32;

struct Sym64Plan {
    int nb;      // tiles
    int L;       // tiles of a run
    int qs;      // CTAs that share a run, each a part of the 32 rotations of a unit
    int64_t runs;
};

// Runs of the rows with m = 1 .. n source tiles: sum of ceil(m / L).
RPB_HD inline int64_t sym64_runs(int64_t n, int L)
{
    const int64_t q = n / L, r = n - q * L;
    return (int64_t)L * q * (q + 1) / 2 + r * (q + 1);
}

// First run of row b.
RPB_HD inline int64_t sym64_row_run(const Sym64Plan &p, int b)
{
    return p.runs - sym64_runs(p.nb - b, p.L);
}

// Row of a run (the largest b whose first run is not after it).
RPB_HD inline int sym64_row_of(const Sym64Plan &p, int64_t run)
{
    int lo = 0, hi = p.nb - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (sym64_row_run(p, mid) <= run)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Column partial of unit (b, t), t > b, part s of qs (units of 96 doubles).
RPB_HD inline int64_t sym64_col_slot(const Sym64Plan &p, int b, int t, int s)
{
    return ((int64_t)t * (t - 1) / 2 + b) * p.qs + s;
}

// A unit is 32 rotations (each lane of a warp against every source of the tile), eight for each of a
// CTA's four warps.  Up to 60 x SMs runs of one tile, longer ones beyond: their partial sums then stay
// below one per unit.  With fewer units than a wave holds, qs CTAs share a unit: a warp's chain of float64
// instructions is what a small product waits for.  The cost of a wave is its rotations per warp plus what a
// CTA spends besides, staging and adding its partials, about 0.7 of one.
inline Sym64Plan sym64_plan(int64_t N, int num_sms)
{
    Sym64Plan p;
    p.nb = (int)((N + kTile64 - 1) / kTile64);
    const int64_t units = (int64_t)p.nb * (p.nb + 1) / 2, cap = 60 * (int64_t)num_sms;
    p.L = (int)((units + cap - 1) / cap);
    p.qs = 1;
    if (units < 8 * (int64_t)num_sms) {
        double best = 0.0;
        for (int q = 1; q <= 8; q *= 2) {
            const double c = (double)((units * q + num_sms - 1) / num_sms) * (8.0 / q + 0.7);
            if (q == 1 || c < best) {
                best = c;
                p.qs = q;
            }
        }
    }
    p.runs = sym64_runs(p.nb, p.L);
    return p;
}

// Scratch (doubles) that the plans of every N <= max_N need: row partials, then column partials.
// A plan with qs > 1 has fewer than 8 x 8 x SMs parts.
inline int64_t sym64_tgt_elems(int64_t max_N, int num_sms)
{
    const int64_t nb = (max_N + kTile64 - 1) / kTile64;
    const int64_t runs = 60 * (int64_t)num_sms + nb, parts = nb * (nb + 1) / 2 * 8;
    const int64_t small = parts < 64 * (int64_t)num_sms ? parts : 64 * (int64_t)num_sms;
    return 96 * (runs > small ? runs : small);
}
inline int64_t sym64_src_elems(int64_t max_N, int num_sms)
{
    const int64_t nb = (max_N + kTile64 - 1) / kTile64;
    const int64_t units = nb * (nb - 1) / 2, parts = units * 8;
    const int64_t small = parts < 64 * (int64_t)num_sms ? parts : 64 * (int64_t)num_sms;
    return 96 * (units > small ? units : small);
}

// A Lanczos solve in float64 keeps the blocks of its pairs (pair64.cu): 64 bytes for each pair of lanes of each unit.
inline int64_t blocks64_bytes(int64_t N)
{
    const int64_t nb = (N + kTile64 - 1) / kTile64;
    return nb * (nb + 1) / 2 * 32 * 8 * 32 * (int64_t)sizeof(double);
}

// Contexts whose blocks take no more than this (1,400 spheres) hold them from the start, as part of their scratch: a
// first solve of 300 spheres takes 345 us, and the allocation would be 100 of its own.
constexpr int64_t kBlocks64SmallBytes = (int64_t)64 << 20;
// Spheres that a solve of N makes room for when there is room for `held` of at most max_N: N at first, then with some
// to spare, so that a slowly growing suspension does not ask each time; 0: none, evaluate the pairs.  Up to 8 GB
// (16,000 spheres), and an eighth of the device stays free for others.
constexpr int64_t kBlocks64MaxBytes = (int64_t)8 << 30;
inline int64_t blocks64_room(int64_t N, int64_t held, int64_t max_N, int64_t free_bytes, int64_t total_bytes)
{
    const int64_t more = held + held / 4 < max_N ? held + held / 4 : max_N;
    const int64_t left = free_bytes + (held > 0 ? blocks64_bytes(held) : 0) - total_bytes / 8;
    const int64_t most = left < kBlocks64MaxBytes ? left : kBlocks64MaxBytes;
    if (more > N && blocks64_bytes(more) <= most) return more;
    return blocks64_bytes(N) <= most ? N : 0;
}

}  // namespace rpb
