// sp_split.h -- how the launchers split a grid into runs of rows or planes: plain host functions
// of sizes and occupancy, taken anew by every launch.
#pragma once

#include <algorithm>

namespace sp {

// smallest divisor of n that is at least lo; 0 if there is none
inline long long divisor_from(long long n, long long lo) {
    long long d = lo;
    for (; d <= n / d; ++d)
        if (n % d == 0) return d;
    if (d > n) return 0;
    for (long long k = n / d; k >= 1; --k)
        if (n % k == 0) return n / k;
    return 0;
}

// The run length p in [ceil(total / (n_sm occ)), limit] of the lowest cost(q, p), the shorter one of
// two that differ by under 0.1 percent.  q is the number of CTAs, ceil(total / p) in all, on the
// fullest SM; runs for which it is 1 already only get longer with p.  The cost rises with p
// while q stays, except that it may drop at a divisor of `period` (0: none).  So only the first p of
// each q (at most occ of them) and the divisors are looked at: a search over every p took 11 us
// per launch at 4096^2 and 700 us at 32768^2, more than the launch itself where none is queued
// before it; now 0.1 to 0.6 us.
template <typename Cost>
inline long long best_run(long long total, int occ, int n_sm, long long limit, long long period, const Cost &cost) {
    const long long wave = (long long)n_sm * std::max(occ, 1), p0 = (total + wave - 1) / wave;
    auto fullest = [&](long long p) { return ((total + p - 1) / p + n_sm - 1) / n_sm; };
    long long best = p0;
    double best_cost = cost(fullest(p0), p0);
    auto weigh = [&](long long q, long long p) {
        const double c = cost(q, p);
        if (c < best_cost * 0.999) {
            best = p;
            best_cost = c;
        }
    };
    for (long long p = p0; p <= limit;) {
        const long long q = fullest(p);
        weigh(q, p);
        if (q == 1) break;
        const long long next = std::max(p + 1, (total + (q - 1) * n_sm - 1) / ((q - 1) * n_sm));
        if (period > 0)
            for (long long d = divisor_from(period, p + 1); d > 0 && d < next && d <= limit; d = divisor_from(period, d + 1))
                weigh(q, d);
        p = next;
    }
    return best;
}

// Rows per CTA of the 2D warp-strip kernel, whose CTAs own equal runs of the flattened
// (strip group, row) space: p rows cost p + halo, q CTAs of `load` (their share of 8
// warps) on the fullest SM take about q load + latency of them (see planes_per_cta).
// Runs of at least 32 rows left most SMs idle on small grids: 444 x 568 Cahn-Hilliard 9.2
// us per step, 3.0 now; 1504 x 1000 4th order 13.2 -> 6.2 (runs of 8 rows; of 4: 7.5).
inline long long rows_per_cta(long long total, int halo, double load, double latency, int occ, int n_sm) {
    const long long wave = (long long)n_sm * std::max(occ, 1), p0 = (total + wave - 1) / wave;
    return best_run(total, occ, n_sm, std::min(total, 8 * p0 + 32), 0,
                    [=](long long q, long long p) { return (q * load + latency) * (p + halo); });
}

// Warps per CTA of the 2D warp-strip kernels, whose CTAs take that many adjacent strips: the
// most of at least max / 2 that leave the fewest warps without a strip (13 strips: two CTAs of
// 7 warps, not of 8).
inline int warps_per_cta(int strips, int max) {
    if (strips <= max) return strips;
    int best = max;
    for (int w = max - 1; 2 * w >= max; --w)
        if ((strips + w - 1) / w * w < (strips + best - 1) / best * best) best = w;
    return best;
}

// Rows per CTA (one warp on grids of few strips, whose last CTA would be half empty, else
// two on adjacent strips): p rows cost p + halo iterations, each the issue time of the warps that
// share a scheduler of the fullest SM, at least that of five (a warp's own chain of K steps).
inline long long warptb_rows(long long total, int halo, int wpc, int occ, int n_sm) {
    const long long wave = (long long)n_sm * occ, p0 = (total + wave - 1) / wave;
    return best_run(total, occ, n_sm, std::min(total, 8 * p0 + 32), 0,
                    [=](long long q, long long p) { return std::max(5.0, q * wpc / 4.0) * (p + halo); });
}

// Planes per CTA of a persistent 3D kernel whose CTAs own equal contiguous runs of
// the flattened (tile, z) space; at most one resident wave (n_sm x occ CTAs).  A run
// of p planes costs p + halo planes, halo standing for the planes it only warms its
// rings with, once more where runs cross from one tile into the next.  With q CTAs on
// the fullest SM the kernel takes about q + 1 runs: the FP64 pipe is shared, but the
// barriers and loads of one run are not hidden.  Grids that fill the wave with long runs keep p =
// total / wave; small ones are spread over all SMs down to single planes (64^3 FP64
// Gray-Scott 7-point: 417 us per step with runs of at least 32 planes, 17 us now;
// 32^3 Cahn-Hilliard 179 -> 11.5 us; 129 x 32 x 208 Cahn-Hilliard 189 -> 47 us, where
// the balance of q against p decides between runs of 3 (53 us) and 4 planes).
inline long long planes_per_cta(long long tiles, int nz, double halo, int occ, int n_sm) {
    const long long total = tiles * nz, wave = (long long)n_sm * std::max(occ, 1);
    const long long p0 = (total + wave - 1) / wave;
    return best_run(total, occ, n_sm, std::min(total, 4 * p0 + 8), nz,
                    [=](long long q, long long p) { return (q + 1.0) * (p + (nz % p ? 2 : 1) * halo); });
}

// Number of equal z segments for a lockstep schedule of `tiles` x segments work
// items over `wave` resident CTAs: minimises rounds x (planes per segment +
// halo planes), the time of the slowest CTA.
inline int lockstep_segments(long long tiles, int nz, int halo, long long wave) {
    int best = 1;
    double best_cost = 0;
    for (int sgs = 1; sgs <= std::min(nz, 64); ++sgs) {
        const long long rounds = (tiles * sgs + wave - 1) / wave;
        const double cost = (double)rounds * ((double)nz / sgs + halo);
        if (sgs == 1 || cost < best_cost * 0.999) {
            best = sgs;
            best_cost = cost;
        }
    }
    return best;
}

}  // namespace sp
