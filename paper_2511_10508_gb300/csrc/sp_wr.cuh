// sp_wr.cuh -- launch of the 3D warp-row kernel (step3d_wr_kernel) and the choice of its tile.
#pragma once

#include <algorithm>

#include "sp_internal.h"
#include "sp_step.cuh"

namespace sp {

// resident CTAs per SM of one instantiation
template <int MODEL, int ST, typename T, int TY, int LN, bool AL> int wr_occupancy() {
    typedef Step3dWrShape<MODEL, ST, T, TY, LN> Sh;
    static const int occ = [] {
        auto kern = step3d_wr_kernel<MODEL, ST, T, TY, LN, AL>;
        const size_t smem = Sh::smem_bytes + (AL ? 0 : Sh::stage_bytes);
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int o = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, Sh::NT, smem);
        return std::max(o, 1);
    }();
    return occ;
}

// `segs` equal z segments per tile, (segment, tile) items in lockstep
template <int MODEL, int ST, typename T, int TY, int LN, bool AL>
cudaError_t launch_wr(const StepArgs &a, cudaStream_t s, int n_sm, int segs) {
    typedef Step3dWrShape<MODEL, ST, T, TY, LN> Sh;
    const int occ = wr_occupancy<MODEL, ST, T, TY, LN, AL>();
    const int tx = (a.nx + Sh::TX - 1) / Sh::TX, ty = (a.ny + TY - 1) / TY;
    const long long items = (long long)tx * ty * segs, wave = (long long)n_sm * occ;
    return launch_pdl(step3d_wr_kernel<MODEL, ST, T, TY, LN, AL>, dim3((unsigned)std::min(items, wave)), dim3(Sh::NT),
                      Sh::smem_bytes + (AL ? 0 : Sh::stage_bytes), s, a, tx, ty, segs);
}

#ifdef SP_WR_MODEL

// Tiles of the FP32 kernel: TY rows of LN lanes (LN - 2 of them output, 4 cells each).  Rows of
// 32 lanes cover 120 cells, which a 256-wide grid fills to 71 percent of three; rows of 16
// lanes (two per warp) cover 56, and tall tiles of them have less halo in y.  COST: SM time per
// plane of a tile, measured on 512^3 (us per step / tiles; only ratios matter).
template <int TY_, int LN_, int COST_> struct WrTile {
    static constexpr int TY = TY_, LN = LN_, COST = COST_;
};

// The cheapest of the tiles for a grid: rounds x (planes per segment + halo planes) x the time
// of a plane with the SM full, as in lockstep_segments.  Measured, us per step, 32-lane rows
// before and the choice now: Cahn-Hilliard 7-point 256^3 52.8 / 44.0, 384^3 151 / 122, 512^3 340 / 301;
// 27-point 384^3 263 / 179, 512^3 571 / 456; 13-point (plane ring before) 384^3 257 / 245; Allen-Cahn
// 13-point 384^3 172 / 114; Gray-Scott 27-point 384^3 256 / 190, 13-point 287 / 235.
template <int MODEL, int ST, bool AL, typename... Tiles>
cudaError_t choose_wr(const StepArgs &a, cudaStream_t s, int n_sm, double other) {
    // the last choice of this thread, by shape
    struct Last { int nx = 0, ny = 0, nz = 0, n_sm = 0, pick = 0, segs = 1; };
    static thread_local Last last;
    if (last.nx != a.nx || last.ny != a.ny || last.nz != a.nz || last.n_sm != n_sm) {
        double best = other;
        int i = 0;
        last = Last{a.nx, a.ny, a.nz, n_sm, -1, 1};
        auto weigh = [&](auto t) {
            typedef decltype(t) W;
            typedef Step3dWrShape<MODEL, ST, float, W::TY, W::LN> Sh;
            const int occ = wr_occupancy<MODEL, ST, float, W::TY, W::LN, AL>();
            const long long tiles = (long long)((a.nx + Sh::TX - 1) / Sh::TX) * ((a.ny + W::TY - 1) / W::TY);
            const long long wave = (long long)n_sm * occ;
            const int segs = lockstep_segments(tiles, a.nz, 2 * Sh::R, wave);
            const double cost = (double)((tiles * segs + wave - 1) / wave) * ((double)a.nz / segs + 2 * Sh::R) * W::COST * occ;
            if (best < 0 || cost < best) {
                best = cost;
                last.pick = i;
                last.segs = segs;
            }
            ++i;
        };
        (weigh(Tiles{}), ...);
    }
    cudaError_t e = cudaErrorNotSupported;
    int i = 0;
    auto go = [&](auto t) {
        typedef decltype(t) W;
        if (i++ == last.pick) e = launch_wr<MODEL, ST, float, W::TY, W::LN, AL>(a, s, n_sm, last.segs);
    };
    (go(Tiles{}), ...);
    return e;
}

template <int MODEL, int ST, typename... Tiles>
cudaError_t choose_wr_any(const StepArgs &a, cudaStream_t s, int n_sm) {
    const bool al = a.nx % 4 == 0 &&
                    ((uintptr_t)a.in0 | (uintptr_t)a.in1 | (uintptr_t)a.out0 | (uintptr_t)a.out1) % 16 == 0;
    if (!al) return choose_wr<MODEL, ST, false, Tiles...>(a, s, n_sm, -1.0);
    double other = -1.0;
    if constexpr (MODEL == CH && ST == L13X4) {
        // the plane ring (step3d_async_kernel, tiles of 64 x 16), one CTA of 256 threads per SM
        const long long tiles = (long long)((a.nx + 63) / 64) * ((a.ny + 15) / 16);
        const int segs = lockstep_segments(tiles, a.nz, 2 * 4, n_sm);
        other = (double)((tiles * segs + n_sm - 1) / n_sm) * ((double)a.nz / segs + 8) * 2350;
    }
    return choose_wr<MODEL, ST, true, Tiles...>(a, s, n_sm, other);
}

#endif  // SP_WR_MODEL

}  // namespace sp
