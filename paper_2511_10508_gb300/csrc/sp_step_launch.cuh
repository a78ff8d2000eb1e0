// sp_step_launch.cuh -- host-side launch of the step kernels: tile choices per
// storage type and stencil radius, and the grid size.
//
// Grid sizing.  The streaming kernels (strips and warp rows in 2D, plane rings in 3D) are
// persistent: the work is the flattened space of (column strip or xy tile, row or plane)
// pairs, the grid at most one resident wave, and each CTA takes an equal contiguous run of it or
// an equal z segment per tile (sp_split.h).  The tile and box kernels (2D FP64 on small grids, fused
// steps on tiles, 16-bit storage with unaligned rows) take one CTA per tile or box.
#pragma once

#include <algorithm>
#include <type_traits>

#include "sp_internal.h"
#include "sp_step.cuh"
#include "sp_wr.cuh"

namespace sp {

// 3D FP64 tiles: 32 x 16 points, 128 threads.  Against 64 x 32 (27-point: 32 x 32) tiles of
// 256 threads they are as fast or faster on whole tiles (256^3 7-point: Gray-Scott 711 ->
// 708 us per step, Allen-Cahn 362 -> 357, Model C 748 -> 687; 27-point Gray-Scott 1127 ->
// 1096) and waste less at ragged edges (236^3 Gray-Scott 658 -> 610).  Cahn-Hilliard is a little
// faster with large tiles (256^3: two passes 566 against 574 us, the fused ring, whose
// halo mu grows with the tile's edge, 635 against 664): it takes the small tile where
// that covers 3 (fused: 10) percent fewer points.
constexpr int kTX64 = 32, kTY64 = 16, kNT64 = 128;
inline bool small_tile(int nx, int ny, int TX, int TY, double margin) {
    auto area = [&](int tx, int ty) {
        return (double)((nx + tx - 1) / tx) * tx * ((double)((ny + ty - 1) / ty) * ty);
    };
    return area(kTX64, kTY64) < margin * area(TX, TY);
}

constexpr size_t kMaxSmemPerCta = 227 * 1024;  // opt-in maximum of dynamic shared memory per CTA

// Batched persistent 2D kernel (FP64): rows per batch and CTAs per SM.
template <int MODEL> struct Batch2d { static constexpr int NT = 128, RB = (MODEL == CH) ? 8 : (MODEL == AC ? 4 : 2), CPS = 4; };

// The FP64 2D strip kernel with NT threads, RB rows per batch, at most CPS CTAs
// per SM; persistent grid with equal rows per CTA.
template <int MODEL, int ST, typename T, int NT, int RB, int CPS>
cudaError_t launch_strips(const StepArgs &a, cudaStream_t s, int n_sm) {
    typedef Step2dBatchShape<MODEL, ST, T, NT, RB> Sh;
    auto kern = step2d_batch_kernel<MODEL, ST, T, NT, RB>;
    static const int occ = [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
        int o = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, NT, Sh::smem_bytes);
        return o;
    }();
    const int strips = (a.nx + Sh::TW - 1) / Sh::TW;
    const long long total = (long long)strips * a.ny;
    // equal rows per CTA; at least 4*RB rows each so that the ring warm-up stays small
    long long ctas = (long long)n_sm * std::max(1, std::min(occ, CPS));
    ctas = std::max(1LL, std::min(ctas, total / (4 * RB)));
    const long long rows = (total + ctas - 1) / ctas;
    ctas = (total + rows - 1) / rows;
    return launch_pdl(kern, dim3((unsigned)ctas), dim3(NT), Sh::smem_bytes, s, a, strips, rows);
}

// Temporally blocked 2D tile kernel: K steps per launch.  FP32 / BF16 tiles of
// 128 x 16; FP64 (small grids, where the fixed cost of a launch matters) tiles
// of 32 x 14, so that a 256^2 grid spreads over 8 x 19 = 152 CTAs, one per SM.
template <int MODEL, int ST, typename T, int K>
cudaError_t launch_tb(const StepArgs &a, cudaStream_t s) {
    constexpr bool f64 = std::is_same<T, double>::value;
    constexpr int BX = f64 ? 32 : 128, BY = f64 ? 14 : 16, NT = f64 ? 128 : 256;
    typedef Step2dTbShape<MODEL, ST, T, BX, BY, K> Sh;
    auto kern = step2d_tb_kernel<MODEL, ST, T, BX, BY, K, NT>;
    static const bool attr = [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
        return true;
    }();
    (void)attr;
    dim3 grid((a.nx + BX - 1) / BX, (a.ny + BY - 1) / BY);
    return launch_pdl(kern, grid, dim3(NT), Sh::smem_bytes, s, a);
}

// 3D FP32 / BF16 Allen-Cahn, Gray-Scott and Model C with a plane ring per time level: K
// steps per pass (temporal blocking for K = 2) on tiles of 4 (LN - 2) x TY
// outputs; lockstep z segments.  AL: nx a multiple of 4 and 16-byte aligned fields, which K = 2 and
// 16-bit storage need; one step of FP32 takes any row (AL = false).
template <int MODEL, int ST, typename T, int TY, int K, bool AL, int LN = 32>
cudaError_t launch_tbs(const StepArgs &a, cudaStream_t s, int n_sm) {
    typedef Step3dTbsShape<MODEL, ST, T, TY, K, LN> Sh;
    constexpr size_t smem = Sh::smem_bytes + (AL ? 0 : Sh::stage_bytes);
    auto kern = step3d_tbs_kernel<MODEL, ST, T, TY, K, LN, AL>;
    static const int occ = [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int o = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, Sh::NT, smem);
        return o;
    }();
    const int tx = (a.nx + Sh::TX - 1) / Sh::TX, ty = (a.ny + TY - 1) / TY;
    const long long wave = (long long)n_sm * std::max(occ, 1);
    const int segs = lockstep_segments((long long)tx * ty, a.nz, 2 * K * Sh::r, wave);
    const long long items = (long long)tx * ty * segs;
    return launch_pdl(kern, dim3((unsigned)std::min(items, wave)), dim3(Sh::NT), smem, s, a, tx, ty, segs);
}

// Model C, one step: tiles of 120 x 8 (32-lane rows) or 56 x 16 (16-lane rows), whichever covers
// the grid in less time (us per 1000 planes of a tile, 384^3: 7-point 2.5 both, 27-point 4.4 / 4.9,
// 13-point 5.0 / 3.4; 256^3 7-point 64.9 against 55.2 us per step, 360^3 128 / 146).
template <int ST, typename T, bool AL>
cudaError_t launch_mc_rows(const StepArgs &a, cudaStream_t s, int n_sm) {
    constexpr double c32 = ST == L7 ? 0.955 : ST == L27 ? 1.675 : 1.918, c16 = ST == L7 ? 0.935 : ST == L27 ? 1.883 : 1.295;
    const double t32 = c32 * ((a.nx + 119) / 120) * ((a.ny + 7) / 8), t16 = c16 * ((a.nx + 55) / 56) * ((a.ny + 15) / 16);
    if (t16 < t32) return launch_tbs<MC, ST, T, 16, 1, AL, 16>(a, s, n_sm);
    return launch_tbs<MC, ST, T, 8, 1, AL>(a, s, n_sm);
}

// FP64 27-point: z-streaming kernel with per-plane partial sums in registers.
template <int MODEL, typename T>
cudaError_t launch_zreg(const StepArgs &a, cudaStream_t s, int n_sm) {
    constexpr int TX = 32, TY = 32, NT = 256;
    typedef Step3dZregShape<MODEL, TX, TY, NT> Sh;
    auto kern = step3d_zreg_kernel<MODEL, TX, TY, NT>;
    static const int occ = [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
        int o = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, NT, Sh::smem_bytes);
        return o;
    }();
    const int tx = (a.nx + TX - 1) / TX, ty = (a.ny + TY - 1) / TY;
    const long long planes = planes_per_cta((long long)tx * ty, a.nz, 1.0, occ, n_sm);
    return launch_pdl(kern, dim3((unsigned)(((long long)tx * ty * a.nz + planes - 1) / planes)), dim3(NT), Sh::smem_bytes, s, a, tx, ty, planes);
}

// FP64 27-point with shared pair sums: one pass per mode (Cahn-Hilliard: mode 0
// then mode 1 through the mu buffer).
template <int MODE>
cudaError_t launch_planes27_mode(const Planes27Args &a, cudaStream_t s, int n_sm) {
    typedef Planes27Shape<MODE> Sh;
    auto kern = planes27_kernel<MODE>;
    static const int occ = [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
        int o = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, Sh::NT, Sh::smem_bytes);
        return o;
    }();
    const int tx = (a.nx + Sh::TX - 1) / Sh::TX, ty = (a.ny + Sh::TY - 1) / Sh::TY;
    const long long total = (long long)tx * ty * a.nz;
    const long long planes = planes_per_cta((long long)tx * ty, a.nz, 1.0, occ, n_sm);
    return launch_pdl(kern, dim3((unsigned)((total + planes - 1) / planes)), dim3(Sh::NT), Sh::smem_bytes, s, a, tx, planes, total);
}
template <int ST, int MODE, int TY>
cudaError_t launch_ring2pass_tile(const Planes27Args &a, cudaStream_t s, int n_sm) {
    typedef Ring2PassShape<ST, TY> Sh;
    auto kern = ring2pass_kernel<ST, MODE, TY>;
    static const int occ = [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
        int o = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, Sh::NT, Sh::smem_bytes);
        return o;
    }();
    const int tx = (a.nx + Sh::TX - 1) / Sh::TX, ty = (a.ny + Sh::TY - 1) / Sh::TY;
    const long long total = (long long)tx * ty * a.nz;
    const long long planes = planes_per_cta((long long)tx * ty, a.nz, 0.7 * Sh::R, occ, n_sm);
    return launch_pdl(kern, dim3((unsigned)((total + planes - 1) / planes)), dim3(Sh::NT), Sh::smem_bytes, s, a, tx, planes, total);
}
template <int ST, int MODE>
cudaError_t launch_ring2pass_mode(const Planes27Args &a, cudaStream_t s, int n_sm) {
    return small_tile(a.nx, a.ny, 32, 32, 0.97) ? launch_ring2pass_tile<ST, MODE, 16>(a, s, n_sm)
                                          : launch_ring2pass_tile<ST, MODE, 32>(a, s, n_sm);
}

// 3D FP64, accessor-based plane ring.
template <int MODEL, int ST, int TX, int TY, int NT>
cudaError_t launch_step3d_tile(const StepArgs &a, cudaStream_t s, int n_sm) {
    typedef Step3dShape<MODEL, ST, double, TX, TY, NT> Sh;
    auto kern = step3d_kernel<MODEL, ST, double, TX, TY, NT>;
    static const int occ = [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
        int o = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, NT, Sh::smem_bytes);
        return o;
    }();
    const int tx = (a.nx + TX - 1) / TX, ty = (a.ny + TY - 1) / TY;
    const long long planes = planes_per_cta((long long)tx * ty, a.nz, 0.7 * Sh::RIN, occ, n_sm);
    return launch_pdl(kern, dim3((unsigned)(((long long)tx * ty * a.nz + planes - 1) / planes)), dim3(NT), Sh::smem_bytes, s, a, tx, ty, planes);
}

// FP32 / BF16 2D: one warp per column strip, up to 8 adjacent strips per CTA,
// persistent equal shares of (strip group, row).
template <int MODEL, int ST, typename T, bool AL>
cudaError_t launch_warp2d(const StepArgs &a, cudaStream_t s, int n_sm) {
    typedef Step2dWarpShape<MODEL, ST, T> WS;
    constexpr int NT = 256;
    auto kern = step2d_warp_kernel<MODEL, ST, T, NT, AL>;
    static const auto occ = warp_occupancy<NT / 32>(kern, WS::warp_smem(AL));
    const int strips = (a.nx + WS::OUT_COLS - 1) / WS::OUT_COLS;
    const int wpc = warps_per_cta(strips, NT / 32), groups = (strips + wpc - 1) / wpc;
    const size_t smem = WS::warp_smem(AL) * wpc;
    const long long total = (long long)groups * a.ny;
    const long long rows = rows_per_cta(total, 2 * WS::RIN, wpc / 8.0, AL ? 1.0 : 4.0, occ[wpc], n_sm);
    const long long ctas = (total + rows - 1) / rows;
    return launch_pdl(kern, dim3((unsigned)ctas), dim3(32 * wpc), smem, s, a, strips, groups, rows);
}

template <int MODEL, int ST, typename T>
cudaError_t launch_step_t(const StepArgs &a, cudaStream_t s, int n_sm, int k) {
    if constexpr (StencilInfo<ST>::dims == 2) {
        if constexpr (sizeof(T) == 4) {
            if (k > 1) {
                const cudaError_t e = launch_w2d(MODEL, ST, a, s, n_sm, k);
                if (e != cudaErrorNotSupported) return e;
            }
        }
        if (k == 4) return launch_tb<MODEL, ST, T, 4>(a, s);
        if (k == 2) return launch_tb<MODEL, ST, T, 2>(a, s);
    } else if (k != 1) {
        // two steps per pass: 16-byte loads and stores of every row, no other kernel behind them
        const bool al = a.nx % 4 == 0 &&
                        ((uintptr_t)a.in0 | (uintptr_t)a.in1 | (uintptr_t)a.out0 | (uintptr_t)a.out1) % 16 == 0;
        if (k != 2 || MODEL == CH || sizeof(T) == 8 || !al) return cudaErrorInvalidValue;
    }
    if constexpr (StencilInfo<ST>::dims == 2 && std::is_same<T, double>::value) {
        const bool small = (long long)a.nx * a.ny <= kSmallGrid2d;
        const bool strip_shape = g_step_variant == 2 || g_step_variant == 4;
        if (!strip_shape && small != (g_step_variant == 1)) {
            // small grids are latency bound: many small tiles instead of a few long strips
            constexpr int BX = 32, BY = 16, NT = 128;
            typedef Step2dTileShape<MODEL, ST, T, BX, BY> Sh;
            auto kern = step2d_tile_kernel<MODEL, ST, T, BX, BY, NT>;
            static const bool attr = [&] {
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
                return true;
            }();
            (void)attr;
            return launch_pdl(kern, dim3((a.nx + BX - 1) / BX, (a.ny + BY - 1) / BY), dim3(NT), Sh::smem_bytes, s, a);
        }
        // strip families: 0 the default shape, 2 narrower CTAs (64 threads), 4 half
        // the rows per batch; the autotuner picks per grid
        typedef Batch2d<MODEL> B;
        if (g_step_variant == 2) return launch_strips<MODEL, ST, T, 64, B::RB, 2 * B::CPS>(a, s, n_sm);
        if (g_step_variant == 4)
            return launch_strips<MODEL, ST, T, B::NT, (B::RB > 1 ? B::RB / 2 : 1), 2 * B::CPS>(a, s, n_sm);
        return launch_strips<MODEL, ST, T, B::NT, B::RB, B::CPS>(a, s, n_sm);
    } else if constexpr (StencilInfo<ST>::dims == 2) {
        typedef Step2dWarpShape<MODEL, ST, T> WS;
        const bool aligned = ((uintptr_t)a.in0 | (uintptr_t)a.in1 | (uintptr_t)a.out0 | (uintptr_t)a.out1) % 16 == 0;
        // (16-bit storage has no element-wise asynchronous copy)
        const bool al = a.nx % WS::V == 0 && aligned;
        if (g_step_variant == 0 && al) return launch_warp2d<MODEL, ST, T, true>(a, s, n_sm);
        if constexpr (sizeof(T) == 4) {
            if (g_step_variant == 0) return launch_warp2d<MODEL, ST, T, false>(a, s, n_sm);
        }
        // FP32 / BF16: one CTA per 128 x 32 tile
        constexpr int BX = 128, BY = 32, NT = 256;
        typedef Step2dTileShape<MODEL, ST, T, BX, BY> Sh;
        auto kern = step2d_tile_kernel<MODEL, ST, T, BX, BY, NT>;
        static const bool attr = [&] {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
            return true;
        }();
        (void)attr;
        dim3 grid((a.nx + BX - 1) / BX, (a.ny + BY - 1) / BY);
        return launch_pdl(kern, grid, dim3(NT), Sh::smem_bytes, s, a);
    } else if constexpr (!std::is_same<T, double>::value && MODEL == MC) {
        // Model C, FP32 / BF16 3D: plane rings (two steps per launch: families 0 and 1,
        // tiles of 8 and 16 rows; one step: families 0 and 4, 5); one CTA per box
        // (families 1 and 2, and 16-bit storage with unaligned rows)
        const bool al = a.nx % 4 == 0 &&
                        ((uintptr_t)a.in0 | (uintptr_t)a.in1 | (uintptr_t)a.out0 | (uintptr_t)a.out1) % 16 == 0;
        if (al) {
            constexpr bool tall2 = Step3dTbsShape<MODEL, ST, T, 16, 2>::smem_bytes <= kMaxSmemPerCta;
            if (k == 2 && g_step_variant == 1 && tall2) return launch_tbs<MODEL, ST, T, (tall2 ? 16 : 8), 2, true>(a, s, n_sm);
            if (k == 2) return launch_tbs<MODEL, ST, T, 8, 2, true>(a, s, n_sm);
            if (g_step_variant == 5) return launch_tbs<MODEL, ST, T, 16, 1, true>(a, s, n_sm);
            if (g_step_variant == 4) return launch_tbs<MODEL, ST, T, 8, 1, true>(a, s, n_sm);
            if (g_step_variant == 0) return launch_mc_rows<ST, T, true>(a, s, n_sm);
        } else if constexpr (sizeof(T) == 4) {
            if (g_step_variant == 0) return launch_mc_rows<ST, T, false>(a, s, n_sm);
        }
        constexpr int BX = 32, BY = 8, BZ = 8, NT = 256;
        typedef Step3dBoxShape<MODEL, ST, T, BX, BY, BZ> Sh;
        auto kern = step3d_box_kernel<MODEL, ST, T, BX, BY, BZ, NT>;
        static const bool attr = [&] {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
            return true;
        }();
        (void)attr;
        const int bx = (a.nx + BX - 1) / BX, by = (a.ny + BY - 1) / BY, bz = (a.nz + BZ - 1) / BZ;
        return launch_pdl(kern, dim3((unsigned)bx, (unsigned)by, (unsigned)bz), dim3(NT), Sh::smem_bytes, s, a);
    } else if constexpr (!std::is_same<T, double>::value) {
        if constexpr (MODEL == AC || MODEL == GS) {
            // two steps per launch with a plane ring per time level (families 0 and 1:
            // tiles of 8 and 16 rows; the taller ones only where their rings fit)
            constexpr bool tall2 = Step3dTbsShape<MODEL, ST, T, 16, 2>::smem_bytes <= kMaxSmemPerCta;
            if (k == 2 && g_step_variant == 1 && tall2) return launch_tbs<MODEL, ST, T, (tall2 ? 16 : 8), 2, true>(a, s, n_sm);
            if (k == 2) return launch_tbs<MODEL, ST, T, 8, 2, true>(a, s, n_sm);
        }
        constexpr int ATX = 16, ATY = 16;
        typedef Step3dAsyncShape<MODEL, ST, T, ATX, ATY> AS;
        const bool aligned = ((uintptr_t)a.in0 | (uintptr_t)a.in1 | (uintptr_t)a.out0 | (uintptr_t)a.out1) % 16 == 0;
        constexpr int WTY = 8;
        typedef Step3dWrShape<MODEL, ST, T, WTY> WS;
        // Family 0: the warp-row kernel.  FP32 chooses among its tiles, any alignment
        // (sp_wr.cuh); 16-bit storage takes rows of 32 lanes unless its queues spill.
        int fam = g_step_variant;
        if constexpr (sizeof(T) == 4) {
            if (fam == 0) {
                const cudaError_t e = launch_wr_f32(MODEL, ST, a, s, n_sm);
                if (e != cudaErrorNotSupported) return e;
                fam = 1;  // the plane ring is the cheaper one
            }
        } else if (fam == 0) {
            auto wkern = step3d_wr_kernel<MODEL, ST, T, WTY, 32, true>;
            static const bool spills = [&] {
                cudaFuncAttributes fa{};
                return cudaFuncGetAttributes(&fa, wkern) != cudaSuccess || fa.localSizeBytes > 16;
            }();
            if (!spills && a.nx % 4 == 0 && aligned) {
                const int tx = (a.nx + WS::TX - 1) / WS::TX, ty = (a.ny + WTY - 1) / WTY;
                const long long wave = (long long)n_sm * std::max(wr_occupancy<MODEL, ST, T, WTY, 32, true>(), 1);
                return launch_wr<MODEL, ST, T, WTY, 32, true>(
                    a, s, n_sm, lockstep_segments((long long)tx * ty, a.nz, 2 * WS::R, wave));
            }
            fam = 1;
        }
        if (fam == kTmaFamily && a.nx % AS::V == 0 && aligned) {
            // FP32 / BF16 3D: the plane ring with tensor-map plane loads
            TmaMaps maps;
            const cudaError_t e = encode_plane_maps(&maps, sizeof(T) == 2, a.in0, a.in1, a.nx, a.ny, a.nz, AS::SW,
                                                    AS::HIN);
            if (e != cudaSuccess) return e;
            auto kern = step3d_async_kernel<MODEL, ST, T, ATX, ATY, true>;
            static const int occ = [&] {
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AS::smem_bytes);
                int o = 1;
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, AS::NT, AS::smem_bytes);
                return o;
            }();
            const int tx = (a.nx + AS::TX - 1) / AS::TX, ty = (a.ny + ATY - 1) / ATY;
            const long long wave = (long long)n_sm * std::max(occ, 1);
            const int segs = lockstep_segments((long long)tx * ty, a.nz, 2 * AS::R, wave);
            const long long items = (long long)tx * ty * segs;
            return launch_pdl(kern, dim3((unsigned)std::min(items, wave)), dim3(AS::NT), AS::smem_bytes, s, a, tx, ty, segs, maps);
        }
        if (fam != 2 && a.nx % AS::V == 0 && aligned) {
            // FP32 / BF16 3D: cp.async plane ring with planes in flight
            auto kern = step3d_async_kernel<MODEL, ST, T, ATX, ATY, false>;
            static const int occ = [&] {
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AS::smem_bytes);
                int o = 1;
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, AS::NT, AS::smem_bytes);
                return o;
            }();
            const int tx = (a.nx + AS::TX - 1) / AS::TX, ty = (a.ny + ATY - 1) / ATY;
            const long long wave = (long long)n_sm * std::max(occ, 1);
            const int segs = lockstep_segments((long long)tx * ty, a.nz, 2 * AS::R, wave);
            const long long items = (long long)tx * ty * segs;
            return launch_pdl(kern, dim3((unsigned)std::min(items, wave)), dim3(AS::NT), AS::smem_bytes, s, a, tx, ty, segs, TmaMaps{});
        }
        // FP32 / BF16 3D, any nx: vectorised plane kernel, 64 x 32 tiles
        constexpr int TXT = 16, TYT = 32;
        typedef Step3dVecShape<MODEL, ST, T, TXT, TYT> Sh;
        auto kern = step3d_vec_kernel<MODEL, ST, T, TXT, TYT>;
        static const int occ = [&] {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
            int o = 1;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, Sh::NT, Sh::smem_bytes);
            return o;
        }();
        const int tx = (a.nx + Sh::TX - 1) / Sh::TX, ty = (a.ny + Sh::TY - 1) / Sh::TY;
        const long long planes = planes_per_cta((long long)tx * ty, a.nz, Sh::R, occ, n_sm);
        return launch_pdl(kern, dim3((unsigned)(((long long)tx * ty * a.nz + planes - 1) / planes)), dim3(Sh::NT), Sh::smem_bytes, s, a, tx, ty, planes);
    } else {
        if constexpr (MODEL != MC) {
            if (ST == L27 && g_step_variant == 0) return launch_zreg<MODEL, T>(a, s, n_sm);
        }
        if constexpr (MODEL == CH) {
            constexpr int TX = StencilInfo<ST>::r == 1 ? 64 : 32, TY = 32, NT = 256;
            if (!small_tile(a.nx, a.ny, TX, TY, 0.9)) return launch_step3d_tile<MODEL, ST, TX, TY, NT>(a, s, n_sm);
        }
        return launch_step3d_tile<MODEL, ST, kTX64, kTY64, kNT64>(a, s, n_sm);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_step_dispatch(int model, int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k) {
#define SP_STENCILS(M)                                                   \
    switch (stencil) {                                                   \
    case L5: return launch_step_t<M, L5, T>(a, s, n_sm, k);              \
    case L9BOX: return launch_step_t<M, L9BOX, T>(a, s, n_sm, k);        \
    case L9X4: return launch_step_t<M, L9X4, T>(a, s, n_sm, k);          \
    case L7: return launch_step_t<M, L7, T>(a, s, n_sm, k);              \
    case L27: return launch_step_t<M, L27, T>(a, s, n_sm, k);            \
    case L13X4: return launch_step_t<M, L13X4, T>(a, s, n_sm, k);        \
    }                                                                    \
    break;
    switch (model) {
    case AC: SP_STENCILS(AC)
    case CH: SP_STENCILS(CH)
    case GS: SP_STENCILS(GS)
    case MC: SP_STENCILS(MC)
    }
#undef SP_STENCILS
    return cudaErrorInvalidValue;
}

}  // namespace sp
