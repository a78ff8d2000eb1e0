// sp_w2d.cuh -- launch of the 2D FP32 kernel that takes K steps on warp rows (step2d_warptb_kernel).
#pragma once

#include <algorithm>

#include "sp_internal.h"
#include "sp_step.cuh"

namespace sp {

template <int MODEL, int ST, int K, bool AL>
cudaError_t launch_warptb(const StepArgs &a, cudaStream_t s, int n_sm) {
    typedef Step2dWarpTbShape<MODEL, ST, float, K> Sh;
    constexpr int WPC = Sh::NT / 32;
    auto kern = step2d_warptb_kernel<MODEL, ST, float, K, AL>;
    static const auto occ = warp_occupancy<WPC>(kern, Sh::warp_smem(AL));
    const int strips = (a.nx + Sh::OUT_COLS - 1) / Sh::OUT_COLS;
    const int wpc = strips >= 32 ? WPC : 1, groups = (strips + wpc - 1) / wpc;
    const long long total = (long long)groups * a.ny;
    const long long rows = warptb_rows(total, 2 * Sh::LAG, wpc, occ[wpc], n_sm);
    return launch_pdl(kern, dim3((unsigned)((total + rows - 1) / rows)), dim3(32 * wpc), Sh::warp_smem(AL) * wpc, s, a,
                      strips, groups, rows);
}

template <int MODEL, int ST, int K>
cudaError_t launch_warptb_any(const StepArgs &a, cudaStream_t s, int n_sm) {
    if constexpr (Step2dWarpTbShape<MODEL, ST, float, K>::fits) {
        const bool al = a.nx % 4 == 0 && ((uintptr_t)a.in0 | (uintptr_t)a.in1 | (uintptr_t)a.out0 | (uintptr_t)a.out1) % 16 == 0;
        // Aligned grids of middling size stay on tiles, which fill the SMs with less redundant
        // work (us per step of four, tiles / warp rows: Allen-Cahn 256^2 1.41 / 1.35, 512^2 1.47 / 1.65,
        // 700^2 1.60 / 1.91, 1024^2 2.24 / 2.23; Gray-Scott 1.80 / 1.64, 1.82 / 2.20, 2.20 / 2.52, 3.44 / 3.46;
        // 1280^2 4.58 / 3.2).
        const long long n = (long long)a.nx * a.ny;
        if (al && n > 1LL << 17 && n < 1LL << (StencilInfo<ST>::r == 1 ? 20 : 18)) return cudaErrorNotSupported;
        return al ? launch_warptb<MODEL, ST, K, true>(a, s, n_sm) : launch_warptb<MODEL, ST, K, false>(a, s, n_sm);
    } else {
        return cudaErrorNotSupported;
    }
}

template <int MODEL>
cudaError_t launch_warptb_model(int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k) {
    switch (stencil) {
    case L5: return k == 4 ? launch_warptb_any<MODEL, L5, 4>(a, s, n_sm) : launch_warptb_any<MODEL, L5, 2>(a, s, n_sm);
    case L9BOX: return k == 4 ? launch_warptb_any<MODEL, L9BOX, 4>(a, s, n_sm) : launch_warptb_any<MODEL, L9BOX, 2>(a, s, n_sm);
    case L9X4: return k == 4 ? launch_warptb_any<MODEL, L9X4, 4>(a, s, n_sm) : launch_warptb_any<MODEL, L9X4, 2>(a, s, n_sm);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sp
