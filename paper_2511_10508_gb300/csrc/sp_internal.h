// sp_internal.h -- declarations shared by the library's translation units
// (kernels, launchers and the C-ABI runtime).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <array>

#include "sp.h"
#include "sp_common.cuh"
#include "sp_split.h"

namespace sp {

constexpr int kMaxPatches = 2048;       // Gray-Scott seeded patches per grid
constexpr int kReduceThreads = 256;
constexpr int kReduceBlocksPerSM = 2;

struct ReduceGeom {
    int nx, ny, nz, dims;
    double h, cell_volume, c1, c2;
    double c3 = 0.0;            // Model C free energy: coupling
    const void *rho = nullptr;  // Model C free energy: the density field (else null)
    const void *jq[3] = {nullptr, nullptr, nullptr};  // Model H free energy: |j|^2/2 terms
    int nq = 0;
};

// Step launchers, one per storage type (sp_step_f64.cu, sp_step_f32.cu,
// sp_step_bf16.cu).  k forward-Euler steps from a.in* to a.out* in one launch;
// k: 1, or 2 or 4 (2D) or 2 (3D FP32 / BF16, see steps_per_launch_3d).
cudaError_t launch_step_f64(int model, int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k);
cudaError_t launch_step_f32(int model, int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k);
cudaError_t launch_step_bf16(int model, int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k);

// Kernel variant chosen per launch: 0 = the default for the grid, 1 (and 2) =
// alternative families (2D FP64: small tiles instead of strips, or strips instead
// of small tiles for grids up to 1024^2, and 2 / 4 = strips of 64 threads / of
// half the rows per batch; 2D FP32/BF16 single steps: shared-
// memory tiles instead of warp strips; 3D FP32/BF16: 1 = cp.async plane ring,
// 2 = register-staged plane rings, instead of warp rows; 3D FP64 27-point:
// shared-memory plane rings instead of z-streaming).  Set around each launch by
// the runtime.
extern thread_local int g_step_variant;

// 3D FP32 warp-row kernel, any alignment (sp_wr.cuh, one translation unit per model);
// cudaErrorNotSupported where the plane ring is the cheaper one.
cudaError_t launch_wr_ac(int stencil, const StepArgs &a, cudaStream_t s, int n_sm);
cudaError_t launch_wr_ch(int stencil, const StepArgs &a, cudaStream_t s, int n_sm);
cudaError_t launch_wr_gs(int stencil, const StepArgs &a, cudaStream_t s, int n_sm);
inline cudaError_t launch_wr_f32(int model, int stencil, const StepArgs &a, cudaStream_t s, int n_sm) {
    return model == AC ? launch_wr_ac(stencil, a, s, n_sm)
           : model == CH ? launch_wr_ch(stencil, a, s, n_sm) : launch_wr_gs(stencil, a, s, n_sm);
}

// 2D FP32, k = 2 or 4 steps per launch on warp rows (sp_w2d.cuh, one translation unit per
// model); cudaErrorNotSupported where the tiles are to be used.
cudaError_t launch_w2d_ac(int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k);
cudaError_t launch_w2d_ch(int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k);
cudaError_t launch_w2d_gs(int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k);
cudaError_t launch_w2d_mc(int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k);
inline cudaError_t launch_w2d(int model, int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k) {
    return model == AC   ? launch_w2d_ac(stencil, a, s, n_sm, k)
           : model == CH ? launch_w2d_ch(stencil, a, s, n_sm, k)
           : model == GS ? launch_w2d_gs(stencil, a, s, n_sm, k) : launch_w2d_mc(stencil, a, s, n_sm, k);
}

// Resident CTAs per SM by warps per CTA (1 .. MAXW) of a kernel that takes `smem` bytes per warp.
template <int MAXW, typename Kern> std::array<int, MAXW + 1> warp_occupancy(Kern kern, size_t smem) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(smem * MAXW));
    std::array<int, MAXW + 1> o{};
    for (int w = 1; w <= MAXW; ++w) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o[w], kern, 32 * w, smem * w);
        o[w] = std::max(o[w], 1);
    }
    return o;
}

// FP64 2D grids up to 1024^2 use small tiles by default (and may fuse steps).
constexpr long long kSmallGrid2d = 1LL << 20;

// 3D: two steps per launch for FP32 / BF16 Allen-Cahn, Gray-Scott and Model C
// (plane rings, grids with nx a multiple of 4), when asked for or autotuned.
inline int steps_per_launch_3d(int dtype, int model, int nx, int requested) {
    const bool ok = dtype != SP_F64 && (model == SP_ALLEN_CAHN || model == SP_GRAY_SCOTT || model == SP_MODEL_C) &&
                    nx % 4 == 0;
    return (ok && requested >= 2) ? 2 : 1;
}

// Steps fused per launch (temporal blocking) for a request of `requested`
// (0 = the library's choice, 1 = none): 2D grids support 2 and 4 (FP64 on small
// tiles, where a launch is short enough for its fixed cost to matter); 3D grids
// see steps_per_launch_3d.
// 2D FP32 grids fuse steps by default where warp rows do (sp_w2d.cuh; us per step with 1, 2 and 4):
// Allen-Cahn, Gray-Scott and Model C four with a radius-1 stencil (Gray-Scott 300 x 301 2.2 / 2.2 /
// 1.9, 2048^2 10.4 / 6.9 / 5.8, 16384^2 785 / 398 / 216).  A radius-2 stencil leaves room for two; four
// on tiles are the better choice on small grids (Allen-Cahn 1024^2 4.8 / 4.0 / 3.3, 2048^2 7.8 /
// 5.4 / 8.7; Gray-Scott 512^2 3.4 / 3.5 / 2.5, 1024^2 5.6 / 3.9 / 5.5).  Cahn-Hilliard
// (a step takes two halos) two with a radius-1 stencil on large grids (5-point 1024^2 3.7 / 3.1,
// 8192^2 98 / 57, odd rows 1503 x 1001 4.6 / 5.0, 4097 x 4095 27 / 18; 9-point box 2048^2 7.7 / 9.1, 3000^2
// 12.8 / 11.5, 8192^2 104 / 66).
// 2D FP64 grids with a radius-1 stencil fuse two steps while the
// 32 x 14 tiles of that kernel do not cost an SM one more tile than the 32 x 16 tiles of one step:
// up to one tile per SM, and from two per SM up to 2^18 points (us per step with 1 and 2:
// Allen-Cahn 256^2 3.5 / 2.7, 512^2 6.9 / 6.0, Gray-Scott 256^2 5.5 / 4.4; 257^2, where it does cost
// one, 5.7 / 6.5).
inline int steps_per_launch(int dims, int dtype, int model, int stencil, int64_t nx, int64_t ny, int n_sm, int requested) {
    const int radius = stencil == SP_LAP_9CROSS4 ? 2 : 1;
    if (dims != 2 || model == SP_MODEL_H) return 1;
    const int64_t npts = nx * ny;
    if (requested == 0) {
        if (dtype == SP_F64 && radius == 1 && npts <= (int64_t)1 << 18) {
            const int64_t tx = (nx + 31) / 32, one = tx * ((ny + 15) / 16), two = tx * ((ny + 13) / 14);
            return two <= n_sm || one >= 2 * n_sm ? 2 : 1;
        }
        if (dtype != SP_F32) return 1;
        if (model == SP_CAHN_HILLIARD)
            return radius == 1 && npts >= (int64_t)1 << (stencil != SP_LAP_5 ? 23 : nx % 4 == 0 ? 20 : 22) ? 2 : 1;
        return radius == 1 || npts <= (int64_t)1 << (model == SP_ALLEN_CAHN ? 21 : 18) ? 4 : 2;
    }
    if (requested >= 4) return 4;
    if (requested >= 2) return 2;
    return 1;
}

// 3D FP64 27-point Allen-Cahn, Cahn-Hilliard (two passes through `mu`, N
// doubles), Gray-Scott and Model C with x-pair sums shared between y neighbours:
// kernel family 0 of these grids.  Family 2 (not for Model C) is then the z-streaming kernel with plane
// sums in registers (step3d_zreg_kernel, family 0 of launch_step_f64), family 1
// the accessor-based plane ring.
constexpr int kZregFamily = 2;
cudaError_t launch_planes27_f64(int model, const StepArgs &a, void *mu, cudaStream_t s, int n_sm);
// 3D FP64 Cahn-Hilliard with the 7- and 13-point stencils in two passes through
// `mu` (N doubles): kernel family 0 of these grids; family kFusedFamily is the
// one-pass plane ring with mu on a halo ring (launch_step_f64's family 0).
constexpr int kFusedFamily = 2;
cudaError_t launch_ch_twopass_f64(int stencil, const StepArgs &a, void *mu, cudaStream_t s, int n_sm);
inline bool twopass_applies(int dims, int dtype, int stencil, int model) {
    return dims == 3 && dtype == SP_F64 && (stencil == SP_LAP_7 || stencil == SP_LAP_13CROSS4) && model == SP_CAHN_HILLIARD;
}
inline bool planes27_applies(int dims, int dtype, int stencil, int model) {
    return dims == 3 && dtype == SP_F64 && stencil == SP_LAP_27 &&
           (model == SP_ALLEN_CAHN || model == SP_CAHN_HILLIARD || model == SP_GRAY_SCOTT || model == SP_MODEL_C);
}

// Tensor-map (TMA) plane loads (sp_tma.cu): kernel family kTmaFamily of 3D
// FP32/BF16 Allen-Cahn, Cahn-Hilliard and Gray-Scott grids with nx a multiple of
// 16 bytes' worth of cells.  encode_plane_maps describes fields f0 and f1 (f1 may
// equal f0) as nx x ny x nz tensors with box_x x box_y x 1 boxes.
constexpr int kTmaFamily = 6;
bool tma_available();
cudaError_t encode_plane_maps(TmaMaps *maps, bool bf16, const void *f0, const void *f1, int nx, int ny, int nz,
                              int box_x, int box_y);

// Generated cross stencils (sp_generated.cu), radius up to kMaxGenRadius.
constexpr int kMaxGenRadius = 4;
int generated_weights(int order, int dims, double *wk, double *lambda_max);
cudaError_t launch_generated(int model, int dtype, int order, int dims, const double *wk, const StepArgs &a, void *mu,
                             cudaStream_t s, int n_sm);

// Model H (sp_model_h.cu): one step from in[0..nf) to out[0..nf) (m, then the
// components of j; unused entries null) through the mu buffer of N compute-
// precision values; c3g = c3 times the central-difference scale.
cudaError_t launch_model_h(int dtype, int stencil, void *const in[4], void *const out[4], void *mu, int nx, int ny,
                           int nz, const StepConsts &k, double c3g, cudaStream_t s, int n_sm);
cudaError_t launch_ic_currents(int dtype, void *const j[3], int dims, uint64_t N, uint64_t seed, int ic_kind, double amp,
                               cudaStream_t s, int n_sm);

// Unfused Cahn-Hilliard step (ablation only, kernel family kUnfusedFamily): mu
// into the caller's temporary of N compute-precision values, then the update.
constexpr int kUnfusedFamily = 3;
cudaError_t launch_unfused_ch(int dtype, int stencil, const StepArgs &a, void *mu, cudaStream_t s, int n_sm);

// Semi-implicit Fourier spectral scheme (sp_spectral.cu, with its own FFTs): a
// plan holds the twiddle tables, the resident spectrum and the transform
// buffer.  Functions return SP_* status codes.  spectral_step with `more` set
// also transforms the cubic term of the new field for the step that follows.
struct SpectralPlan;
int spectral_create(int dtype, int dims, int nx, int ny, int nz, double h, double growth, SpectralPlan **out);
void spectral_destroy(SpectralPlan *P);
int spectral_load(SpectralPlan *P, const void *phi, cudaStream_t s);
int spectral_step(SpectralPlan *P, int model, void *phi, double dt, double c1, double c2, double kappa, cudaStream_t s,
                  bool more);
const char *spectral_last_error();

cudaError_t launch_ic(int dtype, void *u, void *v, int model, int dims, int nx, int ny, int nz,
                      uint64_t seed, int ic_kind, double mean, double amp, int patches, int patch,
                      cudaStream_t s, int n_sm);

int reduce_blocks(uint64_t N, int n_sm);
cudaError_t launch_reduce(int dtype, int what, const void *f, const ReduceGeom &g, double *partials,
                          int nblocks, double *out, cudaStream_t s);

// Element-wise conversion between FP64 staging and the storage type.
cudaError_t launch_convert_from_f64(int dtype, const double *src, void *dst, uint64_t n, cudaStream_t s);
cudaError_t launch_convert_to_f64(int dtype, const void *src, double *dst, uint64_t n, cudaStream_t s);

// Launch with programmatic stream serialisation (the kernel calls pdl_enter() before
// touching global memory).  No kernel triggers its dependents early, so the next step's CTAs start
// as this one's exit, before its writes are flushed and its end is reported, and wait for that in
// pdl_enter(): about 0.5 us per launch (444 x 568 Cahn-Hilliard 2.96 -> 2.59 us per step).  Grids of many waves of
// CTAs gain nothing and lose a little (16384^2 Gray-Scott, 131072 tiles: 4.84 -> 4.90 ms),
// so they are launched plainly.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned long long)grid.x * grid.y * grid.z <= 8192 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace sp
