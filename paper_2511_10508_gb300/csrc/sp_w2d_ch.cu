// sp_w2d_ch.cu -- the 2D FP32 kernel of several steps on warp rows instantiated for Cahn-Hilliard.
#include "sp_w2d.cuh"

namespace sp {

cudaError_t launch_w2d_ch(int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k) {
    return launch_warptb_model<CH>(stencil, a, s, n_sm, k);
}

}  // namespace sp
