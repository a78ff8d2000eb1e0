// sp_w2d_gs.cu -- the 2D FP32 kernel of several steps on warp rows instantiated for Gray-Scott.
#include "sp_w2d.cuh"

namespace sp {

cudaError_t launch_w2d_gs(int stencil, const StepArgs &a, cudaStream_t s, int n_sm, int k) {
    return launch_warptb_model<GS>(stencil, a, s, n_sm, k);
}

}  // namespace sp
