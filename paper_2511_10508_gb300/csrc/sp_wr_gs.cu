// sp_wr_gs.cu -- the 3D FP32 warp-row kernel instantiated for Gray-Scott.
#define SP_WR_MODEL
#include "sp_wr.cuh"

namespace sp {

cudaError_t launch_wr_gs(int stencil, const StepArgs &a, cudaStream_t s, int n_sm) {
    switch (stencil) {
    case L7: return choose_wr_any<GS, L7, WrTile<8, 32, 1190>, WrTile<16, 16, 1214>>(a, s, n_sm);
    case L27: return choose_wr_any<GS, L27, WrTile<8, 32, 1707>, WrTile<12, 16, 1119>>(a, s, n_sm);
    case L13X4: return choose_wr_any<GS, L13X4, WrTile<8, 32, 1930>, WrTile<16, 16, 1771>>(a, s, n_sm);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sp
