// sp_wr_ch.cu -- the 3D FP32 warp-row kernel instantiated for Cahn-Hilliard.
#define SP_WR_MODEL
#include "sp_wr.cuh"

namespace sp {

cudaError_t launch_wr_ch(int stencil, const StepArgs &a, cudaStream_t s, int n_sm) {
    switch (stencil) {
    case L7: return choose_wr_any<CH, L7, WrTile<8, 32, 1060>, WrTile<12, 16, 755>, WrTile<24, 16, 1367>>(a, s, n_sm);
    case L27: return choose_wr_any<CH, L27, WrTile<8, 32, 1797>, WrTile<12, 16, 1059>>(a, s, n_sm);
    case L13X4: return choose_wr_any<CH, L13X4, WrTile<16, 16, 1843>>(a, s, n_sm);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sp
