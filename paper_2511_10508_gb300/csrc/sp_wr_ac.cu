// sp_wr_ac.cu -- the 3D FP32 warp-row kernel instantiated for Allen-Cahn.
#define SP_WR_MODEL
#include "sp_wr.cuh"

namespace sp {

cudaError_t launch_wr_ac(int stencil, const StepArgs &a, cudaStream_t s, int n_sm) {
    switch (stencil) {
    case L7: return choose_wr_any<AC, L7, WrTile<8, 32, 604>, WrTile<12, 16, 448>, WrTile<24, 16, 888>>(a, s, n_sm);
    case L27: return choose_wr_any<AC, L27, WrTile<8, 32, 717>, WrTile<12, 16, 589>>(a, s, n_sm);
    case L13X4: return choose_wr_any<AC, L13X4, WrTile<8, 32, 1182>, WrTile<12, 16, 666>>(a, s, n_sm);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sp
