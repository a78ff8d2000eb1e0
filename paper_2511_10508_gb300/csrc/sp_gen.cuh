// sp_gen.cuh -- arguments of the generated-stencil kernels, and the 2D FP32 strip kernel's launch.
#pragma once

#include "sp_internal.h"

namespace sp {

struct GenW {
    double w[kMaxGenRadius + 1];  // d w_0, w_1, ..., w_r
    float wf[kMaxGenRadius + 1];
};

struct GenArgs {
    StepArgs a;
    GenW W;
    void *mu;
};

// 2D FP32 on warp rows (sp_gen2d.cu); cudaErrorNotSupported where the tiles are to be used
cudaError_t launch_gen2d_f32(int model, int r, const GenArgs &g, cudaStream_t s, int n_sm);

}  // namespace sp
