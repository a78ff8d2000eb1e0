// sp_spectral_f32.cu -- spectral transforms instantiated for float.
#define SP_SPECTRAL_KERNELS
#include "sp_spectral.cuh"

namespace sp {

template cudaError_t run_rows<float>(const SpectralPlan *, RowMode, float *, Cplx<float>::type *, float, cudaStream_t);
template cudaError_t run_lines<float>(const SpectralPlan *, int, LineMode, int, const SpecCoef<float> &, Cplx<float>::type *,
                                      cudaStream_t);

}  // namespace sp
