// sp_spectral_f64.cu -- spectral transforms instantiated for double.
#define SP_SPECTRAL_KERNELS
#include "sp_spectral.cuh"

namespace sp {

template cudaError_t run_rows<double>(const SpectralPlan *, RowMode, double *, Cplx<double>::type *, double, cudaStream_t);
template cudaError_t run_lines<double>(const SpectralPlan *, int, LineMode, int, const SpecCoef<double> &, Cplx<double>::type *,
                                      cudaStream_t);

}  // namespace sp
