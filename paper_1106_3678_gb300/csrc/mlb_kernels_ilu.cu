// Real FP64 solve and batch kernels and the refined kernels with the ILU(0)
// preconditioner passes (see mlb_solve.cuh), in a translation unit of their
// own so that they compile in parallel with the rest of the library.
#include "mlb_solve.cuh"

namespace mlb {

template cudaError_t launch_batch_pc<double, kIluAny>(const BatchItem<double> *, const BatchPlan &, int, cudaStream_t);
template int batch_blocks_per_sm_pc<double, kIluAny>();
template cudaError_t launch_batch_refine_pc<float, double, kIluAny>(const BatchItemR<float, double> *,
                                                                 const BatchPlan &, int, cudaStream_t);
template cudaError_t launch_batch_refine_pc<cfloat, cdouble, kIluAny>(const BatchItemR<cfloat, cdouble> *,
                                                                   const BatchPlan &, int, cudaStream_t);
template int batch_refine_blocks_per_sm_pc<float, double, kIluAny>();
template int batch_refine_blocks_per_sm_pc<cfloat, cdouble, kIluAny>();

}  // namespace mlb
