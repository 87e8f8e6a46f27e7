// Refined batch kernels with the ILU(0) preconditioner passes, likewise (see
// mlb_kernels_ilu.cu).
#include "mlb_solve.cuh"

namespace mlb {

template cudaError_t launch_batch_refine_pc<float, double, kIluWide>(const BatchItemR<float, double> *,
                                                            const BatchPlan &, int, cudaStream_t);
template int batch_refine_blocks_per_sm_pc<float, double, kIluWide>();
template cudaError_t launch_batch_refine_pc<float, double, kIluLevels>(const BatchItemR<float, double> *,
                                                            const BatchPlan &, int, cudaStream_t);
template int batch_refine_blocks_per_sm_pc<float, double, kIluLevels>();
template cudaError_t launch_batch_refine_pc<float, double, kIluAny>(const BatchItemR<float, double> *,
                                                            const BatchPlan &, int, cudaStream_t);
template int batch_refine_blocks_per_sm_pc<float, double, kIluAny>();
template cudaError_t launch_batch_refine_pc<cfloat, cdouble, kIluWide>(const BatchItemR<cfloat, cdouble> *,
                                                            const BatchPlan &, int, cudaStream_t);
template int batch_refine_blocks_per_sm_pc<cfloat, cdouble, kIluWide>();
template cudaError_t launch_batch_refine_pc<cfloat, cdouble, kIluLevels>(const BatchItemR<cfloat, cdouble> *,
                                                            const BatchPlan &, int, cudaStream_t);
template int batch_refine_blocks_per_sm_pc<cfloat, cdouble, kIluLevels>();
template cudaError_t launch_batch_refine_pc<cfloat, cdouble, kIluAny>(const BatchItemR<cfloat, cdouble> *,
                                                            const BatchPlan &, int, cudaStream_t);
template int batch_refine_blocks_per_sm_pc<cfloat, cdouble, kIluAny>();

}  // namespace mlb
