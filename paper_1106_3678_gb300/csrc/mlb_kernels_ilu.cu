// FP64 batch kernels with the ILU(0) preconditioner passes (see
// mlb_solve.cuh): one per form of the passes, and one for a batch whose systems
// differ in it.  In a translation unit of their own so that they compile in
// parallel with the rest of the library.
#include "mlb_solve.cuh"

namespace mlb {

template cudaError_t launch_batch_pc<double, kIluWide>(const BatchItem<double> *, const BatchPlan &, int,
                                             cudaStream_t);
template int batch_blocks_per_sm_pc<double, kIluWide>();
template cudaError_t launch_batch_pc<double, kIluLevels>(const BatchItem<double> *, const BatchPlan &, int,
                                             cudaStream_t);
template int batch_blocks_per_sm_pc<double, kIluLevels>();
template cudaError_t launch_batch_pc<double, kIluAny>(const BatchItem<double> *, const BatchPlan &, int,
                                             cudaStream_t);
template int batch_blocks_per_sm_pc<double, kIluAny>();
template cudaError_t launch_batch_pc<cdouble, kIluWide>(const BatchItem<cdouble> *, const BatchPlan &, int,
                                             cudaStream_t);
template int batch_blocks_per_sm_pc<cdouble, kIluWide>();
template cudaError_t launch_batch_pc<cdouble, kIluLevels>(const BatchItem<cdouble> *, const BatchPlan &, int,
                                             cudaStream_t);
template int batch_blocks_per_sm_pc<cdouble, kIluLevels>();
template cudaError_t launch_batch_pc<cdouble, kIluAny>(const BatchItem<cdouble> *, const BatchPlan &, int,
                                             cudaStream_t);
template int batch_blocks_per_sm_pc<cdouble, kIluAny>();

}  // namespace mlb
