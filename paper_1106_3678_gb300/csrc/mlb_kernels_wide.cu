// Solve kernels and refined kernels with the streamed ILU(0)
// passes (Engine::ilu_wide), in a translation unit of their own so that they
// compile in parallel with the rest of the library.
#include "mlb_solve.cuh"

namespace mlb {

template cudaError_t launch_solve_pc<double, kIluWide>(const SysView<double> &, const SolveCtl &, int, cudaStream_t);
template int solve_blocks_per_sm_pc<double, kIluWide>();
template cudaError_t launch_solve_pc<cdouble, kIluWide>(const SysView<cdouble> &, const SolveCtl &, int, cudaStream_t);
template int solve_blocks_per_sm_pc<cdouble, kIluWide>();
template cudaError_t launch_refine_pc<float, double, kIluWide>(const SysView<float> &, const RefView<double> &,
                                                           const SolveCtl &, const RefCtl &, int, cudaStream_t);
template cudaError_t launch_refine_pc<cfloat, cdouble, kIluWide>(const SysView<cfloat> &, const RefView<cdouble> &,
                                                             const SolveCtl &, const RefCtl &, int, cudaStream_t);
template int refine_blocks_per_sm_pc<float, double, kIluWide>();
template int refine_blocks_per_sm_pc<cfloat, cdouble, kIluWide>();

}  // namespace mlb
