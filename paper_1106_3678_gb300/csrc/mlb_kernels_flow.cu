// Solve and refined kernels for factors with many levels: real values by slots
// (Engine::ilu_flow), complex ones with a barrier per level
// (Engine::ilu_levels), in a translation unit of their own so that they compile
// in parallel with the rest of the library.
#include "mlb_solve.cuh"

namespace mlb {

template cudaError_t launch_solve_pc<double, kIluFlow>(const SysView<double> &, const SolveCtl &, int, cudaStream_t);
template int solve_blocks_per_sm_pc<double, kIluFlow>();
template cudaError_t launch_refine_pc<float, double, kIluFlow>(const SysView<float> &, const RefView<double> &,
                                                               const SolveCtl &, const RefCtl &, int, cudaStream_t);
template int refine_blocks_per_sm_pc<float, double, kIluFlow>();
template cudaError_t launch_solve_pc<cdouble, kIluLevels>(const SysView<cdouble> &, const SolveCtl &, int,
                                                          cudaStream_t);
template int solve_blocks_per_sm_pc<cdouble, kIluLevels>();
template cudaError_t launch_refine_pc<cfloat, cdouble, kIluLevels>(const SysView<cfloat> &, const RefView<cdouble> &,
                                                                   const SolveCtl &, const RefCtl &, int,
                                                                   cudaStream_t);
template int refine_blocks_per_sm_pc<cfloat, cdouble, kIluLevels>();

}  // namespace mlb
