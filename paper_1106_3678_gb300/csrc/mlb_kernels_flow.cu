// Real solve and refined kernels with the ILU(0) passes by slots
// (Engine::ilu_flow), in a translation unit of their own so that they compile
// in parallel with the rest of the library.
#include "mlb_solve.cuh"

namespace mlb {

template cudaError_t launch_solve_pc<double, kIluFlow>(const SysView<double> &, const SolveCtl &, int, cudaStream_t);
template int solve_blocks_per_sm_pc<double, kIluFlow>();
template cudaError_t launch_refine_pc<float, double, kIluFlow>(const SysView<float> &, const RefView<double> &,
                                                               const SolveCtl &, const RefCtl &, int, cudaStream_t);
template int refine_blocks_per_sm_pc<float, double, kIluFlow>();

}  // namespace mlb
