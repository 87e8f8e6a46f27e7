// Persistent solve and batch kernels of the FP64 method, templated on PC, the
// forms of the ILU(0) passes that the engine is built with (kNoIlu: no call to
// them anywhere in the kernel, so the unpreconditioned kernels keep their
// register allocation).  Included by mlb_kernels.cu (kNoIlu, and the dispatch),
// mlb_kernels_ilu.cu and mlb_kernels_ilu32.cu (batches), mlb_kernels_cplx.cu,
// mlb_kernels_bsr.cu, mlb_kernels_wide.cu (kIluWide) and mlb_kernels_flow.cu
// (kIluFlow, kIluLevels), which compile in parallel.
#pragma once

#include "mlb_internal.h"
#include "mlb_refine.cuh"

namespace mlb {

// ===========================================================================
// persistent solve kernel
// ===========================================================================
// One solve by the team described by `gs`: repeated calls of the method
// from the current x while the recursive residual met tol but the true
// residual did not (restart rule of this library), all iterations counted
// against one maxit; then the true residual; the team's rank-0 CTA writes
// the result record.  Consumer threads only.
template <typename T, int PC, int EW>
__device__ __forceinline__ void run_fp64_solve() {
    Engine<T, PC, EW> E;
    GridSync &gs = the_gs();
    const SolveCtl &ctl = the_ctl();
    const Acct &acct = the_acct();
    DevResult *const res = ctl.res;
    int64_t total = 0;
    int outer = 0;
    typename Engine<T, PC, EW>::Out o{1, 0, 0, 0, 0.0};
    // ILU(0): the method iterates on y = M x (y_0 = M x_0; x = M^{-1} y at
    // the end, from the final residual pass, which forms M^{-1} y)
    if constexpr (PC != kNoIlu) {
        if (E.sys().ilu.lu && E.ilu_begin()) E.ilu_to_y();
    }
    double true_rel = __longlong_as_double(0x7ff8000000000000LL);
    for (bool last = false; gs.ok;) {
        const auto r = E.inner(last, ctl.maxit - total, outer == 0, ctl.tol);
        if (!gs.ok) break;
        if (last) {
            double bn = sqrt(the_red().total[0]);
            if (bn == 0.0) bn = 1.0;
            true_rel = sqrt(the_red().total[1]) / bn;
            if constexpr (PC != kNoIlu) {
                if (E.sys().ilu.lu) E.ilu_to_x();
            }
            break;
        }
        o = r;
        total += o.iter;
        gs.sync();   // the residual pass that follows gathers x
        last = o.flag != 0 || o.iter == 0 || total >= ctl.maxit || outer >= ctl.max_outer;
        if (!last) outer++;
    }
    consumer_sync();   // the accounting is complete
    if (gs.bid == 0 && threadIdx.x == 0) {
        res->flag = o.flag;
        res->j = o.j;
        res->i = o.i;
        res->status = gs.ok ? 0 : (gs.bar ? ld_relaxed_i32(&gs.bar->status) : kStatusTimeout);
        if (!gs.ok && res->status == 0) res->status = kStatusTimeout;
        res->iter = total;
        res->spmv = acct.spmv;
        res->outer = outer;
        res->err = o.err;
        res->true_relres = true_rel;
        res->bytes = (double)acct.bytes;
        res->flops = (double)acct.flops;
        for (int q = 0; q < 5; ++q) res->ops[q] = acct.ops[q];
        res->ctas = (int32_t)gs.nblocks;
    }
}

// Allow the ring's dynamic shared memory for a kernel (idempotent).
static cudaError_t allow_ring(const void *fn) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRingBytes);
}

__device__ __forceinline__ void acct_reset() {
    Acct &acct = the_acct();
    if (threadIdx.x == 0) {
        for (int q = 0; q < 5; ++q) acct.ops[q] = 0;
        acct.spmv = 0;
        acct.bytes = 0;
        acct.flops = 0;
    }
    __syncthreads();
}

// One FP64 solve by a CTA: its producer warp and its consumer warps.
template <typename T, int PC, int EW>
__device__ __forceinline__ void run_cta() {
    Engine<T, PC, EW> E;
    E.attach();
    if ((threadIdx.x >> 5) == kConsumerWarps) {
        E.template serve<false>([](unsigned &) { return 0; });
    } else {
        run_fp64_solve<T, PC, EW>();
        the_gs().end_system();
    }
    __syncthreads();
}

template <typename T, int PC, int EW = 1>
__global__ void __launch_bounds__(kThreads, 1) solve_kernel(SysView<T> sys, SolveCtl ctl) {
    ring_init(the_ring(), ctl.timeout_ns);
    the_gs().seq() = 0;
    if (threadIdx.x == 0) {
        the_sys<T>() = sys;
        the_ctl() = ctl;
        the_gs().init(ctl.bar, ctl.slots, gridDim.x, blockIdx.x, ctl.timeout_ns);
    }
    acct_reset();   // includes the __syncthreads that publishes the objects
    run_cta<T, PC, EW>();
    ring_drain(the_ring(), the_gs().seqs[kConsumers], the_gs().seqs[0]);
}

// ===========================================================================
// batch: many independent systems in one persistent launch
// ===========================================================================
// Work distribution of a batch launch (BatchPlan).  team_next: the team's
// next position in order_big, agreed on by the team's CTAs: the rank-0 CTA
// takes it from the queue into one of two slots (a slot is rewritten two
// turns later, after every CTA of the team has passed the turn between),
// and a team barrier publishes it.  -1 when order_big is exhausted or the
// barrier failed.
__device__ __forceinline__ int team_next(const BatchPlan &p, unsigned team, unsigned rank, unsigned &tepoch,
                                         unsigned turn, int *sflag, int *s_next) {
    int *slot = p.team_item + 2 * team + (turn & 1u);
    if (rank == 0 && threadIdx.x == 0) *(volatile int *)slot = (int)atomicAdd(&p.queue[1], 1u);
    if (!grid_barrier(p.tbar + team, tepoch, (unsigned)p.team, p.timeout_ns, sflag)) return -1;
    if (threadIdx.x == 0) *s_next = ld_relaxed_i32(slot);
    __syncthreads();
    const int q = *s_next;
    return q < p.count_big ? q : -1;
}

// Runs the plan: solve(item index, team size, rank, barrier, slots) for
// each system this CTA takes (team size 1: this CTA alone).
template <typename Solve>
__device__ __forceinline__ void run_batch_plan(const BatchPlan &p, int *sflag, int *s_next, Solve solve) {
    if (blockIdx.x < (unsigned)(p.teams * p.team)) {
        const unsigned team = blockIdx.x / p.team, rank = blockIdx.x % p.team;
        unsigned tepoch = 0;
        for (unsigned turn = 0;; ++turn) {
            const int q = team_next(p, team, rank, tepoch, turn, sflag, s_next);
            if (q < 0) break;
            solve(p.order_big[q], (unsigned)p.team, rank, p.sbar + q,
                  p.sslots + (size_t)q * 2 * kMaxSums * p.team);
        }
    }
    for (;;) {
        if (threadIdx.x == 0) *s_next = (int)atomicAdd(&p.queue[0], 1u);
        __syncthreads();
        const int q = *s_next;
        if (q >= p.count_small) break;
        solve(p.order_small[q], 1u, 0u, (BarrierState *)nullptr, (Slot *)nullptr);
    }
}

// Each system is solved by the same method as a single solve: by a team
// (the same arithmetic as a solve with grid = team) or by one CTA alone
// with CTA-wide barriers and reductions in shared memory.
template <typename T, int PC>
__global__ void __launch_bounds__(kThreads, 1) batch_kernel(const BatchItem<T> *items, BatchPlan plan) {
    __shared__ int sflag;
    __shared__ int s_next;
    ring_init(the_ring(), plan.timeout_ns);
    the_gs().seq() = 0;
    run_batch_plan(plan, &sflag, &s_next, [&](int idx, unsigned nb, unsigned rk, BarrierState *bar, Slot *slots) {
        if (threadIdx.x == 0) {
            the_sys<T>() = items[idx].sys;
            the_ctl() = items[idx].ctl;
            the_gs().init(bar, slots, nb, rk, the_ctl().timeout_ns);
        }
        acct_reset();   // includes the __syncthreads that publishes the objects
        run_cta<T, PC, 1>();
    });
    ring_drain(the_ring(), the_gs().seqs[kConsumers], the_gs().seqs[0]);
}

template <typename T, int PC>
cudaError_t launch_batch_pc(const BatchItem<T> *items, const BatchPlan &plan, int grid, cudaStream_t st) {
    cudaError_t e = allow_ring((const void *)batch_kernel<T, PC>);
    if (e != cudaSuccess) return e;
    const BatchItem<T> *it = items;
    BatchPlan p = plan;
    void *args[] = {(void *)&it, (void *)&p};
    if (plan.teams > 0)
        return cudaLaunchCooperativeKernel((const void *)batch_kernel<T, PC>, dim3(grid), dim3(kThreads), args,
                                           kRingBytes, st);
    return cudaLaunchKernel((const void *)batch_kernel<T, PC>, dim3(grid), dim3(kThreads), args, kRingBytes, st);
}

template <typename T, int PC>
int batch_blocks_per_sm_pc() {
    int nb = 0;
    if (allow_ring((const void *)batch_kernel<T, PC>) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_kernel<T, PC>, kThreads, kRingBytes) != cudaSuccess)
        return 0;
    return nb;
}

template <typename T, int PC, int EW = 1>
cudaError_t launch_solve_pc(const SysView<T> &sys, const SolveCtl &ctl, int grid, cudaStream_t st) {
    SysView<T> s = sys;
    SolveCtl c = ctl;
    void *args[] = {(void *)&s, (void *)&c};
    cudaError_t e = allow_ring((const void *)solve_kernel<T, PC, EW>);
    if (e != cudaSuccess) return e;
    if (grid <= 1)
        return cudaLaunchKernel((const void *)solve_kernel<T, PC, EW>, dim3(1), dim3(kThreads), args, kRingBytes,
                                st);
    return cudaLaunchCooperativeKernel((const void *)solve_kernel<T, PC, EW>, dim3(grid), dim3(kThreads), args,
                                       kRingBytes, st);
}

template <typename T, int PC, int EW = 1>
int solve_blocks_per_sm_pc() {
    int nb = 0;
    if (allow_ring((const void *)solve_kernel<T, PC, EW>) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, solve_kernel<T, PC, EW>, kThreads, kRingBytes) !=
            cudaSuccess)
        return 0;
    return nb;
}

// ===========================================================================
// FP32-inner / FP64-refined persistent solve and batch kernels
// ===========================================================================
// One refined solve by a CTA: its producer warp and its consumer warps; the
// team's rank-0 CTA writes the result record.
template <typename T32, typename T64, int PC, int EW>
__device__ __forceinline__ void refine_cta() {
    Engine<T32, PC, EW> E;
    Refiner<T64, T32, EW> R;
    E.attach();
    RefineOut o{1, 0, 0, 0.0};
    if ((threadIdx.x >> 5) == kConsumerWarps) {
        E.template serve<true>([&](unsigned &sq) { return R.issue(sq); });
    } else {
        o = refine_solve<T32, T64, PC, EW>(E, R, the_ctl(), the_refctl());
        the_gs().end_system();
    }
    __syncthreads();
    GridSync &gs = the_gs();
    if (gs.bid == 0 && threadIdx.x == 0) {
        const Acct &acct = the_acct();
        DevResult *res = the_ctl().res;
        res->flag = o.flag;
        res->j = 0;
        res->i = 0;
        res->status = gs.ok ? 0 : (gs.bar ? ld_relaxed_i32(&gs.bar->status) : kStatusTimeout);
        if (!gs.ok && res->status == 0) res->status = kStatusTimeout;
        res->iter = o.iter;
        res->spmv = acct.spmv;
        res->outer = o.outer;
        res->err = o.err;
        res->true_relres = o.err;
        res->bytes = (double)acct.bytes;
        res->flops = (double)acct.flops;
        for (int k = 0; k < 5; ++k) res->ops[k] = acct.ops[k];
        res->ctas = (int32_t)gs.nblocks;
    }
    __syncthreads();
}

template <typename T32, typename T64, int PC>
__global__ void __launch_bounds__(kThreads, 1)
    batch_refine_kernel(const BatchItemR<T32, T64> *items, BatchPlan plan) {
    __shared__ int sflag;
    __shared__ int s_next;
    ring_init(the_ring(), plan.timeout_ns);
    the_gs().seq() = 0;
    run_batch_plan(plan, &sflag, &s_next, [&](int idx, unsigned nb, unsigned rk, BarrierState *bar, Slot *slots) {
        if (threadIdx.x == 0) {
            the_sys<T32>() = items[idx].sys;
            the_ref<T64>() = items[idx].rv;
            the_ctl() = items[idx].ctl;
            the_refctl() = items[idx].rc;
            the_gs().init(bar, slots, nb, rk, the_ctl().timeout_ns);
        }
        acct_reset();   // includes the __syncthreads that publishes the objects
        refine_cta<T32, T64, PC, 1>();
    });
    ring_drain(the_ring(), the_gs().seqs[kConsumers], the_gs().seqs[0]);
}

template <typename T32, typename T64, int PC>
cudaError_t launch_batch_refine_pc(const BatchItemR<T32, T64> *items, const BatchPlan &plan, int grid,
                                   cudaStream_t st) {
    cudaError_t e = allow_ring((const void *)batch_refine_kernel<T32, T64, PC>);
    if (e != cudaSuccess) return e;
    const BatchItemR<T32, T64> *it = items;
    BatchPlan p = plan;
    void *args[] = {(void *)&it, (void *)&p};
    if (plan.teams > 0)
        return cudaLaunchCooperativeKernel((const void *)batch_refine_kernel<T32, T64, PC>, dim3(grid),
                                           dim3(kThreads), args, kRingBytes, st);
    return cudaLaunchKernel((const void *)batch_refine_kernel<T32, T64, PC>, dim3(grid), dim3(kThreads), args,
                            kRingBytes, st);
}

template <typename T32, typename T64, int PC>
int batch_refine_blocks_per_sm_pc() {
    int nb = 0;
    if (allow_ring((const void *)batch_refine_kernel<T32, T64, PC>) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_refine_kernel<T32, T64, PC>, kThreads, kRingBytes) !=
            cudaSuccess)
        return 0;
    return nb;
}

// ===========================================================================
// FP32-inner / FP64-refined persistent solve kernel
// ===========================================================================
template <typename T32, typename T64, int PC, int EW = 1>
__global__ void __launch_bounds__(kThreads, 1)
    refine_kernel(SysView<T32> sys, RefView<T64> rv, SolveCtl ctl, RefCtl rc) {
    ring_init(the_ring(), ctl.timeout_ns);
    the_gs().seq() = 0;
    if (threadIdx.x == 0) {
        the_sys<T32>() = sys;
        the_ref<T64>() = rv;
        the_ctl() = ctl;
        the_refctl() = rc;
        the_gs().init(ctl.bar, ctl.slots, gridDim.x, blockIdx.x, ctl.timeout_ns);
    }
    acct_reset();   // includes the __syncthreads that publishes the objects
    refine_cta<T32, T64, PC, EW>();
    ring_drain(the_ring(), the_gs().seqs[kConsumers], the_gs().seqs[0]);
}

template <typename T32, typename T64, int PC, int EW = 1>
cudaError_t launch_refine_pc(const SysView<T32> &sys, const RefView<T64> &rv, const SolveCtl &ctl,
                          const RefCtl &rc, int grid, cudaStream_t st) {
    SysView<T32> s = sys;
    RefView<T64> r = rv;
    SolveCtl c = ctl;
    RefCtl q = rc;
    void *args[] = {(void *)&s, (void *)&r, (void *)&c, (void *)&q};
    cudaError_t e = allow_ring((const void *)refine_kernel<T32, T64, PC, EW>);
    if (e != cudaSuccess) return e;
    if (grid <= 1)
        return cudaLaunchKernel((const void *)refine_kernel<T32, T64, PC, EW>, dim3(1), dim3(kThreads), args, kRingBytes,
                                st);
    return cudaLaunchCooperativeKernel((const void *)refine_kernel<T32, T64, PC, EW>, dim3(grid), dim3(kThreads),
                                       args, kRingBytes, st);
}

template <typename T32, typename T64, int PC, int EW = 1>
int refine_blocks_per_sm_pc() {
    int nb = 0;
    if (allow_ring((const void *)refine_kernel<T32, T64, PC, EW>) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, refine_kernel<T32, T64, PC, EW>, kThreads, kRingBytes) !=
            cudaSuccess)
        return 0;
    return nb;
}

// 3x3-block storage (real values only), instantiated in mlb_kernels_bsr.cu.
extern template cudaError_t launch_solve_pc<double, kNoIlu, 3>(const SysView<double> &, const SolveCtl &, int,
                                                              cudaStream_t);
extern template cudaError_t launch_solve_pc<double, kIluFlow, 3>(const SysView<double> &, const SolveCtl &, int,
                                                             cudaStream_t);
extern template cudaError_t launch_solve_pc<double, kIluWide, 3>(const SysView<double> &, const SolveCtl &, int,
                                                             cudaStream_t);
extern template int solve_blocks_per_sm_pc<double, kNoIlu, 3>();
extern template int solve_blocks_per_sm_pc<double, kIluFlow, 3>();
extern template int solve_blocks_per_sm_pc<double, kIluWide, 3>();
extern template cudaError_t launch_refine_pc<float, double, kNoIlu, 3>(const SysView<float> &,
                                                                      const RefView<double> &, const SolveCtl &,
                                                                      const RefCtl &, int, cudaStream_t);
extern template cudaError_t launch_refine_pc<float, double, kIluFlow, 3>(const SysView<float> &,
                                                                     const RefView<double> &, const SolveCtl &,
                                                                     const RefCtl &, int, cudaStream_t);
extern template cudaError_t launch_refine_pc<float, double, kIluWide, 3>(const SysView<float> &,
                                                                     const RefView<double> &, const SolveCtl &,
                                                                     const RefCtl &, int, cudaStream_t);
extern template int refine_blocks_per_sm_pc<float, double, kNoIlu, 3>();
extern template int refine_blocks_per_sm_pc<float, double, kIluFlow, 3>();
extern template int refine_blocks_per_sm_pc<float, double, kIluWide, 3>();

// Instantiated in mlb_kernels_wide.cu.
extern template cudaError_t launch_solve_pc<double, kIluWide>(const SysView<double> &, const SolveCtl &, int,
                                                              cudaStream_t);
extern template cudaError_t launch_solve_pc<cdouble, kIluWide>(const SysView<cdouble> &, const SolveCtl &, int,
                                                               cudaStream_t);
extern template int solve_blocks_per_sm_pc<double, kIluWide>();
extern template int solve_blocks_per_sm_pc<cdouble, kIluWide>();
extern template cudaError_t launch_refine_pc<float, double, kIluWide>(const SysView<float> &, const RefView<double> &,
                                                                  const SolveCtl &, const RefCtl &, int,
                                                                  cudaStream_t);
extern template cudaError_t launch_refine_pc<cfloat, cdouble, kIluWide>(const SysView<cfloat> &,
                                                                    const RefView<cdouble> &, const SolveCtl &,
                                                                    const RefCtl &, int, cudaStream_t);
extern template int refine_blocks_per_sm_pc<float, double, kIluWide>();
extern template int refine_blocks_per_sm_pc<cfloat, cdouble, kIluWide>();

// Instantiated in mlb_kernels_ilu32.cu.
extern template cudaError_t launch_batch_refine_pc<float, double, kIluWide>(const BatchItemR<float, double> *,
                                                                   const BatchPlan &, int, cudaStream_t);
extern template int batch_refine_blocks_per_sm_pc<float, double, kIluWide>();
extern template cudaError_t launch_batch_refine_pc<float, double, kIluLevels>(const BatchItemR<float, double> *,
                                                                   const BatchPlan &, int, cudaStream_t);
extern template int batch_refine_blocks_per_sm_pc<float, double, kIluLevels>();
extern template cudaError_t launch_batch_refine_pc<float, double, kIluAny>(const BatchItemR<float, double> *,
                                                                   const BatchPlan &, int, cudaStream_t);
extern template int batch_refine_blocks_per_sm_pc<float, double, kIluAny>();
extern template cudaError_t launch_batch_refine_pc<cfloat, cdouble, kIluWide>(const BatchItemR<cfloat, cdouble> *,
                                                                   const BatchPlan &, int, cudaStream_t);
extern template int batch_refine_blocks_per_sm_pc<cfloat, cdouble, kIluWide>();
extern template cudaError_t launch_batch_refine_pc<cfloat, cdouble, kIluLevels>(const BatchItemR<cfloat, cdouble> *,
                                                                   const BatchPlan &, int, cudaStream_t);
extern template int batch_refine_blocks_per_sm_pc<cfloat, cdouble, kIluLevels>();
extern template cudaError_t launch_batch_refine_pc<cfloat, cdouble, kIluAny>(const BatchItemR<cfloat, cdouble> *,
                                                                   const BatchPlan &, int, cudaStream_t);
extern template int batch_refine_blocks_per_sm_pc<cfloat, cdouble, kIluAny>();

// Instantiated in mlb_kernels_cplx.cu.
extern template cudaError_t launch_solve_pc<cdouble, kNoIlu>(const SysView<cdouble> &, const SolveCtl &, int,
                                                            cudaStream_t);
extern template int solve_blocks_per_sm_pc<cdouble, kNoIlu>();
extern template cudaError_t launch_batch_pc<cdouble, kNoIlu>(const BatchItem<cdouble> *, const BatchPlan &, int,
                                                            cudaStream_t);
extern template int batch_blocks_per_sm_pc<cdouble, kNoIlu>();

// Instantiated in mlb_kernels_ilu.cu.
extern template cudaError_t launch_batch_pc<double, kIluWide>(const BatchItem<double> *, const BatchPlan &, int,
                                                    cudaStream_t);
extern template int batch_blocks_per_sm_pc<double, kIluWide>();
extern template cudaError_t launch_batch_pc<double, kIluLevels>(const BatchItem<double> *, const BatchPlan &, int,
                                                    cudaStream_t);
extern template int batch_blocks_per_sm_pc<double, kIluLevels>();
extern template cudaError_t launch_batch_pc<double, kIluAny>(const BatchItem<double> *, const BatchPlan &, int,
                                                    cudaStream_t);
extern template int batch_blocks_per_sm_pc<double, kIluAny>();
extern template cudaError_t launch_batch_pc<cdouble, kIluWide>(const BatchItem<cdouble> *, const BatchPlan &, int,
                                                    cudaStream_t);
extern template int batch_blocks_per_sm_pc<cdouble, kIluWide>();
extern template cudaError_t launch_batch_pc<cdouble, kIluLevels>(const BatchItem<cdouble> *, const BatchPlan &, int,
                                                    cudaStream_t);
extern template int batch_blocks_per_sm_pc<cdouble, kIluLevels>();
extern template cudaError_t launch_batch_pc<cdouble, kIluAny>(const BatchItem<cdouble> *, const BatchPlan &, int,
                                                    cudaStream_t);
extern template int batch_blocks_per_sm_pc<cdouble, kIluAny>();

// Instantiated in mlb_kernels_flow.cu.
extern template cudaError_t launch_solve_pc<double, kIluFlow>(const SysView<double> &, const SolveCtl &, int,
                                                              cudaStream_t);
extern template int solve_blocks_per_sm_pc<double, kIluFlow>();
extern template cudaError_t launch_refine_pc<float, double, kIluFlow>(const SysView<float> &, const RefView<double> &,
                                                                      const SolveCtl &, const RefCtl &, int,
                                                                      cudaStream_t);
extern template int refine_blocks_per_sm_pc<float, double, kIluFlow>();
extern template cudaError_t launch_solve_pc<cdouble, kIluLevels>(const SysView<cdouble> &, const SolveCtl &, int,
                                                                 cudaStream_t);
extern template int solve_blocks_per_sm_pc<cdouble, kIluLevels>();
extern template cudaError_t launch_refine_pc<cfloat, cdouble, kIluLevels>(const SysView<cfloat> &,
                                                                          const RefView<cdouble> &, const SolveCtl &,
                                                                          const RefCtl &, int, cudaStream_t);
extern template int refine_blocks_per_sm_pc<cfloat, cdouble, kIluLevels>();

}  // namespace mlb
