// Persistent solve engine: ML(n)BiCGStabt (Algorithm 7.1 with M = I, i.e.
// Algorithm 4.1 with its k-loop split as k = jn + i, eq. 2.1) as one
// kernel launch.
//
// Every step of the method is a "pass" over the rows: a streaming update of
// a few N-vectors fused with the inner product(s) the next step needs, or a
// SELL-32 SpMV fused with its inner products.  Each pass ends in a
// deterministic reduction over the team (GridSync::reduce).  All scalars
// (alpha, beta~, beta, omega, c, e, err) are therefore bit-identical in
// every CTA, and every CTA takes the same branches (convergence, breakdown,
// g_n/r_n bookkeeping) without any host round trip.
//
// The iteration is an interpreter: the sequence of passes depends on n
// alone (Step), each pass is one case of one switch, and everything that
// lives from one pass to the next is in shared memory (Scalars, c, bt).  So
// a pass has the registers to itself (inlined into nested loops, the
// passes' values crowded each other out into local memory, which misses
// the small L1 beside the tile ring), and the producer warp follows the
// same sequence on its own, one pass ahead of the sums.
//
// Work distribution: every CTA of the team owns a contiguous, balanced range
// of 32-row slices (and the matching rows of every vector).  Every pass
// reads its streamed operands through a TMA-fed shared-memory tile
// pipeline (one producer warp, 15 consumer warps): vector chunks for the
// streaming passes, SELL slices (values and columns) for the SpMV, whose
// consumers gather x directly.
// Every vector a CTA bulk-loads was last written by that same CTA (its own
// rows) or is read-only.
//
// Storage ("ring"): g_k, w_k, c_k of iterate k = jn + s live in slot
// s = k mod n of G, W, c.  During step jn+i, slots < i hold block j and
// slots >= i still hold block j-1, as Algorithm 7.1 reads them.
//
// Fusions (none changes the order of any floating-point operation of a
// single element):
//   * x and r updates (alpha step) fused with ||r||^2, q_{i+1}^H r and, in
//     block 0, f_1^H r.
//   * the z_w sweep over block j-1 (Algorithm 7.1, steps 10-17) makes one
//     pass per coefficient over z_w only; the g-updates of that sweep feed
//     no inner product, so all of them run in the last pass, in the same
//     order, fused with the omega-correction (step 18) and the first
//     f-inner product (step 20).
//   * each f-sweep pass applies one update and computes the next f^H g.
//   * SpMV with the epilogue inner products c = q^H w (step 32), or
//     (A u)^H (A u) and (A u)^H u (step 38).
#pragma once

#include <type_traits>

#include "mlb_device.cuh"
#include "mlb_tiles.cuh"

namespace mlb {

constexpr int kThreads = kTileThreads;   // 15 consumer warps + 1 producer warp
constexpr int kMaxN = 64;       // largest number of shadow vectors
constexpr int kMaxSums = 5;     // doubles reduced per pass (max)
// Shared scratch of a team's reductions.
struct RedScratch {
    double part[kMaxSums][kConsumers / 2];
    double total[kMaxSums];
    int fail;
};

// Result record written by CTA 0 at the end of a solve.
struct DevResult {
    int32_t flag, j, i, status;
    int64_t iter, spmv, outer;
    double err, true_relres, bytes;
    int64_t ops[5];
    double flops;
    int32_t ctas, pad;   // CTAs that solved the system
};

enum { OP_MATVEC = 0, OP_DOT = 1, OP_SAXPY = 2, OP_SCALE = 3, OP_NORM = 4 };

// Per-CTA accounting in shared memory (identical in every CTA), kept by
// consumer thread kAcctThread: integer adds, beside the threads that work
// out the pass's scalars.
constexpr int kAcctThread = 64;
struct Acct {
    int64_t ops[5];   // Table 4.3 categories of the current inner call
    int64_t spmv;     // all sparse products of the solve
    // Algorithmic bytes and floating-point operations of the solve.
    int64_t bytes;
    int64_t flops;
};

// Scalars of the iteration, in shared memory.  After a pass's reduction
// consumer thread 0 works out the coefficient of the next pass (one FP64
// division, ~0.3 us on this GPU) while thread kErrThread takes the residual
// norm's decisions; the other threads only read `coef` and `exit`, so no
// FP64 instruction of 480 threads sits between two passes.
constexpr int kErrThread = 32;
template <typename S>
struct Scalars {
    S coef;          // coefficient of the next pass
    S e;             // q_{i+1}^H r
    S omega, inv_omega;
    double bnrm2;    // ||b|| (1 when b = 0)
    double rr;       // ||r||^2 (or ||u||^2) of the last update
    double far;      // a ||r||^2 above this is certainly not below tol
    double err;      // ||r|| / ||b|| where it was worked out
    int64_t iter;
    int exit;        // the iteration ends
    int flag, j, i;  // its result
    int act;         // (refined mode) replace the residual
    int conv;        // (refined mode) the true residual met its tolerance
};

// ILU(0) preconditioner M = L U of Algorithm 7.1 (the preconditioner of
// the paper's experiments, §5), stored in A's pattern: in row i, entries
// before the diagonal are L's (unit diagonal implied), the rest U's.  The
// solve iterates on y = M x, with every product A M^{-1} v formed as
// A (M^{-1} v).  Rows are grouped by level for the triangular solves: a
// row of level l depends only on rows of lower levels (of L, or of U taken
// from the last row upwards).  lu == nullptr: no ILU(0) preconditioner.
template <typename T>
struct IluView {
    const int64_t *rp;          // N+1; columns increase within each row
    const int32_t *ci;
    const T *lu;
    const int32_t *dpos;        // position of row i's diagonal, relative to rp[i]
    const int32_t *lrows;       // rows of L's levels: level l = lrows[lptr[l] .. lptr[l+1])
    const int32_t *lptr;
    const int32_t *urows;       // rows of U's levels
    const int32_t *uptr;
    int nlev_l, nlev_u;
    int64_t nnz;
    T *t;                       // ld: M^{-1} of the current product's input
    // the same rows in level-position order: entry count and the first
    // kIluEll entries of position q at e * N + q, U's diagonal at q
    const int32_t *lcnt, *ucnt, *lell_c, *uell_c;
    const T *lell_a, *uell_a, *udiag;
};

// Device view of one linear system.  Vectors have leading dimension `ld`
// (a multiple of 512 elements); entries N..ld-1 are zero and stay zero.
template <typename T>
struct SysView {
    int64_t N, ld, nnz;
    int64_t nslices;            // ld / 32
    const int64_t *slice_ptr;   // SELL-32: slice s spans [slice_ptr[s], slice_ptr[s+1])
    const int32_t *scol;        // column of entry (slice, k, lane) at off + 32k + lane
    const T *sval;
    int spt[3];                 // slices per SpMV tile with 0, 1, 2 epilogue vectors (<= 0: no tiles)
    int ew;                     // 1: scalar entries; 3: 3x3-block entries (three values, one column)
    int narrow_rows;            // no slice is wider than 7 entries (blocks)
    const T *Q;                 // ld x n
    const T *F;                 // ld x (n-1), F = A^H Q(:,0:n-2)
    T *G, *W;                   // ld x n rings
    T *x, *r, *z;               // ld
    T *b;                       // ld (written only by the refined-mode inner start)
    int n;
    IluView<T> ilu;             // ILU(0) preconditioner (ilu.lu == nullptr: none)
};

struct SolveCtl {
    double tol;
    int64_t maxit;
    double kappa;
    int max_outer;
    double *err_hist;           // device, may be null
    int64_t hist_cap;
    Slot *slots;                // [2][kMaxSums][gridDim], zeroed before the launch
    BarrierState *bar;
    DevResult *res;
    uint64_t timeout_ns;
};

// ---- element helpers used by Engine ---------------------------------------
__device__ __forceinline__ double subT(double a, double b) { return a - b; }
__device__ __forceinline__ float subT(float a, float b) { return a - b; }
template <typename R>
__device__ __forceinline__ cx<R> subT(cx<R> a, cx<R> b) { return {a.re - b.re, a.im - b.im}; }

__device__ __forceinline__ double ldg_val(const double *p) { return __ldg(p); }
__device__ __forceinline__ float ldg_val(const float *p) { return __ldg(p); }
__device__ __forceinline__ cdouble ldg_val(const cdouble *p) {
    double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ cfloat ldg_val(const cfloat *p) {
    float2 v = __ldg(reinterpret_cast<const float2 *>(p));
    return {v.x, v.y};
}
// Loads through L2 only: values another CTA wrote since the last team
// barrier (an SM's L1 may still hold an older copy of the line).
__device__ __forceinline__ double ldcg_val(const double *p) { return __ldcg(p); }
__device__ __forceinline__ float ldcg_val(const float *p) { return __ldcg(p); }
__device__ __forceinline__ cdouble ldcg_val(const cdouble *p) {
    double2 v = __ldcg(reinterpret_cast<const double2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ cfloat ldcg_val(const cfloat *p) {
    float2 v = __ldcg(reinterpret_cast<const float2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ double ldcs_val(const double *p) { return __ldcs(p); }
__device__ __forceinline__ float ldcs_val(const float *p) { return __ldcs(p); }
__device__ __forceinline__ cdouble ldcs_val(const cdouble *p) {
    double2 v = __ldcs(reinterpret_cast<const double2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ cfloat ldcs_val(const cfloat *p) {
    float2 v = __ldcs(reinterpret_cast<const float2 *>(p));
    return {v.x, v.y};
}

// FP32 counterpart of an FP64 element type, and the FP64 element type of
// an FP32 one (refined mode).
template <typename T> struct wide_of { using type = T; };
template <> struct wide_of<float> { using type = double; };
template <> struct wide_of<cfloat> { using type = cdouble; };
template <typename T> struct is_narrow { static constexpr bool value = false; };
template <> struct is_narrow<float> { static constexpr bool value = true; };
template <> struct is_narrow<cfloat> { static constexpr bool value = true; };

__device__ __forceinline__ float narrow_scaled(double v, double s) { return (float)(v * s); }
__device__ __forceinline__ cfloat narrow_scaled(cdouble v, double s) {
    return {(float)(v.re * s), (float)(v.im * s)};
}

// Balanced contiguous share [lo, hi) of `total` items for member `bid` of
// `nblocks`.
__device__ __forceinline__ void own_range(int64_t total, unsigned nblocks, unsigned bid, int64_t &lo, int64_t &hi) {
    lo = total * (int64_t)bid / nblocks;
    hi = total * (int64_t)(bid + 1) / nblocks;
}

// One SELL-32 slice (32 rows, width w, entries at slice offset `off`):
// the row sum of this lane, for slices of any width.
template <typename T>
__device__ __forceinline__ T sell_slice_sum(const int32_t *cp, const T *vp, int w, const T *xin) {
    T sum{};
    int k = 0;
    for (; k + 4 <= w; k += 4) {
        int32_t cc[4];
        T vv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) cc[u] = __ldcs(cp + 32 * (k + u));
#pragma unroll
        for (int u = 0; u < 4; ++u) vv[u] = ldcs_val(vp + 32 * (k + u));
#pragma unroll
        for (int u = 0; u < 4; ++u) sum = efma(vv[u], xin[cc[u]], sum);
    }
    if (k < w) {
        int32_t cc[3];
        T vv[3];
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (k + u < w) cc[u] = __ldcs(cp + 32 * (k + u));
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (k + u < w) vv[u] = ldcs_val(vp + 32 * (k + u));
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (k + u < w) sum = efma(vv[u], xin[cc[u]], sum);
    }
    return sum;
}

// 3x3-block storage ("triplet" SELL-32): entry k of lane l holds the three
// values of the lane's row in one 3x3 block, a_{row,c}, a_{row,c+1},
// a_{row,c+2}, at vp[3 (32 k)] .. (lane-strided by 96), and the block's first
// column c at cp[32 k]: one column index per three values.  The row sum is
// taken value by value in column order, which is the order of the row's
// scalar entries when the blocks are listed by block column.
template <typename T>
__device__ __forceinline__ T sell_slice_sum3(const int32_t *cp, const T *vp, int w, const T *xin) {
    T sum{};
    for (int k = 0; k < w; ++k) {
        const int32_t c = __ldcs(cp + 32 * k);
        const T v0 = ldcs_val(vp + 96 * k), v1 = ldcs_val(vp + 96 * k + 1), v2 = ldcs_val(vp + 96 * k + 2);
        sum = efma(v0, xin[c], sum);
        sum = efma(v1, xin[c + 1], sum);
        sum = efma(v2, xin[c + 2], sum);
    }
    return sum;
}
template <typename T>
__device__ __noinline__ T sell_slice_sum3_wide(const int32_t *cp, const T *vp, int w, const T *xin) {
    T sum{};
    for (int k = 0; k < w; ++k) {
        const int32_t c = cp[32 * k];
        const T x0 = xin[c], x1 = xin[c + 1], x2 = xin[c + 2];
        sum = efma(vp[96 * k], x0, sum);
        sum = efma(vp[96 * k + 1], x1, sum);
        sum = efma(vp[96 * k + 2], x2, sum);
    }
    return sum;
}

// Row sum of a slice wider than the pipelined path takes, from a stage
// (values at vp, column indices at cp, lane-strided by 32).  Out of line
// so that its registers do not weigh on the pipelined loop.
template <typename T>
__device__ __noinline__ T sell_slice_sum_wide(const int32_t *cp, const T *vp, int w, const T *xin) {
    T sum{};
    int k = 0;
    for (; k + 8 <= w; k += 8) {
        T xw[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) xw[u] = xin[cp[32 * (k + u)]];
#pragma unroll
        for (int u = 0; u < 8; ++u) sum = efma(vp[32 * (k + u)], xw[u], sum);
    }
    if (k < w) {
        T xw[7];
#pragma unroll
        for (int u = 0; u < 7; ++u)
            if (k + u < w) xw[u] = xin[cp[32 * (k + u)]];
#pragma unroll
        for (int u = 0; u < 7; ++u)
            if (k + u < w) sum = efma(vp[32 * (k + u)], xw[u], sum);
    }
    return sum;
}

// SELL-32 product over the slices [s_lo, s_hi) owned by this CTA: for
// every row, y = sum_k a_{row,k} xin[col_k], then fin(row, y, e, acc) where
// e[i] = epi[i][row] for the NE epilogue vectors (rows of this CTA).  The
// producer warp streams tiles of `spt` slices (values, column indices and
// the epilogue entries of the tile's rows) into the shared-memory ring;
// consumer warp w takes slice w of each tile.  Each warp is
// software-pipelined across tiles: the x gathers of tile t+1 are issued
// between the FMAs of tile t (each gather reuses the register its FMA has
// just read), so the FP64 pipe and the memory system work at the same time
// and the only global loads on a warp's critical path are the gathers.
// The epilogue's stores are fenced for later bulk (async-proxy) reads.
// EW = 3: the 3x3-block storage (see sell_slice_sum3); slice offsets and
// widths then count blocks.  Slices up to PW entries wide take the
// pipelined path (PW registers of gathered x per thread), wider ones a
// direct loop.  Returns false when a tile wait timed out.
//
// sell_consume is the consumer warps' part.
template <int NE, int EW = 1, int PW = 8, typename T, typename Fin, typename AccArr>
__device__ __forceinline__ bool sell_consume(TileRing *R, unsigned &cseq, uint64_t timeout_ns, int64_t s_lo,
                                             int64_t s_hi, int spt, const int64_t *slice_ptr, const int32_t *scol,
                                             const T *sval, const T *xin, const T *const (&epi)[NE > 0 ? NE : 1],
                                             int lane, Fin fin, AccArr &acc) {
    static_assert(EW == 1 || EW == 3, "scalar entries or 3x3 blocks");
    constexpr int kPipeW = PW;
    constexpr int NEA = NE > 0 ? NE : 1;
    const int cw = threadIdx.x >> 5;
    const SliceOffsets off(R, slice_ptr, s_lo, s_hi);
    bool ok = true;
    if (spt <= 0) {
        // slices too wide for one stage: direct loads, no pipeline
        for (int64_t s = s_lo + cw; s < s_hi; s += kConsumerWarps) {
            const int64_t o = off(s);
            const int w = (int)((off(s + 1) - o) >> 5);
            const int64_t row = s * 32 + lane;
            T e[NEA];
#pragma unroll
            for (int i = 0; i < NE; ++i) e[i] = epi[i][row];
            if constexpr (EW == 3)
                fin(row, sell_slice_sum3(scol + o + lane, sval + 3 * (o + lane), w, xin), e, acc);
            else
                fin(row, sell_slice_sum(scol + o + lane, sval + o + lane, w, xin), e, acc);
        }
        fence_proxy_async_global();
        return true;
    }
    // one slice of one tile, as seen by this warp: stage, entry offset of
    // the slice in the stage (o), entries of the tile (nv), slice width w
    // (w < 0: no slice for this warp in this tile)
    struct Job {
        int st, o, nv, w;
    };
    const int nt = (int)((s_hi - s_lo + spt - 1) / spt);
    // copies in registers (the epilogue's generic stores could alias them)
    unsigned char *const rbuf = R->buf;
    const unsigned cs0 = cseq;
    auto stage_of = [&](const Job &j) { return rbuf + (size_t)j.st * kStageBytes; };
    auto vals = [&](const Job &j) { return reinterpret_cast<const T *>(stage_of(j)) + EW * (j.o + lane); };
    auto cols = [&](const Job &j) {
        return reinterpret_cast<const int32_t *>(stage_of(j) + (size_t)j.nv * EW * sizeof(T)) + j.o + lane;
    };
    // epilogue entry i of this warp's row in the tile
    auto epv = [&](const Job &j, int i) {
        return reinterpret_cast<const T *>(stage_of(j) + (size_t)j.nv * (EW * sizeof(T) + 4))[(i * spt + cw) * 32 +
                                                                                             lane];
    };
    // wait for tile t and locate this warp's slice in it
    auto locate = [&](int t, Job &j) -> bool {
        const unsigned q = cs0 + (unsigned)t;
        j.st = (int)(q % kStages);
        j.o = j.nv = 0;
        j.w = -1;
        if (!mbar_wait(&R->full[j.st], (q / kStages) & 1u, timeout_ns)) return false;
        const int64_t s0 = s_lo + (int64_t)t * spt;
        const int64_t s1 = s0 + spt < s_hi ? s0 + spt : s_hi;
        const int64_t s = s0 + cw;
        if (s < s1) {
            const int64_t e0 = off(s0), es = off(s);
            j.nv = (int)(off(s1) - e0);
            j.o = (int)(es - e0);
            j.w = (int)((off(s + 1) - es) >> 5);
        }
        return true;
    };
    auto row_of = [&](int t) { return (s_lo + (int64_t)t * spt + cw) * 32 + lane; };
    int done = 0;
    // x gathers of slice j into xv (pipelined path: widths up to kPipeW)
    auto gather = [&](const Job &j, T (&xv)[kPipeW * EW]) {
        if (j.w >= 0 && j.w <= kPipeW) {
            const int32_t *cp = cols(j);
#pragma unroll
            for (int u = 0; u < kPipeW; ++u)
                if (u < j.w) {
                    const int32_t c = cp[32 * u];
#pragma unroll
                    for (int q = 0; q < EW; ++q) xv[EW * u + q] = xin[c + q];
                }
        }
    };
    // Tile t (slice jc, its x in xc): the FMAs, each followed by the gather
    // of slice jn (tile t+1, when `more`) into the register it has just
    // read; then the epilogue and the release of the stage.  (Gathering two
    // tiles ahead measured slower: 228 against 206 us per iteration at 128^3.)
    auto step = [&](int t, const Job &jc, T (&xc)[kPipeW * EW], const Job &jn, bool more) {
        const bool na = jc.w >= 0 && jc.w <= kPipeW;
        const bool nb = more && jn.w >= 0 && jn.w <= kPipeW;
        const T *va = vals(jc);
        const int32_t *cb = cols(jn);
        T sum{};
#pragma unroll
        for (int u = 0; u < kPipeW; ++u) {
            if (na && u < jc.w) {
#pragma unroll
                for (int q = 0; q < EW; ++q) sum = efma(va[32 * EW * u + q], xc[EW * u + q], sum);
            }
            if (nb && u < jn.w) {
                const int32_t c = cb[32 * u];
#pragma unroll
                for (int q = 0; q < EW; ++q) xc[EW * u + q] = xin[c + q];
            }
        }
        if (jc.w > kPipeW) {
            if constexpr (EW == 3) sum = sell_slice_sum3_wide(cols(jc), va, jc.w, xin);
            else sum = sell_slice_sum_wide(cols(jc), va, jc.w, xin);
        }
        if (jc.w >= 0) {
            T e[NEA];
#pragma unroll
            for (int i = 0; i < NE; ++i) e[i] = epv(jc, i);
            fin(row_of(t), sum, e, acc);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&R->empty[jc.st]);
        ++done;
    };
    if (nt > 0) {
        Job ja, jb;
        T xv[kPipeW * EW];
        ok = locate(0, ja);
        if (ok) gather(ja, xv);
        for (int t = 0; ok && t < nt; ++t) {
            const bool more = t + 1 < nt;
            if (more && !locate(t + 1, jb)) {
                ok = false;
                break;
            }
            step(t, ja, xv, jb, more);
            ja = jb;
        }
    }
    cseq = cs0 + (unsigned)done;
    fence_proxy_async_global();
    return ok;
}

// Producer and consumers of one product in one call (the fused product's
// kernel): pseq is the producer lane's tile counter, cseq a consumer's.
template <int NE, int EW = 1, int PW = 8, typename T, typename Fin, typename AccArr>
__device__ __forceinline__ bool sell_spmv(TileRing *R, unsigned &pseq, unsigned &cseq, uint64_t timeout_ns,
                                          int64_t s_lo, int64_t s_hi, int spt, const int64_t *slice_ptr,
                                          const int32_t *scol, const T *sval, const T *xin,
                                          const T *const (&epi)[NE > 0 ? NE : 1], int lane, Fin fin, AccArr &acc) {
    constexpr int NEA = NE > 0 ? NE : 1;
    if ((threadIdx.x >> 5) == kConsumerWarps) {
        if (lane != 0 || spt <= 0) return true;
        const SliceOffsets off(R, slice_ptr, s_lo, s_hi);
        const void *ep[NEA];
#pragma unroll
        for (int i = 0; i < NE; ++i) ep[i] = epi[i];
        return produce_sell(R, s_lo, s_hi, spt, off, sval, EW * (int)sizeof(T), (int)sizeof(T), scol, ep, NE, pseq,
                            timeout_ns);
    }
    return sell_consume<NE, EW, PW>(R, cseq, timeout_ns, s_lo, s_hi, spt, slice_ptr, scol, sval, xin, epi, lane, fin,
                                    acc);
}

// A 16-byte chunk of input i of a tile, from shared memory.
template <typename T>
__device__ __forceinline__ Pack<T> lds(const unsigned char *stage, int tc, int i, int k) {
    Pack<T> p;
    *reinterpret_cast<uint4 *>(&p) = *reinterpret_cast<const uint4 *>(stage + ((size_t)i * tc + k) * 16);
    return p;
}

// Coefficient from reduced sums (re[, im]).
template <typename T>
__device__ __forceinline__ typename coef_of<T>::type mk_coef(const double *v) {
    if constexpr (is_cx<T>::value) return cdouble{v[0], v[1]};
    else return v[0];
}

// Synchronisation state of one CTA within the team of CTAs that solves one
// system: the whole grid (a single solve), a group of CTAs of a batch
// launch (a large system of a batch), or the CTA alone (the other systems
// of a batch).  Every CTA of a team passes the same sequence of
// barriers and reductions, so the epochs advance in lock step.
// Several engines in one kernel share one GridSync.  Its members are called
// by every consumer thread; the producer warp takes no part.
//
// The object lives in shared memory, one per CTA (thread-private copies
// would sit in local memory, which the L1 left beside the tile ring cannot
// hold for 512 threads, so every access would go to L2).  Writers: the
// epochs thread 0; `ok` any thread (only ever set to false).  The tile
// sequence counters are per thread, in `seqs[threadIdx.x]` (the producer
// warp counts issued tiles, a consumer thread consumed ones): one shared
// counter would race, since in a pass of at most kStages tiles a fast warp
// can finish the pass before a slow one has read where it starts.
struct GridSync {
    unsigned nblocks;   // CTAs in the team
    unsigned bid;       // this CTA's rank in the team
    BarrierState *bar;
    Slot *slots;        // [2][kMaxSums][nblocks]: exchange e uses half e & 1
    RedScratch *red;    // shared
    uint64_t timeout_ns;
    unsigned epoch;     // exchanges this CTA has passed
    unsigned bepoch;    // barriers (sync) this CTA has passed
    bool ok;            // false once a barrier or a tile wait failed
    TileRing *ring;     // shared-memory tile pipeline of this CTA
    unsigned *seqs;     // shared, kThreads per-thread tile counters

    __device__ __forceinline__ unsigned &seq() const { return seqs[threadIdx.x]; }

    // Team of `nb` CTAs (rank `id`) with their own barrier state and slots;
    // nb = 1: this CTA alone (b and p null).
    __device__ GridSync(BarrierState *b, Slot *p, unsigned nb, unsigned id, RedScratch *r, uint64_t to, TileRing *rg,
                        unsigned *sq)
        : nblocks(nb), bid(id), bar(b), slots(p), red(r), timeout_ns(to), epoch(0), bepoch(0), ok(!rg->failed),
          ring(rg), seqs(sq) {
        r->fail = 0;
    }

    // Slots of sum k of the exchange `ep`.  Two halves suffice: a CTA
    // puts exchange ep + 2 only after it has seen every slot of ep + 1,
    // which a CTA puts after it has read every slot of ep.
    __device__ __forceinline__ Slot *slot_of(unsigned ep, int k) const {
        return slots + ((size_t)(ep & 1u) * kMaxSums + k) * nblocks;
    }

    // The last levels of reduce(), by one warp.  Out of line: its registers
    // stay out of the passes.
    __device__ __noinline__ void team_total(int k, bool fence) {
        const int lane = threadIdx.x & 31;
        const double *p = red->part[k] + lane;
        double t = p[0] + p[32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (nblocks > 1) {
            const unsigned ep = epoch + 1;
            Slot *const q = slot_of(ep, k);
            if (lane == 0) {
                if (fence) fence_acq_rel_gpu();   // this CTA's writes before its slot
                slot_put(q + bid, t, ep);
            }
            const bool got = slots_sum(q, nblocks, ep, bar, timeout_ns, t);
            if (fence) fence_acq_rel_gpu();       // the other CTAs' writes after their slots
            if (!got && lane == 0) red->fail = 1;
        }
        if (lane == 0) red->total[k] = t;
    }

    // Sum K values over the team into red->total[0, K), the same bits in
    // every CTA.  A dependent FP64 add costs about 60 cycles on this GPU and
    // one warp issues at most one FP64 instruction per ~60 cycles, so the
    // sums are short trees spread over many warps, independent sums
    // interleaved:
    //   CTA level 0: lanes l < 16 of every warp add their value to lane
    //                l+16's (240 partials per sum);
    //   CTA level 1: task (k, g), g < 64, on its own thread, adds partials
    //                g, g+64, g+128, g+192 as a pair tree;
    //   CTA level 2: warp k adds the 64 level-1 results of sum k (lane l:
    //                l and l+32), then an xor tree over the lanes;
    //   team:        with several CTAs, warp k of every CTA adds the CTA
    //                totals of sum k the same way, from their slots.
    // Fixed order for a given team size: deterministic.
    // fence: what any CTA of the team wrote before is visible to all of them
    // after (needed before a pass that gathers; the streaming passes read
    // their own CTA's rows only).  False (uniformly) when a wait failed.
    template <int K>
    __device__ __forceinline__ bool reduce(const double (&v)[K], bool fence) {
        static_assert(K <= kMaxSums && kMaxSums <= kConsumerWarps && kConsumers == 480, "reduction layout");
        constexpr int G1 = 64;
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const double h = v[k] + __shfl_down_sync(0xffffffffu, v[k], 16);
            if (lane < 16) red->part[k][warp * 16 + lane] = h;
        }
        consumer_sync();
        if (tid < K * G1) {
            double *p = red->part[tid / G1] + tid % G1;
            const double a0 = p[0], a1 = p[G1], a2 = p[2 * G1];
            // the last group has 48 partials
            p[0] = (a0 + a1) + (tid % G1 < 48 ? a2 + p[3 * G1] : a2);   // only this task reads slot 0
        }
        consumer_sync();
        if (warp < K) team_total(warp, fence);
        consumer_sync();
        if (tid == 0) epoch += 1;   // read again only after another barrier
        if (red->fail) { ok = false; return false; }
        return true;
    }

    // Team barrier (a counter: cheaper than an exchange where no value goes
    // with it).
    __device__ __forceinline__ bool sync() {
        arrive();
        return wait();
    }

    // sync() in two halves: arrive() once this CTA's writes are done,
    // wait() before reading other CTAs' writes; work between the two that
    // reads nothing written in this step overlaps the wait.  wait() returns
    // false (uniformly) when the barrier failed.
    __device__ __forceinline__ void arrive() {
        consumer_sync();
        if (nblocks > 1 && threadIdx.x == 0) grid_arrive(bar, bepoch);
    }
    __device__ __forceinline__ bool wait() {
        if (nblocks == 1) return true;   // arrive()'s barrier ordered the CTA
        if (threadIdx.x == 0 && !grid_wait(bar, bepoch, nblocks, timeout_ns)) red->fail = 1;
        consumer_sync();
        if (red->fail) { ok = false; return false; }
        return true;
    }

    // Hand a command to the producer warp (every consumer thread calls it).
    __device__ __forceinline__ void post(int cmd) {
        if (threadIdx.x == 0) {
            ring->cmd = cmd;
            ring->stop = 0;
        }
        __syncthreads();
    }
    // End of an iteration: stop the producer, meet it, and discard the tiles
    // it has issued ahead (their stages are released as if consumed).
    // `passes`: passes this CTA's consumers have finished.
    __device__ __forceinline__ void end_inner(unsigned &sq, unsigned passes) {
        if (threadIdx.x == 0) {
            *(volatile int *)&ring->stop = 1;
            ring->passes = passes;
        }
        __syncthreads();
        for (const unsigned last = ring->issued; sq != last; ++sq) {
            if (!mbar_wait(&ring->full[sq % kStages], (sq / kStages) & 1u, timeout_ns)) {
                ring->failed = 1;
                ok = false;
                break;
            }
            __syncwarp();
            if ((threadIdx.x & 31) == 0) mbar_arrive(&ring->empty[sq % kStages]);
        }
        consumer_sync();
    }
};

// One pass of the iteration (Engine::inner) and the pass after it: a
// function of n alone, which the producer warp follows too.  i: the slot the
// step builds (ALPHA uses slot i - 1; i = n: the block's last update); s:
// the column a sweep's pass uses; first: block 0.
enum { P_SPMV_C, P_ALPHA, P_SPMV_Z, P_OMEGA, P_W_FIRST, P_W_ROUND, P_W_LAST, P_F_ROUND, P_G_J0 };
struct Step {
    int op = P_SPMV_C, i = 0, s = 0;
    bool first = true;
    __device__ __forceinline__ void advance(int n) {
        switch (op) {
        case P_SPMV_C: ++i; op = P_ALPHA; break;
        case P_ALPHA: op = i == n ? P_SPMV_Z : first ? P_G_J0 : i == n - 1 ? P_W_LAST : P_W_FIRST; break;
        case P_SPMV_Z: op = P_OMEGA; break;
        case P_OMEGA:
            i = 0;
            first = false;
            op = n == 1 ? P_W_LAST : P_W_FIRST;
            break;
        case P_W_FIRST: s = i + 1; op = s < n - 1 ? P_W_ROUND : P_W_LAST; break;
        case P_W_ROUND: ++s; op = s < n - 1 ? P_W_ROUND : P_W_LAST; break;
        case P_W_LAST: s = 0; op = i == 0 ? P_SPMV_C : P_F_ROUND; break;
        case P_F_ROUND: ++s; op = s <= i - 1 ? P_F_ROUND : P_SPMV_C; break;
        default: s = 1; op = i >= 2 ? P_F_ROUND : P_SPMV_C; break;   // P_G_J0
        }
    }
};

// A call of Engine::inner without residual replacement (every solve but
// the refined mode's FP32 inner one).
struct NoHook {
    static constexpr bool kActive = false;
};

// PC: built with the ILU(0) preconditioner passes (ilu_pre and the
// product passes' switch to M^{-1} of their input); without it none of
// that code is reachable.  EW: the matrix storage of the products (1:
// scalar SELL-32; 3: 3x3 blocks, see sell_slice_sum3).
//
// The consumer threads run inner() and the other members; the producer warp
// runs serve() beside them.
template <typename T, bool PC = false, int EW = 1>
struct Engine {
    using S = typename coef_of<T>::type;                      // FP64 coefficient
    using ACC = typename real_of<T>::type;                    // thread accumulator
    static constexpr int DS = dslots<T>();
    static constexpr int PW = Pack<T>::W;
    static constexpr int CPS = 32 * sizeof(T) / 16;           // 16-byte chunks per slice

    const SysView<T> &sys;
    const SolveCtl &ctl;
    GridSync &gs;
    // shared memory
    S *c;            // kMaxN
    S *bt;           // kMaxN
    Acct *acct;
    Scalars<S> *sc;
    // ownership: slices [s_lo, s_hi), chunks [c_lo, c_hi)
    int64_t s_lo, s_hi, c_lo, c_hi;

    // Constructed by one thread in shared memory (one engine per CTA; see
    // GridSync); every thread then calls attach().
    __device__ Engine(const SysView<T> &s, const SolveCtl &k, GridSync &g, S *c_, S *bt_, Acct *acct_,
                      Scalars<S> *sc_)
        : sys(s), ctl(k), gs(g), c(c_), bt(bt_), acct(acct_), sc(sc_) {
        own_range(s.nslices, g.nblocks, g.bid, s_lo, s_hi);
        c_lo = s_lo * CPS;
        c_hi = s_hi * CPS;
    }
    __device__ void attach() { soff_load(gs.ring, sys.slice_ptr, s_lo, s_hi); }
    // Counts one Table 4.3 operation and its algorithmic floating-point
    // operations (real arithmetic): a product 2 per stored entry; an inner
    // product, AXPY or norm 2 per element; a scaling 1 per element.
    // Complex values: a multiply-add is 8 real operations, |v|^2 4, a
    // scaling 6.
    __device__ __forceinline__ void op(int which, int cnt = 1) {
        if (threadIdx.x == kAcctThread) {
            acct->ops[which] += cnt;
            constexpr bool cx_ = is_cx<T>::value;
            const int64_t N = sys.N;
            int64_t f;
            if (which == OP_MATVEC) f = (cx_ ? 8 : 2) * sys.nnz;
            else if (which == OP_SCALE) f = (cx_ ? 6 : 1) * N;
            else if (which == OP_NORM) f = (cx_ ? 4 : 2) * N;
            else f = (cx_ ? 8 : 2) * N;
            acct->flops += cnt * f;
        }
    }

    __device__ __forceinline__ const T *Qc(int k) const { return sys.Q + (int64_t)k * sys.ld; }
    __device__ __forceinline__ const T *Fc(int k) const { return sys.F + (int64_t)k * sys.ld; }
    __device__ __forceinline__ T *Gc(int k) const { return sys.G + (int64_t)k * sys.ld; }
    __device__ __forceinline__ T *Wc(int k) const { return sys.W + (int64_t)k * sys.ld; }

    __device__ __forceinline__ void vbytes(int nvec) {
        if (threadIdx.x == kAcctThread) acct->bytes += nvec * sys.N * (int64_t)sizeof(T);
    }
    __device__ __forceinline__ void sbytes(int nextra) {
        // SpMV: entries (values, and a column index per stored entry of EW
        // values), row_ptr-equivalent, x read once, y written once, plus
        // `nextra` epilogue vectors.
        if (threadIdx.x == kAcctThread) {
            acct->bytes += sys.nnz * (int64_t)sizeof(T) + sys.nnz / EW * 4 + 4 * (sys.N + 1) +
                           (2 + nextra) * sys.N * (int64_t)sizeof(T);
            acct->spmv++;
        }
    }

    // ------------------------------------------------------------------
    // the producer warp
    // ------------------------------------------------------------------

    // Issue the tiles of pass `st` (the input order of each pass is that of
    // its consumer side below).
    __device__ __forceinline__ int issue(const Step &st, unsigned &sq) {
        const int lane = threadIdx.x & 31, n = sys.n, i = st.i, s = st.s;
        TileRing *const R = gs.ring;
        const T *p = nullptr;
        int ni = 0;
        switch (st.op) {
        case P_SPMV_C:
        case P_SPMV_Z:
            return issue_product(st.op == P_SPMV_C ? Qc(i) : sys.r, 1, sq);
        case P_ALPHA: {
            const bool hq = i < n, f0 = st.first && hq;
            ni = 4 + (hq ? 1 : 0) + (f0 ? 1 : 0);
            p = lane == 0 ? sys.x : lane == 1 ? Gc(i - 1) : lane == 2 ? sys.r : lane == 3 ? Wc(i - 1)
                : lane == 4 && hq ? Qc(i) : sys.F;
            break;
        }
        case P_OMEGA:
            ni = 4;
            p = lane == 0 ? sys.x : lane == 1 ? sys.r : lane == 2 ? sys.z : sys.Q;
            break;
        case P_W_FIRST:
            ni = 3;
            p = lane == 0 ? sys.r : lane == 1 ? Wc(i) : Qc(i + 1);
            break;
        case P_W_ROUND:
            ni = 3;
            p = lane == 0 ? Wc(i) : lane == 1 ? Wc(s) : Qc(s + 1);
            break;
        case P_W_LAST: {
            const int nt = n - 1 - i, ntile = nt < kMaxInputs - 4 ? nt : kMaxInputs - 4, f = i > 0 ? 1 : 0;
            ni = 3 + f + ntile;
            p = lane == 0 ? Wc(i) : lane == 1 ? Gc(i) : lane == 2 ? (i == n - 1 ? sys.r : Wc(n - 1))
                : lane == 3 && f ? sys.F : Gc(i + 1 + lane - 3 - f);
            break;
        }
        case P_F_ROUND:
            ni = s + 1 <= i - 1 ? 3 : 2;
            p = lane == 0 ? Gc(i) : lane == 1 ? Gc(s) : Fc(s + 1);
            break;
        default:   // P_G_J0
            ni = i >= 2 ? 3 : 2;
            p = lane == 0 ? sys.r : lane == 1 ? sys.G : Fc(1);
            break;
        }
        return produce_lanes(R, p, ni, c_lo, c_hi, sq, gs.timeout_ns);
    }
    // Tiles of a product with `ne` epilogue vectors (lane 2 + k copies
    // vector k, its own `epi`).
    __device__ __forceinline__ int issue_product(const T *epi, int ne, unsigned &sq) {
        if (sys.spt[ne] <= 0) return 0;
        const SliceOffsets off(gs.ring, sys.slice_ptr, s_lo, s_hi);
        return produce_sell_lanes(gs.ring, s_lo, s_hi, sys.spt[ne], off, sys.sval, EW * (int)sizeof(T),
                                  (int)sizeof(T), sys.scol, epi, ne, sq, gs.timeout_ns);
    }
    // Wait until the consumers have finished the pass.
    __device__ __forceinline__ int wait_done(unsigned &passes) {
        int st = 0;
        if ((threadIdx.x & 31) == 0) st = producer_wait(gs.ring, &gs.ring->done, passes & 1u, gs.timeout_ns);
        st = __shfl_sync(0xffffffffu, st, 0);
        if (st == 0) passes += 1;
        return st;
    }
    // The producer warp's side of a system: commands of the consumers until
    // kCmdExit.  Decide: the iteration asks the consumers after every update
    // of r (refined mode).  residual64 issues the FP64 residual's tiles.
    template <bool Decide, typename Fn>
    __device__ __forceinline__ void serve(Fn residual64) {
        TileRing *const R = gs.ring;
        unsigned sq = gs.seq(), passes = R->passes;
        for (;;) {
            __syncthreads();
            const int cmd = R->cmd;
            if (cmd == kCmdExit) break;
            int st = 0;
            if (cmd == kCmdResidual) {
                st = issue_product((threadIdx.x & 31) == 2 ? sys.b : sys.Q, 2, sq);
                if (st == 0) st = wait_done(passes);
            } else if (cmd == kCmdResidual64) {
                st = residual64(sq);
                if (st == 0) st = wait_done(passes);
            } else {
                const int n = sys.n;
                bool met = false;   // the consumers' end_inner has been met at a decision
                for (Step p; st == 0; p.advance(n)) {
                    st = issue(p, sq);
                    if (st == 0) st = wait_done(passes);
                    if constexpr (Decide) {
                        if (st == 0 && (p.op == P_ALPHA || p.op == P_OMEGA)) {
                            if ((threadIdx.x & 31) == 0) R->issued = sq;
                            __syncthreads();
                            if (R->stop) {
                                met = true;
                                break;
                            }
                            if (R->cmd == kCmdResidual64) {
                                st = residual64(sq);
                                if (st == 0) st = wait_done(passes);
                                if (st == 0) {
                                    if ((threadIdx.x & 31) == 0) R->issued = sq;
                                    __syncthreads();
                                    if (R->stop) {
                                        met = true;
                                        break;
                                    }
                                }
                            }
                        }
                    }
                }
                if (st == 2) R->failed = 1;
                if (!met) {
                    if ((threadIdx.x & 31) == 0) R->issued = sq;
                    __syncthreads();
                }
                passes = R->passes;
                continue;
            }
            if (st == 2) R->failed = 1;
            if ((threadIdx.x & 31) == 0) R->passes = passes;
        }
        gs.seq() = sq;
        if ((threadIdx.x & 31) == 0) R->passes = passes;
    }

    // ------------------------------------------------------------------
    // the consumers' side of the passes
    // ------------------------------------------------------------------

    // Streaming pass through the tile pipeline: fn(chunk, stage, k) for
    // every chunk of this CTA.
    template <typename Fn>
    __device__ __forceinline__ void tiles(int tc, unsigned &sq, Fn fn) {
        TileRing *const ring = gs.ring;
        if (!consume(ring, TileGeom{tc, c_lo, c_hi}, sq, gs.timeout_ns, fn)) ring->failed = 1;
        pass_done(ring);
    }
    template <int K>
    __device__ __forceinline__ bool reduce(const ACC (&acc)[K], bool fence) {
        double v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = (double)acc[k];
        return gs.template reduce<K>(v, fence) && ring_ok();
    }
    // A failed tile wait marks the ring; the pass's reduction or barrier
    // then reports it.
    __device__ __forceinline__ bool ring_ok() {
        if (gs.ring->failed) { gs.ok = false; return false; }
        return true;
    }

    // SELL-32 SpMV pass over the owned slices (matrix tiles through the
    // ring).
    template <int NE, typename Fin, int K>
    __device__ __forceinline__ void spmv_rows(const T *xin, const T *const (&epi)[NE], unsigned &sq, Fin fin,
                                              ACC (&acc)[K]) {
        // with ILU(0) the product is A t, t = M^{-1} xin formed by the
        // caller (ilu_pre) before the pass
        if constexpr (PC) {
            if (sys.ilu.lu) xin = sys.ilu.t;
        }
        bool okw;
        // FP32 and complex engines: a pipelined width of 7 where the rows
        // allow it (fewer registers of gathered x); the real FP64 engine
        // keeps 8 (no gain at 7)
        if constexpr (is_narrow<T>::value || is_cx<T>::value) {
            if (sys.narrow_rows)
                okw = sell_consume<NE, EW, 7>(gs.ring, sq, gs.timeout_ns, s_lo, s_hi, sys.spt[NE], sys.slice_ptr,
                                              sys.scol, sys.sval, xin, epi, threadIdx.x & 31, fin, acc);
            else
                okw = sell_consume<NE, EW>(gs.ring, sq, gs.timeout_ns, s_lo, s_hi, sys.spt[NE], sys.slice_ptr,
                                           sys.scol, sys.sval, xin, epi, threadIdx.x & 31, fin, acc);
        } else {
            okw = sell_consume<NE, EW>(gs.ring, sq, gs.timeout_ns, s_lo, s_hi, sys.spt[NE], sys.slice_ptr, sys.scol,
                                       sys.sval, xin, epi, threadIdx.x & 31, fin, acc);
        }
        if (!okw) gs.ring->failed = 1;
        pass_done(gs.ring);
    }

    // ------------------------------------------------------------------
    // ILU(0) preconditioner (Algorithm 7.1 with M = L U)
    // ------------------------------------------------------------------

    // One row of a triangular solve, loaded ahead: its index, up to
    // kIluReg entries (column, factor value) in registers, where the rest
    // of its entries start and end, and the row's right-hand-side entry
    // (forward) or its U diagonal (backward).  i < 0: no row.
    static constexpr int kIluReg = 4;   // == kIluEll (entries stored by position)
    struct IluRow {
        int i, cnt;
        int64_t rest, end;
        int32_t c[kIluReg];
        T a[kIluReg];
        T v;
    };
    // Row q of L's level order (forward: entries before the diagonal).
    // Its count and first entries are read by position, independently of
    // the row index; entries beyond kIluReg come from the pattern.
    __device__ __forceinline__ void ilu_fetch_l(int64_t q, int64_t hi, const T *v, IluRow &R) const {
        R.i = -1;
        if (q >= hi) return;
        const IluView<T> &M = sys.ilu;
        const int64_t N = sys.N;
        const int i = M.lrows[q];
        const int n = M.lcnt[q];
        const int cnt = n < kIluReg ? n : kIluReg;
#pragma unroll
        for (int e = 0; e < kIluReg; ++e)
            if (e < cnt) {
                R.c[e] = M.lell_c[e * N + q];
                R.a[e] = M.lell_a[e * N + q];
            }
        R.i = i;
        R.cnt = cnt;
        R.rest = R.end = 0;
        if (n > kIluReg) {
            R.rest = M.rp[i] + kIluReg;
            R.end = M.rp[i] + n;
        }
        R.v = v[i];
    }
    // Row q of U's level order (backward: entries after the diagonal).
    __device__ __forceinline__ void ilu_fetch_u(int64_t q, int64_t hi, IluRow &R) const {
        R.i = -1;
        if (q >= hi) return;
        const IluView<T> &M = sys.ilu;
        const int64_t N = sys.N;
        const int i = M.urows[q];
        const int n = M.ucnt[q];
        const int cnt = n < kIluReg ? n : kIluReg;
#pragma unroll
        for (int e = 0; e < kIluReg; ++e)
            if (e < cnt) {
                R.c[e] = M.uell_c[e * N + q];
                R.a[e] = M.uell_a[e * N + q];
            }
        R.i = i;
        R.cnt = cnt;
        R.rest = R.end = 0;
        if (n > kIluReg) {
            const int64_t d = M.rp[i] + M.dpos[i];
            R.rest = d + 1 + kIluReg;
            R.end = d + 1 + n;
        }
        R.v = M.udiag[q];
    }
    // s - sum of a_e out[c_e] over the row's entries, in pattern order.
    __device__ __forceinline__ T ilu_row_sum(const IluRow &R, T s, const T *out) const {
        const IluView<T> &M = sys.ilu;
#pragma unroll
        for (int e = 0; e < kIluReg; ++e)
            if (e < R.cnt) s = efma(-R.a[e], ldcg_val(out + R.c[e]), s);
        for (int64_t k = R.rest; k < R.end; ++k) s = efma(-M.lu[k], ldcg_val(out + M.ci[k]), s);
        return s;
    }

    // out = M^{-1} v: L z = v by forward substitution (unit diagonal), then
    // U out = z by backward substitution, in place.  Level scheduling: all
    // rows of one level at once over the team's threads, a team barrier
    // between levels.  Each row is one sequential sum in pattern order, as
    // in the definition; U's diagonal divides.  A thread's first row of the
    // next level (index, entries, right-hand side or diagonal) does not
    // depend on the current level, so it is loaded while the barrier is
    // pending, and only the values of earlier levels are read after it.
    __device__ __noinline__ bool ilu_solve(const T *v, T *out) {
        const IluView<T> &M = sys.ilu;
        // a level's positions split into one contiguous chunk per CTA of
        // ceil(size / CTAs): every CTA shares each level (a level is a few
        // thousand scattered rows), and a warp reads consecutive positions
        const int64_t G = gs.nblocks, bid = gs.bid;
        const int tid = threadIdx.x;
        auto chunk = [&](const int32_t *ptr, int l, int64_t &q0, int64_t &q1) {
            const int64_t lo = ptr[l], hi = ptr[l + 1], ch = (hi - lo + G - 1) / G;
            q0 = lo + bid * ch;
            q1 = q0 + ch < hi ? q0 + ch : hi;
        };
        const int nl = M.nlev_l, nu = M.nlev_u;
        int64_t q0, q1;
        IluRow R;
        chunk(M.lptr, 0, q0, q1);
        ilu_fetch_l(q0 + tid, q1, v, R);
        for (int l = 0; l < nl; ++l) {
            if (R.i >= 0) out[R.i] = ilu_row_sum(R, R.v, out);
            for (int64_t q = q0 + tid + kConsumers; q < q1; q += kConsumers) {   // more rows than threads
                const int i = M.lrows[q];
                const int64_t k0 = M.rp[i], kd = k0 + M.dpos[i];
                T t = v[i];
                for (int64_t k = k0; k < kd; ++k) t = efma(-M.lu[k], ldcg_val(out + M.ci[k]), t);
                out[i] = t;
            }
            gs.arrive();
            if (l + 1 < nl) {
                chunk(M.lptr, l + 1, q0, q1);
                ilu_fetch_l(q0 + tid, q1, v, R);
            } else {
                chunk(M.uptr, 0, q0, q1);
                ilu_fetch_u(q0 + tid, q1, R);
            }
            if (!gs.wait()) return false;
        }
        for (int l = 0; l < nu; ++l) {
            if (R.i >= 0) out[R.i] = ilu_row_sum(R, ldcg_val(out + R.i), out) / R.v;
            for (int64_t q = q0 + tid + kConsumers; q < q1; q += kConsumers) {
                const int i = M.urows[q];
                const int64_t kd = M.rp[i] + M.dpos[i], k1 = M.rp[i + 1];
                T t = ldcg_val(out + i);
                for (int64_t k = kd + 1; k < k1; ++k) t = efma(-M.lu[k], ldcg_val(out + M.ci[k]), t);
                out[i] = t / M.lu[kd];
            }
            gs.arrive();
            if (l + 1 < nu) {
                chunk(M.uptr, l + 1, q0, q1);
                ilu_fetch_u(q0 + tid, q1, R);
            }
            if (!gs.wait()) return false;
        }
        if (threadIdx.x == kAcctThread) {   // factors and row data once, v read, out written and re-read
            acct->bytes += M.nnz * (int64_t)(sizeof(T) + 4) + sys.N * (int64_t)(8 + 4 + 8 + 3 * sizeof(T));
            acct->flops += (is_cx<T>::value ? 8 : 2) * M.nnz;
        }
        return true;
    }

    // Before a product pass with ILU(0): t = M^{-1} in, where `in` is the
    // pass's input vector (the pass then multiplies t).  A separate call,
    // so the product passes themselves carry no call to the solve.
    __device__ __forceinline__ bool ilu_pre(const T *in) {
        if constexpr (!PC) {
            return true;
        } else {
            if (!sys.ilu.lu) return true;
            return ilu_solve(in, sys.ilu.t);
        }
    }

    // y_0 = M x_0 = L (U x_0), in place on x: t = U x, then x = L t (two
    // row-parallel products).
    __device__ __noinline__ bool ilu_to_y() {
        const IluView<T> &M = sys.ilu;
        const int64_t nth = (int64_t)gs.nblocks * kConsumers;
        const int64_t me = (int64_t)gs.bid * kConsumers + threadIdx.x;
        T *const x = sys.x, *const t = M.t;
        for (int64_t i = me; i < sys.N; i += nth) {
            const int64_t kd = M.rp[i] + M.dpos[i], k1 = M.rp[i + 1];
            T s{};
            for (int64_t k = kd; k < k1; ++k) s = efma(M.lu[k], x[M.ci[k]], s);
            t[i] = s;
        }
        if (!gs.sync()) return false;
        for (int64_t i = me; i < sys.N; i += nth) {
            const int64_t k0 = M.rp[i], kd = k0 + M.dpos[i];
            T s = ldcg_val(t + i);
            for (int64_t k = k0; k < kd; ++k) s = efma(M.lu[k], ldcg_val(t + M.ci[k]), s);
            x[i] = s;
        }
        return gs.sync();
    }

    // x = M^{-1} y once the final residual pass has formed t = M^{-1} y.
    __device__ __noinline__ bool ilu_to_x() {
        const int64_t nth = (int64_t)gs.nblocks * kConsumers;
        const int64_t me = (int64_t)gs.bid * kConsumers + threadIdx.x;
        T *const x = sys.x;
        const T *t = sys.ilu.t;
        for (int64_t i = me; i < sys.N; i += nth) x[i] = ldcg_val(t + i);
        return gs.sync();
    }

    // ------------------------------------------------------------------
    // passes (sums in gs.red->total)
    // ------------------------------------------------------------------

    // r = b - A x, g_0 = r; sums ||b||^2, ||r||^2, q_1^H r.  The caller has
    // posted kCmdResidual.
    __device__ __noinline__ bool ph_residual(bool write_g0) {
        constexpr int K = 2 + DS;
        ACC acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = ACC(0);
        T *g0 = Gc(0);
        const T *epi[2] = {sys.b, Qc(0)};
        T *const r = sys.r;
        unsigned sq = gs.seq();
        // epilogues capture by value: a captured reference would keep the
        // pointer in memory, reloaded after every store of the loop
        spmv_rows<2>(sys.x, epi, sq, [=](int64_t row, T y, const T (&e)[2], ACC(&a)[K]) {
            T rv = subT(e[0], y);
            r[row] = rv;
            if (write_g0) g0[row] = rv;
            acc_nrm(&a[0], e[0]);
            acc_nrm(&a[1], rv);
            acc_dot(&a[2], e[1], rv);
        }, acc);
        gs.seq() = sq;
        sbytes(write_g0 ? 4 : 3);
        return reduce<K>(acc, true);
    }

    // Refined mode, inner start with x_0 = 0: b = r = g_0 = src * scale
    // (src is the FP64 residual of the outer iteration, rows of this CTA),
    // x = 0; sums ||b||^2, ||r||^2, q_1^H r.  Direct loads (one pass per
    // outer step).
    __device__ __noinline__ bool ph_init_narrow(const typename wide_of<T>::type *src, double scale, double &bb,
                                                double &rr, S &qr) {
        using TW = typename wide_of<T>::type;
        constexpr int K = 2 + DS;
        static_assert(PW * sizeof(TW) == 32, "a chunk of the FP32 vector is two 16-byte source loads");
        const T *q1 = Qc(0);
        T *g0 = Gc(0);
        ACC acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = ACC(0);
        T *const bq = sys.b;
        T *const rq = sys.r;
        T *const xq = sys.x;
        const int64_t clo = c_lo, chi = c_hi;
        {
            for (int64_t ch = clo + threadIdx.x; ch < chi; ch += kConsumers) {
                const uint4 *sp = reinterpret_cast<const uint4 *>(src) + 2 * ch;
                uint4 w2[2] = {sp[0], sp[1]};
                TW tw[PW];
                memcpy(tw, w2, sizeof(tw));
                Pack<T> p, zero;
                Pack<T> qq = ldp_ro(q1, ch);
#pragma unroll
                for (int e = 0; e < PW; ++e) {
                    p.e[e] = narrow_scaled(tw[e], scale);
                    zero.e[e] = T{};
                }
                stp(bq, ch, p);
                stp(rq, ch, p);
                stp(g0, ch, p);
                stp(xq, ch, zero);
#pragma unroll
                for (int e = 0; e < PW; ++e) {
                    acc_nrm(&acc[0], p.e[e]);
                    acc_nrm(&acc[1], p.e[e]);
                    acc_dot(&acc[2], qq.e[e], p.e[e]);
                }
            }
        }
        fence_proxy_async_global();
        double v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = (double)acc[k];
        if (!gs.template reduce<K>(v, true)) return false;
        bb = gs.red->total[0];
        rr = gs.red->total[1];
        qr = mk_coef<T>(gs.red->total + 2);
        if (threadIdx.x == kAcctThread) acct->bytes += sys.N * (int64_t)(sizeof(TW) + 5 * sizeof(T));
        return true;
    }

    // Refined mode, residual replacement: r = src * scale, with src the
    // FP64 true residual b - A x of the outer iteration (rows of this CTA);
    // sums ||r||^2, q_qcol^H r (qcol >= 0) and, when f0, f_1^H r: the
    // inner products the step that follows the replaced update needs.
    // Direct loads.
    __device__ __noinline__ bool ph_replace_narrow(const typename wide_of<T>::type *src, double scale, int qcol,
                                                   bool f0, double &rr, S &qr, S &fr) {
        using TW = typename wide_of<T>::type;
        constexpr int K = 1 + 2 * DS;
        static_assert(PW * sizeof(TW) == 32, "a chunk of the FP32 vector is two 16-byte source loads");
        const T *qv = qcol >= 0 ? Qc(qcol) : nullptr;
        const T *fv = f0 ? Fc(0) : nullptr;
        ACC acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = ACC(0);
        T *const rq = sys.r;
        const int64_t clo = c_lo, chi = c_hi;
        {
            for (int64_t ch = clo + threadIdx.x; ch < chi; ch += kConsumers) {
                const uint4 *sp = reinterpret_cast<const uint4 *>(src) + 2 * ch;
                uint4 w2[2] = {sp[0], sp[1]};
                TW tw[PW];
                memcpy(tw, w2, sizeof(tw));
                Pack<T> p;
#pragma unroll
                for (int e = 0; e < PW; ++e) p.e[e] = narrow_scaled(tw[e], scale);
                stp(rq, ch, p);
#pragma unroll
                for (int e = 0; e < PW; ++e) acc_nrm(&acc[0], p.e[e]);
                if (qv) {
                    Pack<T> qq = ldp_ro(qv, ch);
#pragma unroll
                    for (int e = 0; e < PW; ++e) acc_dot(&acc[1], qq.e[e], p.e[e]);
                }
                if (fv) {
                    Pack<T> ff = ldp_ro(fv, ch);
#pragma unroll
                    for (int e = 0; e < PW; ++e) acc_dot(&acc[1 + DS], ff.e[e], p.e[e]);
                }
            }
        }
        fence_proxy_async_global();
        double v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = (double)acc[k];
        if (!gs.template reduce<K>(v, true)) return false;
        rr = gs.red->total[0];
        qr = mk_coef<T>(gs.red->total + 1);
        fr = mk_coef<T>(gs.red->total + 1 + DS);
        if (threadIdx.x == kAcctThread)
            acct->bytes += sys.N * (int64_t)(sizeof(TW) + (1 + (qv ? 1 : 0) + (fv ? 1 : 0)) * sizeof(T));
        return true;
    }

    // w_i = A g_i; sum q_i^H w.
    __device__ __forceinline__ bool ph_spmv_c(int i, unsigned &sq) {
        ACC acc[DS];
#pragma unroll
        for (int k = 0; k < DS; ++k) acc[k] = ACC(0);
        T *const w = Wc(i);
        const T *epi[1] = {Qc(i)};
        spmv_rows<1>(Gc(i), epi, sq, [=](int64_t row, T y, const T (&e)[1], ACC(&a)[DS]) {
            w[row] = y;
            acc_dot(&a[0], e[0], y);
        }, acc);
        sbytes(1);
        return reduce<DS>(acc, false);
    }

    // z = A u (u held in r); sums z^H z, z^H u.
    __device__ __forceinline__ bool ph_spmv_z(unsigned &sq) {
        constexpr int K = 1 + DS;
        ACC acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = ACC(0);
        const T *epi[1] = {sys.r};
        T *const z = sys.z;
        spmv_rows<1>(sys.r, epi, sq, [=](int64_t row, T y, const T (&e)[1], ACC(&a)[K]) {
            z[row] = y;
            acc_nrm(&a[0], y);
            acc_dot(&a[1], y, e[0]);
        }, acc);
        sbytes(1);
        return reduce<K>(acc, false);
    }

    // x += alpha g_sl, r -= alpha w_sl; sums ||r||^2, q_qcol^H r (hq) and
    // (when f0) f_1^H r.
    __device__ __forceinline__ bool ph_alpha(S alpha, bool hq, bool f0, unsigned &sq) {
        constexpr int K = 1 + 2 * DS;
        const T a = to_t<T>(alpha), na = to_t<T>(-alpha);
        const int ni = 4 + (hq ? 1 : 0) + (f0 ? 1 : 0), iff = hq ? 5 : 4;
        T *const xo = sys.x;
        T *const ro = sys.r;
        const int tc = tile_chunks_for(ni);
        ACC acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = ACC(0);
        tiles(tc, sq, [&](int64_t ch, const unsigned char *st, int k) {
            Pack<T> xx = lds<T>(st, tc, 0, k), gg = lds<T>(st, tc, 1, k), rv = lds<T>(st, tc, 2, k),
                    ww = lds<T>(st, tc, 3, k);
#pragma unroll
            for (int e = 0; e < PW; ++e) {
                xx.e[e] = efma(a, gg.e[e], xx.e[e]);
                rv.e[e] = efma(na, ww.e[e], rv.e[e]);
            }
            stp(xo, ch, xx);
            stp(ro, ch, rv);
#pragma unroll
            for (int e = 0; e < PW; ++e) acc_nrm(&acc[0], rv.e[e]);
            if (hq) {
                Pack<T> qq = lds<T>(st, tc, 4, k);
#pragma unroll
                for (int e = 0; e < PW; ++e) acc_dot(&acc[1], qq.e[e], rv.e[e]);
            }
            if (f0) {
                Pack<T> ff = lds<T>(st, tc, iff, k);
#pragma unroll
                for (int e = 0; e < PW; ++e) acc_dot(&acc[1 + DS], ff.e[e], rv.e[e]);
            }
        });
        vbytes(6 + (hq ? 1 : 0) + (f0 ? 1 : 0));
        if (f0) return reduce<K>(acc, false);
        // without f the sums are ||r||^2 and q^H r, at the block's end (u in
        // r, which the next pass gathers) ||u||^2 alone
        ACC a1[1 + DS];
#pragma unroll
        for (int k = 0; k < 1 + DS; ++k) a1[k] = acc[k];
        if (hq) return reduce<1 + DS>(a1, false);
        ACC a0[1] = {acc[0]};
        return reduce<1>(a0, true);
    }

    // x += omega u, r = u - omega z (u in r); sums ||r||^2, q_1^H r.
    __device__ __forceinline__ bool ph_omega(S omega, unsigned &sq) {
        constexpr int K = 1 + DS;
        const T om = to_t<T>(omega), nom = to_t<T>(-omega);
        T *const xo = sys.x;
        T *const ro = sys.r;
        const int tc = tile_chunks_for(4);
        ACC acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = ACC(0);
        tiles(tc, sq, [&](int64_t ch, const unsigned char *st, int k) {
            Pack<T> xx = lds<T>(st, tc, 0, k), uu = lds<T>(st, tc, 1, k), zz = lds<T>(st, tc, 2, k),
                    qq = lds<T>(st, tc, 3, k);
#pragma unroll
            for (int e = 0; e < PW; ++e) {
                xx.e[e] = efma(om, uu.e[e], xx.e[e]);
                uu.e[e] = efma(nom, zz.e[e], uu.e[e]);
            }
            stp(xo, ch, xx);
            stp(ro, ch, uu);
#pragma unroll
            for (int e = 0; e < PW; ++e) {
                acc_nrm(&acc[0], uu.e[e]);
                acc_dot(&acc[1], qq.e[e], uu.e[e]);
            }
        });
        vbytes(6);
        return reduce<K>(acc, false);
    }

    // z_w = r + bt0 w_i (first) or z_w += bts w_s, in place; sum q^H z_w.
    __device__ __forceinline__ bool ph_w(bool first, S coef, int i, unsigned &sq) {
        const T b = to_t<T>(coef);
        T *const wp = Wc(i);
        const int tc = tile_chunks_for(3);
        ACC acc[DS];
#pragma unroll
        for (int k = 0; k < DS; ++k) acc[k] = ACC(0);
        // inputs: r, w_i, q; or w_i, w_s, q
        const int ia = first ? 1 : 0, io = first ? 0 : 1;
        tiles(tc, sq, [&](int64_t ch, const unsigned char *st, int k) {
            Pack<T> zw = lds<T>(st, tc, ia, k), o = lds<T>(st, tc, io, k), qq = lds<T>(st, tc, 2, k);
            // first: r + b w_i, else w_i + b w_s
#pragma unroll
            for (int e = 0; e < PW; ++e) zw.e[e] = first ? efma(b, zw.e[e], o.e[e]) : efma(b, o.e[e], zw.e[e]);
            stp(wp, ch, zw);
#pragma unroll
            for (int e = 0; e < PW; ++e) acc_dot(&acc[0], qq.e[e], zw.e[e]);
        });
        vbytes(4);
        return reduce<DS>(acc, false);
    }

    // Last pass of the z_w sweep, fused with every deferred g-update of the
    // sweep and the omega-correction:
    //   first=true : z_w = r + bt[sl] w_sl                (empty s-loop)
    //   first=false: z_w += bt[last] w_last
    //   g = bt[sl] g_sl;  g += bt[t] g_t for t = sl+1..n-1;  g = z_w - g/omega
    // sums f_1^H g when with_f.  The first kMaxInputs-4 columns g_t come
    // through the tile pipeline, any further ones by direct loads.
    __device__ __forceinline__ bool ph_w_last(int sl, unsigned &sq) {
        const int n = sys.n;
        const int last = n - 1;
        const bool first = sl == last, with_f = sl > 0;
        T *wp = Wc(sl);
        T *gp = Gc(sl);
        const T bl = to_t<T>(bt[first ? sl : last]);
        const T b0 = to_t<T>(bt[sl]);
        const T nio = to_t<T>(-sc->inv_omega);
        const int t0 = sl + 1;
        const int nt = n - t0;                                     // g_t columns
        const int ntile = nt < kMaxInputs - 4 ? nt : kMaxInputs - 4;
        const int i_t = with_f ? 4 : 3;
        const T *const Gb = sys.G;
        const int64_t ldv = sys.ld;
        const S *const btl = bt;
        const int tc = tile_chunks_for(i_t + ntile);
        ACC acc[DS];
#pragma unroll
        for (int k = 0; k < DS; ++k) acc[k] = ACC(0);
        tiles(tc, sq, [&](int64_t ch, const unsigned char *st, int k) {
            Pack<T> zw = lds<T>(st, tc, 0, k), g = lds<T>(st, tc, 1, k), o = lds<T>(st, tc, 2, k);
            if (first) {
#pragma unroll
                for (int e = 0; e < PW; ++e) zw.e[e] = efma(bl, zw.e[e], o.e[e]);
            } else {
#pragma unroll
                for (int e = 0; e < PW; ++e) zw.e[e] = efma(bl, o.e[e], zw.e[e]);
            }
#pragma unroll
            for (int e = 0; e < PW; ++e) g.e[e] = emul(b0, g.e[e]);
            for (int t = 0; t < nt; ++t) {
                const T bb = to_t<T>(btl[t0 + t]);
                Pack<T> gt = t < ntile ? lds<T>(st, tc, i_t + t, k) : ldp(Gb + (int64_t)(t0 + t) * ldv, ch);
#pragma unroll
                for (int e = 0; e < PW; ++e) g.e[e] = efma(bb, gt.e[e], g.e[e]);
            }
#pragma unroll
            for (int e = 0; e < PW; ++e) g.e[e] = efma(nio, g.e[e], zw.e[e]);
            stp(wp, ch, zw);
            stp(gp, ch, g);
            if (with_f) {
                Pack<T> ff = lds<T>(st, tc, 3, k);
#pragma unroll
                for (int e = 0; e < PW; ++e) acc_dot(&acc[0], ff.e[e], g.e[e]);
            }
        });
        vbytes(5 + nt + (with_f ? 1 : 0));
        if (!with_f) return gs.sync() && ring_ok();   // the next pass gathers g
        return reduce<DS>(acc, false);
    }

    // g_i += beta g_s, or (block 0's first) g_i = r + beta g_0; sums f^H g_i, or, at the sweep's end (the next pass gathers g_i), a team
    // barrier.
    __device__ __forceinline__ bool ph_g(S beta, int i, bool with_f, unsigned &sq) {
        const T bb = to_t<T>(beta);
        T *gp = Gc(i);
        const int tc = tile_chunks_for(with_f ? 3 : 2);
        ACC acc[DS];
#pragma unroll
        for (int k = 0; k < DS; ++k) acc[k] = ACC(0);
        tiles(tc, sq, [&](int64_t ch, const unsigned char *st, int k) {
            Pack<T> g = lds<T>(st, tc, 0, k), g2 = lds<T>(st, tc, 1, k);
#pragma unroll
            for (int e = 0; e < PW; ++e) g.e[e] = efma(bb, g2.e[e], g.e[e]);
            stp(gp, ch, g);
            if (with_f) {
                Pack<T> ff = lds<T>(st, tc, 2, k);
#pragma unroll
                for (int e = 0; e < PW; ++e) acc_dot(&acc[0], ff.e[e], g.e[e]);
            }
        });
        vbytes(with_f ? 4 : 3);
        if (!with_f) return gs.sync() && ring_ok();
        return reduce<DS>(acc, false);
    }

    // ------------------------------------------------------------------
    // one call of the method (Algorithm 7.1, M = I) from the current x
    // ------------------------------------------------------------------
    struct Out {
        int flag;
        int64_t iter;
        int j, i;
        double err;
    };

    __device__ __forceinline__ void record(bool rec, int64_t iter, double err) {
        if (rec && ctl.err_hist && iter < ctl.hist_cap && gs.bid == 0) ctl.err_hist[iter] = err;
    }
    __device__ __forceinline__ S total(int k) const { return mk_coef<T>(gs.red->total + k); }

    // `init` (refined mode only): start from x_0 = 0 with b = init * scale
    // instead of reading b and x.  `hook` (refined mode only, in shared
    // memory): residual replacement by the FP64 outer iteration.
    // hook->replace(qcol, f0, rr, qr, fr, conv) moves the FP32 iterate into
    // the FP64 solution, replaces r by the scaled FP64 true residual and
    // returns ||r||^2 and the inner products of the replaced r that the next
    // step needs, and whether the true residual met the outer tolerance.  It
    // is called when the recursive residual meets `tol` (instead of
    // stopping: the inner call stops only once the true residual has met the
    // outer tolerance) and, at block ends, when hook->want(err) (reliable
    // updates); a block end also ends the call when hook->stalled(iter, err).
    //
    // After inner() returns, x and r are visible to their own CTA only: a
    // team barrier comes before any pass that gathers them.
    template <typename Hook = NoHook>
    __device__ Out inner(int64_t maxit, bool rec, double tol,
                         const typename wide_of<T>::type *init = nullptr, double scale = 1.0,
                         Hook *hook = nullptr) {
        const int n = sys.n;
        const int tid = threadIdx.x;
        rec = rec && ctl.err_hist != nullptr;
        Out o{1, 0, 0, 0, 0.0};
        if (tid == kAcctThread)
            for (int q = 0; q < 5; ++q) acct->ops[q] = 0;

        // r_0 = b - A x_0 (step 2) with the stopping-rule denominator
        bool started = false;
        if constexpr (is_narrow<T>::value) {
            if (init) {
                double bb, rr;
                S e;
                if (!ph_init_narrow(init, scale, bb, rr, e)) return o;
                op(OP_NORM, 2);
                started = true;
            }
        }
        if (!started) {
            if (!ilu_pre(sys.x)) return o;
            gs.post(kCmdResidual);
            if (!ph_residual(true)) return o;
            op(OP_NORM, 2);
            op(OP_MATVEC, 1);
        }
        if (tid == 0) {
            sc->e = total(2);
            const double t0 = sqrt(gs.red->total[0]);
            const double bn = t0 == 0.0 ? 1.0 : t0, rr = gs.red->total[1], e0 = sqrt(rr) / bn;
            sc->bnrm2 = bn;
            sc->rr = rr;
            sc->err = e0;
            // sqrt(rr) / bn < tol is impossible above this (1e-12 covers
            // the roundings; below 1e-290 the exact test decides)
            const double t = tol * bn, f = t * t * (1.0 + 1e-12);
            sc->far = f > 1e-290 ? f : 1e-290;
            sc->iter = 0;
            sc->flag = 1;
            sc->exit = 0;
            sc->j = sc->i = 0;
            sc->act = sc->conv = 0;
            record(rec, 0, e0);
            if (e0 < tol) {
                sc->flag = 0;
                sc->exit = 1;
            }
            if constexpr (Hook::kActive) hook->reset(e0);
        }
        consumer_sync();
        o.err = sc->err;
        if (sc->exit) {
            o.flag = sc->flag;
            return o;
        }
        // the producer's first step is the product w_0 = A g_0
        gs.post(kCmdInner);
        unsigned sq = gs.seq(), passes = 0;
        const unsigned pass0 = gs.ring->passes;

        int j = 0;
        for (Step st;; st.advance(n)) {
            const int i = st.i;
            bool good = true;
            switch (st.op) {
            case P_SPMV_C:
                // steps 31-32, 51 (and w_0 = A g_0): w = A g, c = q_{i+1}^H w
                good = ilu_pre(Gc(i)) && ph_spmv_c(i, sq);
                op(OP_MATVEC);
                op(OP_DOT);
                if (tid == 0) {
                    const S cv = total(0);
                    c[i] = cv;
                    if (is_zero(cv) || !finite_of(cv)) {
                        sc->flag = -1;
                        sc->exit = 1;
                    }
                    sc->coef = sc->e / cv;
                }
                break;
            case P_ALPHA: {
                // steps 5-8: alpha, x, r, e (and f_1^H r in block 0); steps
                // 34-36 at the block's end (u kept in r)
                const bool hq = i < n, f0 = st.first && hq;
                // the inner product of c_0 belongs to the first block's start
                if (st.first && i == 1) op(OP_DOT);
                good = ph_alpha(sc->coef, hq, f0, sq);
                op(OP_SAXPY, 2);
                op(OP_NORM);
                if (tid == kErrThread) {
                    sc->j = j;
                    sc->i = i;
                    residual_norm<Hook>(gs.red->total[0], hq, false, maxit, rec, tol, hook);
                }
                if (hq && tid == 0) alpha_coef(i, f0);
                break;
            }
            case P_SPMV_Z:
                // step 38: omega = (A u)^H u / ||A u||^2, Eq. 5.1 guard
                good = ilu_pre(sys.r) && ph_spmv_z(sq);
                op(OP_MATVEC);
                op(OP_DOT);
                if (tid == 0) {
                    const double zz = gs.red->total[0];
                    const S zu = total(1);
                    const bool bad = zz == 0.0 || !isfinite(zz);
                    S om = zu / zz;
                    if (ctl.kappa > 0.0) {
                        const double arho = abs_of(zu) / (sqrt(zz) * sqrt(sc->rr));
                        if (arho < ctl.kappa && arho != 0.0) om = (ctl.kappa * om) / arho;
                    }
                    if (bad || is_zero(om) || !finite_of(om)) {
                        sc->flag = -1;
                        sc->exit = 1;
                    }
                    sc->act = bad;   // counted below
                    sc->coef = om;
                    sc->omega = om;
                }
                break;
            case P_OMEGA:
                // steps 39-41: x += omega u, r = u - omega A u, e = q_1^H r
                good = ph_omega(sc->coef, sq);
                op(OP_SAXPY, 2);
                op(OP_NORM);
                if (tid == kErrThread) residual_norm<Hook>(gs.red->total[0], true, true, maxit, rec, tol, hook);
                if (tid == 2 * kErrThread) sc->inv_omega = recip(sc->omega);
                if (tid == 0) omega_coef();
                break;
            case P_W_FIRST:
            case P_W_ROUND: {
                // steps 10-17, 42-48: sweep the rest of block j-1 with q's
                const bool wf = st.op == P_W_FIRST;
                if (wf) {
                    op(OP_SAXPY);
                    op(OP_SCALE);
                } else {
                    op(OP_DOT);
                    op(OP_SAXPY, 2);
                }
                good = ph_w(wf, sc->coef, i, sq);
                if (tid == 0) {
                    const int s = wf ? i + 1 : st.s + 1;
                    const S b = -(total(0) / c[s]);
                    bt[s] = b;
                    sc->coef = b;
                }
                break;
            }
            case P_W_LAST:
                if (i == n - 1) {
                    op(OP_SAXPY);
                    op(OP_SCALE);
                } else {
                    op(OP_DOT);
                    op(OP_SAXPY, 2);
                }
                op(OP_SAXPY);   // omega-correction (steps 18, 50)
                good = ph_w_last(i, sq);
                if (i > 0 && tid == 0) sc->coef = -(total(0) / c[0]);
                break;
            default: {   // P_F_ROUND, P_G_J0
                // steps 19-22 (24-28 in block 0): sweep block j with f's
                const int s1 = st.op == P_F_ROUND ? st.s + 1 : 1;
                const bool more = s1 <= i - 1;
                op(OP_DOT);
                op(OP_SAXPY);
                good = ph_g(sc->coef, i, more, sq);
                if (more && tid == 0) sc->coef = -(total(0) / c[s1]);
                break;
            }
            }
            ++passes;
            consumer_sync();
            if (!good) break;
            if (st.op == P_SPMV_Z) {
                if (!sc->act) op(OP_DOT);
                if (!sc->act && ctl.kappa > 0.0) op(OP_NORM, 2);
            }
            if constexpr (Hook::kActive) {
                if (st.op == P_ALPHA || st.op == P_OMEGA) {
                    if (sc->exit) break;
                    const bool hq = st.op == P_OMEGA || i < n;
                    if (sc->act) {
                        const bool f0 = st.op == P_ALPHA && st.first && hq;
                        gs.seq() = sq;
                        double rr;
                        S qr, fr;
                        bool conv;
                        good = hook->replace(st.op == P_OMEGA ? 0 : hq ? i : -1, f0, rr, qr, fr, conv);
                        sq = gs.seq();
                        ++passes;
                        if (!good) break;
                        if (tid == kErrThread) replaced<Hook>(rr, conv, st.op, hq, maxit, hook);
                        if (tid == 0 && hq) {
                            if (st.op == P_OMEGA) omega_coef();
                            else alpha_coef(i, f0);
                        }
                        consumer_sync();
                        if (sc->exit) break;
                    }
                    gs.post(kCmdGo);
                }
            }
            if (sc->exit) break;
            if (st.op == P_ALPHA && i < n) op(OP_DOT);
            if (st.op == P_OMEGA) {
                op(OP_DOT);
                ++j;
            }
        }
        gs.end_inner(sq, pass0 + passes);
        gs.seq() = sq;
        o.flag = gs.ok ? sc->flag : 1;
        o.iter = sc->iter;
        o.j = sc->j;
        o.i = sc->i;
        o.err = sqrt(sc->rr) / sc->bnrm2;
        return o;
    }

    // Thread 0: the coefficient after an update of r within a block
    // (i: the step's slot): e, then beta~ of the sweep with q's (bt[i]) or,
    // in block 0, beta of the one with f's.
    __device__ __forceinline__ void alpha_coef(int i, bool f0) {
        const S e = total(1);
        sc->e = e;
        if (f0) {
            sc->coef = -(total(1 + DS) / c[0]);
        } else {
            const S b = -(e / c[i]);
            bt[i] = b;
            sc->coef = b;
        }
    }
    // Thread 0: the coefficient after the omega step.
    __device__ __forceinline__ void omega_coef() {
        const S e = total(1);
        sc->e = e;
        const S b = -(e / c[0]);
        bt[0] = b;
        sc->coef = b;
    }
    // Thread kErrThread, after an update of r (or of u at the block's end,
    // counts = false): iteration count, stopping rule, iteration limit.
    // The division and the square root of ||r|| / ||b|| are only taken where
    // the value is recorded or can decide.
    template <typename Hook>
    __device__ __forceinline__ void residual_norm(double rr, bool counts, bool block_end, int64_t maxit, bool rec,
                                                  double tol, Hook *hook) {
        sc->rr = rr;
        int64_t iter = sc->iter + (counts ? 1 : 0);
        sc->iter = iter;
        bool conv = false;
        if (Hook::kActive || rec || !(rr > sc->far)) {
            const double err = sqrt(rr) / sc->bnrm2;
            conv = err < tol;
            if constexpr (Hook::kActive) {
                hook->track(err);
                sc->act = conv || (block_end && hook->want(err));
                if (!sc->act) after_norm(err, counts, block_end, maxit, hook);
                return;
            }
            if (conv && !counts) {
                iter++;
                sc->iter = iter;
            }
            if (counts || conv) record(rec, iter, err);
        }
        if (conv) {
            sc->flag = 0;
            sc->exit = 1;
        } else if (counts && iter >= maxit) {
            sc->exit = 1;
        }
    }
    // Refined mode: the tests that follow the (possibly replaced) residual.
    template <typename Hook>
    __device__ __forceinline__ void after_norm(double err, bool counts, bool block_end, int64_t maxit, Hook *hook) {
        if constexpr (Hook::kActive) {
            if (block_end && hook->stalled(sc->iter, err)) sc->exit = 1;
            else if (counts && sc->iter >= maxit) sc->exit = 1;
        }
    }
    template <typename Hook>
    __device__ __forceinline__ void replaced(double rr, bool conv, int op_, bool hq, int64_t maxit, Hook *hook) {
        if constexpr (Hook::kActive) {
            sc->rr = rr;
            const double err = sqrt(rr) / sc->bnrm2;
            hook->reset(err);
            if (conv) {
                if (!hq) sc->iter += 1;   // the converged half step counts
                sc->flag = 0;
                sc->exit = 1;
            } else {
                after_norm(err, hq, op_ == P_OMEGA, maxit, hook);
            }
        }
    }
};

}  // namespace mlb
