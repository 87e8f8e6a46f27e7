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
    // Whether a wait failed: written before the last barrier of a reduction
    // or a team barrier, read after it, so that every consumer takes the same
    // turn.  (The flag of the ring may be set at any time.)  A writer must
    // find every reader of the barrier before gone: team barriers with no
    // other barrier between them alternate between the two.
    int lost[2];
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
// The consumer thread that looks at the ring's mark of failure for all of
// them (in a warp that has no sum to add up).
constexpr int kFoldThread = kConsumers - 32;
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
    double tol;
    int64_t iter, maxit;
    int rec;         // the residual history is recorded
    int block;       // j of the running block (thread kErrThread)
    int exit;        // the iteration ends
    int flag, j, i;  // its result
    int act;         // (refined mode) replace the residual
    int bad;         // ||A u||^2 was zero or not finite
    int conv;        // (refined mode) the true residual met its tolerance
};

// ILU(0) preconditioner M = L U of Algorithm 7.1 (the preconditioner of
// the paper's experiments, §5), stored in A's pattern: in row i, entries
// before the diagonal are L's (unit diagonal implied), the rest U's.  The
// solve iterates on y = M x, with every product A M^{-1} v formed as
// A (M^{-1} v).  Rows are grouped by level for the triangular solves: a
// row of level l depends only on rows of lower levels (of L, or of U taken
// from the last row upwards).  lu == nullptr: no ILU(0) preconditioner.
// A level of the streamed form of the factors (see IluHost::llev): `ns`
// slices of 32 rows, `w` entries wide.
struct IluLevel {
    int64_t e0;   // its first entry
    int32_t m0;   // its first slice
    int32_t ns, w, pad;
};
// Slices per tile of that form: values, columns, (row, count) pairs and U's
// diagonal; 0 when one slice does not fit a stage.
inline int ilu_slices_per_tile(int64_t w, size_t vbytes) {
    const int64_t spt = kStageBytes / (32 * (w * (int64_t)(vbytes + 4) + 8 + (int64_t)vbytes));
    return (int)(spt < kConsumerWarps ? spt : kConsumerWarps);
}

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
    // few levels: the streamed form (else null); lell/uell and udiag then
    // hold its entries
    const IluLevel *llev, *ulev;
    const int2 *lmeta, *umeta;
    int spt;                    // its slices per tile
    // many levels, real values: one slot per row of L (i) and of U (N + i)
    // and, per 32 positions, the row to wait for first (see ilu_flow)
    typename ValueSlot<sizeof(T)>::type *flow;
    const int32_t *lwatch, *uwatch;
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

// The CTA's views, controls and iteration state (see the_ring).
template <typename T>
__device__ __forceinline__ SysView<T> &the_sys() {
    __shared__ SysView<T> v;
    return v;
}
__device__ __forceinline__ SolveCtl &the_ctl() {
    __shared__ SolveCtl c;
    return c;
}
__device__ __forceinline__ Acct &the_acct() {
    __shared__ Acct a;
    return a;
}
template <typename S>
struct IterState {
    S c[kMaxN];
    S bt[kMaxN];
    Scalars<S> sc;
    int s_lo, s_hi;   // slices this CTA owns
};
template <typename S>
__device__ __forceinline__ IterState<S> &the_iter() {
    __shared__ IterState<S> s;
    return s;
}

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
// widths then count blocks.  The first PW entries of a row are pipelined
// (PW registers of gathered x per thread), further ones follow in batches.
// No call here: a call in a kernel's loop costs every pass of the kernel
// registers (saved across it by convention).  Returns false when a tile wait timed out.
//
// sell_consume is the consumer warps' part.  EMPTY: a pass without tiles has
// one empty tile (see consume_empty).
template <int NE, int EW = 1, int PW = 8, bool EMPTY = false, typename T, typename Fin, typename AccArr>
__device__ __forceinline__ bool sell_consume(TileRing *R, unsigned &cseq, int s_lo, int s_hi, int spt,
                                             const int64_t *slice_ptr, const int32_t *scol, const T *sval,
                                             const T *xin, const T *const (&epi)[NE > 0 ? NE : 1], Fin fin,
                                             AccArr &acc) {
    static_assert(EW == 1 || EW == 3, "scalar entries or 3x3 blocks");
    constexpr int kPipeW = PW;
    constexpr int NEA = NE > 0 ? NE : 1;
    const int cw = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (spt <= 0) {
        // slices too wide for one stage: direct loads, no pipeline
        if (EMPTY && !consume_empty(R, cseq)) return false;
        const SliceOffsets off(R, slice_ptr, s_lo, s_hi);
        for (int s = s_lo + cw; s < s_hi; s += kConsumerWarps) {
            const int64_t o = off(s);
            const int w = (int)((off(s + 1) - o) >> 5);
            const int64_t row = (int64_t)s * 32 + lane;
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
    const bool cached = R->soff_src == slice_ptr && R->soff_lo == s_lo && R->soff_hi == s_hi;
    // entries from slice a to slice b of this CTA's range
    auto span = [&](int a, int b) {
        if (cached) return the_soff()[b - s_lo] - the_soff()[a - s_lo];
        return (int)(__ldg(slice_ptr + b) - __ldg(slice_ptr + a));
    };
    auto stage_of = [&](const Job &j) { return the_stages() + j.st * kStageBytes; };
    auto vals = [&](const Job &j) { return reinterpret_cast<const T *>(stage_of(j)) + EW * (j.o + lane); };
    auto cols = [&](const Job &j) {
        return reinterpret_cast<const int32_t *>(stage_of(j) + j.nv * (int)(EW * sizeof(T))) + j.o + lane;
    };
    // epilogue entry i of this warp's row in the tile
    auto epv = [&](const Job &j, int i) {
        return reinterpret_cast<const T *>(stage_of(j) + j.nv * (int)(EW * sizeof(T) + 4))[(i * spt + cw) * 32 + lane];
    };
    // wait for the tile that starts at slice s0 (its number q) and locate
    // this warp's slice in it
    auto locate = [&](int s0, unsigned q, Job &j) -> bool {
        j.st = (int)(q % kStages);
        j.o = j.nv = 0;
        j.w = -1;
        if (!mbar_wait_warp(&R->full[j.st], (q / kStages) & 1u, R->timeout_ns)) return false;
        const int s1 = s0 + spt < s_hi ? s0 + spt : s_hi, s = s0 + cw;
        if (s < s1) {
            j.nv = span(s0, s1);
            j.o = span(s0, s);
            j.w = span(s, s + 1) >> 5;
        }
        return true;
    };
    // Tile jc (its x in xc; its warp's slice s): the FMAs, each followed by
    // the gather of the slice of tile jn (when `more`) into the register it
    // has just read; then the epilogue and the release of the stage.
    // (Gathering two tiles ahead measured slower: 228 against 206 us per
    // iteration at 128^3.)
    auto step = [&](int s, const Job &jc, T (&xc)[kPipeW * EW], const Job &jn, bool more) {
        const T *va = vals(jc);
        const int32_t *cb = cols(jn);
        T sum{};
#pragma unroll
        for (int u = 0; u < kPipeW; ++u) {
            if (u < jc.w) {
#pragma unroll
                for (int q = 0; q < EW; ++q) sum = efma(va[32 * EW * u + q], xc[EW * u + q], sum);
            }
            if (more && u < jn.w) {
                const int32_t c = cb[32 * u];
#pragma unroll
                for (int q = 0; q < EW; ++q) xc[EW * u + q] = xin[c + q];
            }
        }
        constexpr int B = EW == 3 ? 1 : sizeof(T) == 16 ? 2 : 4;   // entries of a wide row at a time
        const int32_t *ca = cols(jc);
        for (int k = kPipeW; k < jc.w; k += B) {
            T xw[B * EW];
#pragma unroll
            for (int u = 0; u < B; ++u)
                if (k + u < jc.w) {
                    const int32_t c = ca[32 * (k + u)];
#pragma unroll
                    for (int q = 0; q < EW; ++q) xw[EW * u + q] = xin[c + q];
                }
#pragma unroll
            for (int u = 0; u < B; ++u)
                if (k + u < jc.w) {
#pragma unroll
                    for (int q = 0; q < EW; ++q) sum = efma(va[32 * EW * (k + u) + q], xw[EW * u + q], sum);
                }
        }
        if (jc.w >= 0) {
            T e[NEA];
#pragma unroll
            for (int i = 0; i < NE; ++i) e[i] = epv(jc, i);
            fin((int64_t)s * 32 + lane, sum, e, acc);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&R->empty[jc.st]);
    };
    bool ok = true;
    unsigned q = cseq;
    if (EMPTY || s_lo < s_hi) {
        Job ja, jb;
        T xv[kPipeW * EW];
        ok = locate(s_lo, q, ja);
        if (ok) {
            const int32_t *cp = cols(ja);
#pragma unroll
            for (int u = 0; u < kPipeW; ++u)
                if (u < ja.w) {
                    const int32_t c = cp[32 * u];
#pragma unroll
                    for (int m = 0; m < EW; ++m) xv[EW * u + m] = xin[c + m];
                }
        }
        for (int s0 = s_lo; ok && (s0 < s_hi || (EMPTY && s0 == s_lo)); s0 += spt) {
            const bool more = s0 + spt < s_hi;
            if (more && !locate(s0 + spt, q + 1, jb)) {
                ok = false;
                break;
            }
            step(s0 + cw, ja, xv, jb, more);
            ++q;
            ja = jb;
        }
    }
    cseq = q;
    fence_proxy_async_global();
    return ok;
}

// Producer and consumers of one product in one call (the fused product's
// kernel): pseq is the producer lane's tile counter, cseq a consumer's.
template <int NE, int EW = 1, int PW = 8, typename T, typename Fin, typename AccArr>
__device__ __forceinline__ bool sell_spmv(TileRing *R, unsigned &pseq, unsigned &cseq, int s_lo, int s_hi, int spt,
                                          const int64_t *slice_ptr, const int32_t *scol, const T *sval,
                                          const T *xin, const T *const (&epi)[NE > 0 ? NE : 1], Fin fin,
                                          AccArr &acc) {
    constexpr int NEA = NE > 0 ? NE : 1;
    if ((threadIdx.x >> 5) == kConsumerWarps) {
        if ((threadIdx.x & 31) != 0 || spt <= 0) return true;
        const SliceOffsets off(R, slice_ptr, s_lo, s_hi);
        const void *ep[NEA];
#pragma unroll
        for (int i = 0; i < NE; ++i) ep[i] = epi[i];
        return produce_sell(R, s_lo, s_hi, spt, off, sval, EW * (int)sizeof(T), (int)sizeof(T), scol, ep, NE, pseq);
    }
    return sell_consume<NE, EW, PW>(R, cseq, s_lo, s_hi, spt, slice_ptr, scol, sval, xin, epi, fin, acc);
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

__device__ __forceinline__ RedScratch &the_red() {
    __shared__ RedScratch r;
    return r;
}

// A tile wait of this warp failed: its tile counter is no longer that of the
// next pass, which therefore must not begin.  The reduction or the team
// barrier (of that turn) that ends the pass reports it.
__device__ __forceinline__ void tile_lost(int turn = 0) {
    the_ring()->failed = 1;
    the_red().lost[turn & 1] = 1;
}

// Synchronisation state of one CTA within the team of CTAs that solves one
// system: the whole grid (a single solve), a group of CTAs of a batch
// launch (a large system of a batch), or the CTA alone (the other systems
// of a batch).  Every CTA of a team passes the same sequence of
// barriers and reductions, so the epochs advance in lock step.
// The engines of one kernel share one GridSync (the_gs).  Its members are called
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
    uint64_t timeout_ns;
    unsigned epoch;     // exchanges this CTA has passed
    unsigned bepoch;    // barriers (sync) this CTA has passed
    unsigned fepoch;    // triangular solve pairs (Engine::ilu_flow) this CTA has passed
    bool ok;            // false once a barrier or a tile wait failed
    unsigned seqs[kThreads];   // per-thread tile counters, kept across systems

    __device__ __forceinline__ unsigned &seq() { return seqs[threadIdx.x]; }

    // Team of `nb` CTAs (rank `id`) with their own barrier state and slots;
    // nb = 1: this CTA alone (b and p null).  One thread.
    __device__ __forceinline__ void init(BarrierState *b, Slot *p, unsigned nb, unsigned id, uint64_t to) {
        nblocks = nb;
        bid = id;
        bar = b;
        slots = p;
        timeout_ns = to;
        epoch = bepoch = fepoch = 0;
        ok = !the_ring()->failed;
        the_ring()->timeout_ns = to;
        the_red().lost[0] = the_red().lost[1] = 0;
    }

    // Slots of sum k of the exchange `ep`.  Two halves suffice: a CTA
    // puts exchange ep + 2 only after it has seen every slot of ep + 1,
    // which a CTA puts after it has read every slot of ep.
    __device__ __forceinline__ Slot *slot_of(unsigned ep, int k) const {
        return slots + ((size_t)(ep & 1u) * kMaxSums + k) * nblocks;
    }

    // The last levels of reduce(), by one warp; false (uniformly in the warp)
    // when the wait failed.
    __device__ __forceinline__ bool team_total(int k, bool fence) {
        const int lane = threadIdx.x & 31;
        const double *p = the_red().part[k] + lane;
        double t = p[0] + p[32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        bool got = true;
        if (nblocks > 1) {
            const unsigned ep = epoch + 1;
            Slot *const q = slot_of(ep, k);
            if (lane == 0) {
                if (fence) fence_acq_rel_gpu();   // this CTA's writes before its slot
                slot_put(q + bid, t, ep);
            }
            got = slots_sum(q, nblocks, ep, bar, timeout_ns, t);
            if (fence) fence_acq_rel_gpu();       // the other CTAs' writes after their slots
        }
        if (lane == 0) the_red().total[k] = t;
        return got;
    }

    // Sum K values over the team into the_red().total[0, K), the same bits in
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
    // their own CTA's rows only).  False (uniformly) when a wait failed, here
    // or at a tile of the ring.
    __device__ __forceinline__ bool reduce_k(const double (&v)[kMaxSums], int K, bool fence) {
        static_assert(kMaxSums <= kConsumerWarps && kConsumers == 480, "reduction layout");
        constexpr int G1 = 64;
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
        for (int k = 0; k < kMaxSums; ++k) {
            if (k < K) {
                const double h = v[k] + __shfl_down_sync(0xffffffffu, v[k], 16);
                if (lane < 16) the_red().part[k][warp * 16 + lane] = h;
            }
        }
        consumer_sync();
        if (tid < K * G1) {
            double *p = the_red().part[tid / G1] + tid % G1;
            const double a0 = p[0], a1 = p[G1], a2 = p[2 * G1];
            // the last group has 48 partials
            p[0] = (a0 + a1) + (tid % G1 < 48 ? a2 + p[3 * G1] : a2);   // only this task reads slot 0
        }
        consumer_sync();
        if (warp < K && !team_total(warp, fence)) the_red().lost[0] = 1;
        if (tid == kFoldThread && the_ring()->failed) the_red().lost[0] = 1;
        consumer_sync();
        if (tid == 0) epoch += 1;   // read again only after another barrier
        if (the_red().lost[0]) { ok = false; return false; }
        return true;
    }
    // The same for the passes outside the iteration (one copy of the code).
    __device__ __noinline__ bool reduce_ool(double v0, double v1, double v2, double v3, double v4, int K, bool fence) {
        const double v[kMaxSums] = {v0, v1, v2, v3, v4};
        return reduce_k(v, K, fence);
    }
    template <int K>
    __device__ __forceinline__ bool reduce(const double (&v)[K], bool fence) {
        static_assert(K <= kMaxSums && kMaxSums == 5, "sums of a pass");
        return reduce_ool(v[0], v[K > 1 ? 1 : 0], v[K > 2 ? 2 : 0], v[K > 3 ? 3 : 0], v[K > 4 ? 4 : 0], K, fence);
    }

    // Team barrier (a counter: cheaper than an exchange where no value goes
    // with it).
    // turn: see RedScratch::lost.
    __device__ __forceinline__ bool sync(int turn = 0) {
        arrive();
        return wait(turn);
    }

    // sync() in two halves: arrive() once this CTA's writes are done,
    // wait() before reading other CTAs' writes; work between the two that
    // reads nothing written in this step overlaps the wait.  wait() returns
    // false (uniformly) when a wait of the consumers failed (the producer's
    // own is seen by the next reduction, or starves them of tiles).  A CTA
    // alone needs arrive()'s barrier only.
    __device__ __forceinline__ void arrive() {
        consumer_sync();
        if (nblocks > 1 && threadIdx.x == 0) grid_arrive(bar, bepoch);
    }
    __device__ __forceinline__ bool wait(int turn) {
        if (nblocks > 1) {
            if (threadIdx.x == 0 && !grid_wait(bar, bepoch, nblocks, timeout_ns)) the_red().lost[turn & 1] = 1;
            consumer_sync();
        }
        if (the_red().lost[turn & 1]) { ok = false; return false; }
        return true;
    }

    // Hand a command to the producer warp (every consumer thread calls it).
    // Stop and exit also call it out of its waits.  The last command and the
    // call that came with it are only replaced once the producer has taken
    // them.
    __device__ __forceinline__ void post(unsigned cmd) {
        if (threadIdx.x == 0) {
            await_taken(the_ring());
            the_ring()->cmd = cmd;
            *(volatile int *)&the_ring()->stop = cmd == kCmdStop || cmd == kCmdExit;
        }
        __syncthreads();
    }
    // End of an iteration (kCmdStop) or of a system (kCmdExit): stop the
    // producer, and discard the tiles it has issued that no pass has consumed
    // (their stages are released as if consumed).  What follows, the next
    // system of a batch too, finds both sides at the same tile.
    __device__ __forceinline__ void end(unsigned cmd, unsigned &sq) {
        post(cmd);
        for (const unsigned last = the_ring()->issued; sq != last; ++sq) {
            if (!mbar_wait_warp(&the_ring()->full[sq % kStages], (sq / kStages) & 1u, kOwnNs)) {
                the_ring()->failed = 1;
                ok = false;
                break;
            }
            __syncwarp();
            if ((threadIdx.x & 31) == 0) mbar_arrive(&the_ring()->empty[sq % kStages]);
        }
        consumer_sync();
    }
    __device__ __forceinline__ void end_system() {
        unsigned sq = seq();
        end(kCmdExit, sq);
        seq() = sq;
    }
};

__device__ __forceinline__ GridSync &the_gs() {
    __shared__ GridSync g;
    return g;
}

// One pass of the iteration (Engine::inner) and the pass after it: a
// function of n alone, which the producer warp follows too.  i: the slot the
// step builds (ALPHA uses slot i - 1; i = n: the block's last update); s:
// the column a sweep's pass uses; first: block 0.
enum { P_RESIDUAL, P_SPMV_C, P_ALPHA, P_SPMV_Z, P_OMEGA, P_W_FIRST, P_W_ROUND, P_W_LAST, P_F_ROUND, P_G_J0 };
struct Step {
    int op = P_SPMV_C, i = 0, s = 0;
    bool first = true;
    __device__ __forceinline__ void advance(int n) {
        switch (op) {
        case P_RESIDUAL: op = P_SPMV_C; break;
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

// PC: the forms of the ILU(0) preconditioner passes that the engine is built
// with: none, streamed (ilu_wide), by slots (ilu_flow, single solves of real
// systems), a barrier per level (ilu_levels), or, for a batch whose systems
// differ in it, ilu_wide and ilu_levels.  What is not built in takes no
// registers from the kernel's
// loop: with two forms in one kernel the FP64 one spilled 276 bytes a thread,
// with the streamed form alone 120 (multicolour ILU(0) at 96^3: 31.0 -> 30.0
// ms, refined 3x3-block system 2840 -> 2480 us).
// EW: the matrix storage of the products (1:
// scalar SELL-32; 3: 3x3 blocks, see sell_slice_sum3).
//
// The consumer threads run inner() and the other members; the producer warp
// runs serve() beside them.
enum { kNoIlu, kIluWide, kIluFlow, kIluLevels, kIluAny };
template <typename T, int PC = kNoIlu, int EW = 1>
struct Engine {
    using S = typename coef_of<T>::type;                      // FP64 coefficient
    using ACC = typename real_of<T>::type;                    // thread accumulator
    static constexpr int DS = dslots<T>();
    static constexpr int PW = Pack<T>::W;
    static constexpr int CPS = 32 * sizeof(T) / 16;           // 16-byte chunks per slice

    // The CTA's shared objects; the engine has no state of its own.
    __device__ __forceinline__ static const SysView<T> &sys() { return the_sys<T>(); }
    __device__ __forceinline__ static const SolveCtl &ctl() { return the_ctl(); }
    __device__ __forceinline__ static GridSync &gs() { return the_gs(); }
    __device__ __forceinline__ static Acct &acct() { return the_acct(); }
    __device__ __forceinline__ static Scalars<S> &sc() { return the_iter<S>().sc; }
    __device__ __forceinline__ static S *c() { return the_iter<S>().c; }
    __device__ __forceinline__ static S *bt() { return the_iter<S>().bt; }
    // ownership: slices [s_lo(), s_hi()), chunks [c_lo(), c_hi())
    __device__ __forceinline__ static int s_lo() { return the_iter<S>().s_lo; }
    __device__ __forceinline__ static int s_hi() { return the_iter<S>().s_hi; }
    __device__ __forceinline__ static int64_t c_lo() { return (int64_t)s_lo() * CPS; }
    __device__ __forceinline__ static int64_t c_hi() { return (int64_t)s_hi() * CPS; }

    // Every thread, once the system's view and the team are set.
    __device__ void attach() {
        if (threadIdx.x == 0) {
            int64_t lo, hi;
            own_range(sys().nslices, gs().nblocks, gs().bid, lo, hi);
            the_iter<S>().s_lo = (int)lo;
            the_iter<S>().s_hi = (int)hi;
            the_ring()->stop = 0;
        }
        __syncthreads();
        soff_load(the_ring(), sys().slice_ptr, s_lo(), s_hi());
    }
    // Counts one Table 4.3 operation and its algorithmic floating-point
    // operations (real arithmetic): a product 2 per stored entry; an inner
    // product, AXPY or norm 2 per element; a scaling 1 per element.
    // Complex values: a multiply-add is 8 real operations, |v|^2 4, a
    // scaling 6.
    __device__ __forceinline__ void op(int which, int cnt = 1) {
        if (threadIdx.x == kAcctThread) {
            acct().ops[which] += cnt;
            constexpr bool cx_ = is_cx<T>::value;
            const int64_t N = sys().N;
            int64_t f;
            if (which == OP_MATVEC) f = (cx_ ? 8 : 2) * sys().nnz;
            else if (which == OP_SCALE) f = (cx_ ? 6 : 1) * N;
            else if (which == OP_NORM) f = (cx_ ? 4 : 2) * N;
            else f = (cx_ ? 8 : 2) * N;
            acct().flops += cnt * f;
        }
    }

    __device__ __forceinline__ const T *Qc(int k) const { return sys().Q + (int64_t)k * sys().ld; }
    __device__ __forceinline__ const T *Fc(int k) const { return sys().F + (int64_t)k * sys().ld; }
    __device__ __forceinline__ T *Gc(int k) const { return sys().G + (int64_t)k * sys().ld; }
    __device__ __forceinline__ T *Wc(int k) const { return sys().W + (int64_t)k * sys().ld; }

    __device__ __forceinline__ void vbytes(int nvec) {
        if (threadIdx.x == kAcctThread) acct().bytes += nvec * sys().N * (int64_t)sizeof(T);
    }
    __device__ __forceinline__ void sbytes(int nextra) {
        // SpMV: entries (values, and a column index per stored entry of EW
        // values), row_ptr-equivalent, x read once, y written once, plus
        // `nextra` epilogue vectors.
        if (threadIdx.x == kAcctThread) {
            acct().bytes += sys().nnz * (int64_t)sizeof(T) + sys().nnz / EW * 4 + 4 * (sys().N + 1) +
                           (2 + nextra) * sys().N * (int64_t)sizeof(T);
            acct().spmv++;
        }
    }

    // ------------------------------------------------------------------
    // the producer warp
    // ------------------------------------------------------------------

    // Issue the tiles of pass `st` (the input order of each pass is that of
    // its consumer side below).
    __device__ __forceinline__ int issue(const Step &st, unsigned &sq) {
        const int lane = threadIdx.x & 31, n = sys().n, i = st.i, s = st.s;
        TileRing *const R = the_ring();
        const T *p = nullptr;
        int ni = 0;
        switch (st.op) {
        case P_SPMV_C:
        case P_SPMV_Z: {
            const int e = issue_ilu(sq);
            return e ? e : issue_product(st.op == P_SPMV_C ? Qc(i) : sys().r, sys().spt[1], sq);
        }
        case P_ALPHA: {
            const bool hq = i < n, f0 = st.first && hq;
            ni = 4 + (hq ? 1 : 0) + (f0 ? 1 : 0);
            p = lane == 0 ? sys().x : lane == 1 ? Gc(i - 1) : lane == 2 ? sys().r : lane == 3 ? Wc(i - 1)
                : lane == 4 && hq ? Qc(i) : sys().F;
            break;
        }
        case P_OMEGA:
            ni = 4;
            p = lane == 0 ? sys().x : lane == 1 ? sys().r : lane == 2 ? sys().z : sys().Q;
            break;
        case P_W_FIRST:
            ni = 3;
            p = lane == 0 ? sys().r : lane == 1 ? Wc(i) : Qc(i + 1);
            break;
        case P_W_ROUND:
            ni = 3;
            p = lane == 0 ? Wc(i) : lane == 1 ? Wc(s) : Qc(s + 1);
            break;
        case P_W_LAST: {
            const int nt = n - 1 - i, ntile = nt < kMaxInputs - 4 ? nt : kMaxInputs - 4, f = i > 0 ? 1 : 0;
            ni = 3 + f + ntile;
            p = lane == 0 ? Wc(i) : lane == 1 ? Gc(i) : lane == 2 ? (i == n - 1 ? sys().r : Wc(n - 1))
                : lane == 3 && f ? sys().F : Gc(i + 1 + lane - 3 - f);
            break;
        }
        case P_F_ROUND:
            ni = s + 1 <= i - 1 ? 3 : 2;
            p = lane == 0 ? Gc(i) : lane == 1 ? Gc(s) : Fc(s + 1);
            break;
        default:   // P_G_J0
            ni = i >= 2 ? 3 : 2;
            p = lane == 0 ? sys().r : lane == 1 ? sys().G : Fc(1);
            break;
        }
        return produce_lanes(R, p, ni, c_lo(), c_hi(), sq);
    }
    // Tiles of a product with one epilogue vector, `spt` slices each.
    __device__ __forceinline__ int issue_product(const T *epi, int spt, unsigned &sq) {
        const SliceOffsets off(the_ring(), sys().slice_ptr, s_lo(), s_hi());
        return produce_sell_lanes(the_ring(), s_lo(), s_hi(), spt, off, sys().sval, EW * (int)sizeof(T),
                                  (int)sizeof(T), sys().scol, epi, 1, sq);
    }
    // Wait until the consumers have finished the pass.
    __device__ __forceinline__ int wait_done(unsigned &passes, bool limited) {
        int st = 0;
        if ((threadIdx.x & 31) == 0) st = producer_wait(the_ring(), &the_ring()->done, passes & 1u, limited);
        st = __shfl_sync(0xffffffffu, st, 0);
        if (st == 0) passes += 1;
        return st;
    }
    // Meet the consumers: their next command.  `sq`: tiles issued so far.
    __device__ __forceinline__ unsigned command(unsigned sq, unsigned &passes) {
        TileRing *const R = the_ring();
        if ((threadIdx.x & 31) == 0) R->issued = sq;
        __syncthreads();
        const unsigned cmd = *(volatile unsigned *)&R->cmd;
        if (cmd == kCmdStop) {
            // the consumers may have finished the pass that this side was
            // waiting for or issuing
            if (mbar_probe(&R->done, passes & 1u)) passes += 1;
        }
        __syncwarp();
        if ((threadIdx.x & 31) == 0) *(volatile unsigned *)&R->cmd = kCmdNone;
        return cmd;
    }
    // The producer warp's side of a system: commands of the consumers until
    // kCmdExit.  Decide: the iteration asks the consumers after every update
    // of r (refined mode).  residual64 issues the FP64 residual's tiles.
    // After a timeout it only takes commands: the consumers find the ring
    // marked as failed and end the solve.
    template <bool Decide, typename Fn>
    __device__ __forceinline__ void serve(Fn residual64) {
        TileRing *const R = the_ring();
        unsigned sq = gs().seq(), passes = R->passes;
        bool dead = false;
        for (;;) {
            const unsigned cmd = command(sq, passes);
            if (cmd == kCmdExit) break;
            if (dead || cmd == kCmdStop) continue;
            int st = 0;
            if (cmd == kCmdResidual) {
                st = issue_ilu(sq);
                if (st == 0) st = issue_product(sys().b, sys().spt[2], sq);
                if (st == 0) st = wait_done(passes, false);
            } else if (cmd == kCmdResidual64) {
                st = residual64(sq);
                if (st == 0) st = wait_done(passes, false);
            } else if (cmd == kCmdIlu) {
                st = issue_ilu(sq);
            } else {
                const int n = sys().n;
                bool over = false;   // ended by a command
                for (Step p; st == 0 && !over; p.advance(n)) {
                    st = issue(p, sq);
                    if (st == 0) st = wait_done(passes, p.op != P_SPMV_C && p.op != P_SPMV_Z);
                    if constexpr (Decide) {
                        // the consumers' commands (a residual replacement)
                        // until they let the iteration go on or end it
                        while (st == 0 && (p.op == P_ALPHA || p.op == P_OMEGA)) {
                            const unsigned c = command(sq, passes);
                            over = c == kCmdStop;
                            if (over || c == kCmdGo) break;
                            if (c == kCmdIlu) {
                                st = issue_ilu(sq);
                            } else {
                                st = residual64(sq);
                                if (st == 0) st = wait_done(passes, false);
                            }
                        }
                    }
                }
            }
            if (st == 2) {
                R->failed = 1;
                dead = true;
            }
        }
        gs().seq() = sq;
        if ((threadIdx.x & 31) == 0) R->passes = passes;
    }

    // ------------------------------------------------------------------
    // the consumers' side of the passes
    // ------------------------------------------------------------------

    // Streaming pass through the tile pipeline: fn(chunk, stage, k) for
    // every chunk of this CTA.
    template <typename Fn>
    __device__ __forceinline__ void tiles(int tc, unsigned &sq, Fn fn) {
        TileRing *const ring = the_ring();
        if (!consume<true>(ring, TileGeom{tc, c_lo(), c_hi()}, sq, fn)) tile_lost();
        pass_done(ring);
    }

    // SELL-32 SpMV pass over the owned slices (matrix tiles through the
    // ring).
    template <typename Fin, int K>
    __device__ __forceinline__ void spmv_rows(const T *xin, const T *const (&epi)[1], int spt, unsigned &sq, Fin fin,
                                              ACC (&acc)[K]) {
        // with ILU(0) the product is A t, t = M^{-1} xin formed before the
        // pass
        if constexpr (PC != kNoIlu) {
            if (sys().ilu.lu) xin = sys().ilu.t;
        }
        // pipelined entries: what the registers hold.  FP32 engines 7, the
        // widest row of the 3-D stencils, 4 with both forms of ILU(0); the real
        // FP64 engine 8 (no gain at 7); the complex FP64 engine 3 (with 7
        // gathered values of 16 bytes the loop spilled: batch of 96 small
        // systems 4.71 -> 4.33 ms, 4.55 before the passes shared one loop;
        // 128x128x32, 16 iterations, 3.05 -> 2.83 ms)
        constexpr int W = sizeof(T) == 16 ? 3 : is_narrow<T>::value ? (PC == kIluAny ? 4 : 7) : 8;
        const bool okw = sell_consume<1, EW, W, true>(the_ring(), sq, s_lo(), s_hi(), spt, sys().slice_ptr,
                                                      sys().scol, sys().sval, xin, epi, fin, acc);
        if (!okw) tile_lost();
        pass_done(the_ring());
    }

    // ------------------------------------------------------------------
    // ILU(0) preconditioner (Algorithm 7.1 with M = L U)
    // ------------------------------------------------------------------

    // One row of a triangular solve, loaded ahead: its index, up to
    // kIluReg entries (column, factor value) in registers, where the rest
    // of its entries start and end, and the row's right-hand-side entry
    // (forward) or its U diagonal (backward).  i < 0: no row.
    static constexpr bool kFlow = PC == kIluFlow;   // real values only
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
        const IluView<T> &M = sys().ilu;
        const int64_t N = sys().N;
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
        const IluView<T> &M = sys().ilu;
        const int64_t N = sys().N;
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
        const IluView<T> &M = sys().ilu;
#pragma unroll
        for (int e = 0; e < kIluReg; ++e)
            if (e < R.cnt) s = efma(-R.a[e], ldcg_val(out + R.c[e]), s);
        for (int64_t k = R.rest; k < R.end; ++k) s = efma(-M.lu[k], ldcg_val(out + M.ci[k]), s);
        return s;
    }

    // out = M^{-1} v by a team without a barrier between levels: a row's value
    // goes to its slot with the number of this M^{-1}, and a row takes the
    // values it needs from their slots as they arrive.  Warps take 32
    // positions of the level order at a time, L's and then U's, dealt over
    // the CTAs; a row only waits for rows at earlier positions, and a warp
    // takes its positions in increasing order, so the first unfinished
    // position never waits.  A warp first watches one row two levels back,
    // so the warps that poll all their rows' slots are those of the next two
    // levels.  Each row is one sequential sum in pattern order.
    // What bounds it: the chain of levels, each a slot put, its way through
    // L2 to a poll, the row's sum and (U) a division.  us a level, FP64, with
    // barriers (ilu_levels) -> here: 200^2 2.4 -> 1.3, 40^3 2.5 -> 1.7, 48^3 2.5
    // -> 1.7, 96^3 2.9 -> 2.3; 3x3-block system of 393,216 rows, about ten
    // entries a triangle and row: 76 -> 55 ms a solve.
    __device__ __forceinline__ bool ilu_flow(const T *v, T *out) {
        if constexpr (kFlow) {
            const IluView<T> &M = sys().ilu;
            const int lane = threadIdx.x & 31, cw = threadIdx.x >> 5;
            const unsigned ep = gs().fepoch + 1;
            const int64_t N = sys().N, nch = (N + 31) / 32, G = gs().nblocks;
            using VS = typename ValueSlot<sizeof(T)>::type;
            VS *const zl = M.flow, *const zu = zl + N;
            BarrierState *const bar = gs().bar;
            const uint64_t limit = gs().timeout_ns;
            // progress is told seldom: a store per 32 rows to the word that every
            // waiting warp reads doubled the time of a solve
            uint64_t told = globaltimer_ns();
            bool ok = true;
            for (int64_t k = gs().bid + G * cw; ok && k < 2 * nch; k += G * kConsumerWarps) {
                const bool up = k >= nch;
                const int64_t ch = up ? k - nch : k, q = 32 * ch + lane;
                VS *const z = up ? zu : zl;
                const int w = up ? M.uwatch[ch] : M.lwatch[ch];
                // this lane's row i: n entries, the first ones in c and a, and
                // the right-hand side (L) or U's diagonal
                int i = -1, n = 0;
                int64_t p = 0;          // a longer row's entries in the pattern
                int32_t c[kIluReg];
                T a[kIluReg], d{};
                if (q < N) {
                    i = up ? M.urows[q] : M.lrows[q];
                    n = up ? M.ucnt[q] : M.lcnt[q];
                    const int32_t *const pc = (up ? M.uell_c : M.lell_c) + q;
                    const T *const pa = (up ? M.uell_a : M.lell_a) + q;
#pragma unroll
                    for (int u = 0; u < kIluReg; ++u)
                        if (u < n) {
                            c[u] = pc[u * N];
                            a[u] = pa[u * N];
                        }
                    d = up ? M.udiag[q] : v[i];
                    if (n > kIluReg) p = M.rp[i] + (up ? M.dpos[i] + 1 : 0);
                }
                const VS *const watch = w >= 0 ? z + w : up ? zl + ~w : nullptr;
                SlotWait patience;
                T xv;
                while (ok && watch && !__all_sync(0xffffffffu, value_of(value_load(watch), ep, xv))) ok = patience.go_on(bar, limit);
                int e = up ? -1 : 0;    // next entry; -1: the right-hand side
                int e0 = 0;             // the entry in c[0] and a[0]
                T s = d;
                bool done = i < 0;
                while (ok && !__all_sync(0xffffffffu, done)) {
                    if (!done) {
                        VS r{}, x[kIluReg];
                        if (e < 0) r = value_load(zl + i);
#pragma unroll
                        for (int u = 0; u < kIluReg; ++u)
                            if (e0 + u >= e && e0 + u < n) x[u] = value_load(z + c[u]);
                        if (e < 0 && value_of(r, ep, xv)) {
                            s = xv;
                            e = 0;
                        }
#pragma unroll
                        for (int u = 0; u < kIluReg; ++u)
                            if (e0 + u == e && e < n && value_of(x[u], ep, xv)) {
                                s = efma(-a[u], xv, s);
                                e = e0 + u + 1;
                            }
                        if (e == e0 + kIluReg && e < n) {   // the next entries, from the pattern
                            e0 = e;
#pragma unroll
                            for (int u = 0; u < kIluReg; ++u)
                                if (e + u < n) {
                                    c[u] = M.ci[p + e + u];
                                    a[u] = M.lu[p + e + u];
                                }
                        }
                        if (e == n) {
                            if (up) {
                                s = s / d;
                                out[i] = s;
                            }
                            value_put(z + i, s, ep);
                            done = true;
                        }
                    }
                    if (!__all_sync(0xffffffffu, done)) ok = patience.go_on(bar, limit);
                }
                if (lane == 0) {
                    const uint64_t now = globaltimer_ns();
                    if (now - told > limit / 8) {
                        st_relaxed_u32(&bar->progress, (unsigned)k + 1u);
                        told = now;
                    }
                }
            }
            if (!ok) the_red().lost[1] = 1;
            const bool good = gs().sync(1);
            if (threadIdx.x == 0) gs().fepoch = ep;   // read again only after another barrier
            ilu_count();
            return good;
        } else {
            return false;
        }
    }
    // Start of a solve: no slot holds a value yet.
    __device__ __forceinline__ bool ilu_begin() {
        if constexpr (kFlow) {
            using VS = typename ValueSlot<sizeof(T)>::type;
            VS *const z = sys().ilu.flow;
            const int64_t nth = (int64_t)gs().nblocks * kConsumers;
            for (int64_t i = (int64_t)gs().bid * kConsumers + threadIdx.x; i < 2 * sys().N; i += nth)
                z[i] = VS{};
            return gs().sync();
        } else {
            return true;
        }
    }

    __device__ __noinline__ bool ilu_flow_ool(const T *v, T *out) { return ilu_flow(v, out); }
    __device__ __noinline__ bool ilu_wide_ool(const T *v, T *out) { return ilu_wide(v, out); }
    __device__ __noinline__ bool ilu_levels_ool(const T *v, T *out) { return ilu_levels(v, out); }
    // out = M^{-1} v.  In FP32 a function of its own where the loop of the
    // refined kernels, which holds more than the FP64 one, crowds its polls
    // or both forms out of the registers: by slots with scalar storage (24
    // iterations, ms: 48^3 16.9 -> 13.0, 96^3 n = 8 40.4 -> 34.3, 27-point 40^3
    // 90.5 -> 55.8; 3x3 blocks 44.9 -> 46.2, FP64 no change: inlined), and a
    // batch that mixes the forms (192 systems 40.0 -> 38.2; FP64 39.8 -> 40.7).
    __device__ __forceinline__ bool ilu_solve_body(const T *v, T *out) {
        if constexpr (PC == kIluWide) return ilu_wide(v, out);
        else if constexpr (PC == kIluFlow && is_narrow<T>::value && EW == 1) return ilu_flow_ool(v, out);
        else if constexpr (PC == kIluFlow) return ilu_flow(v, out);
        else if constexpr (PC == kIluLevels) return ilu_levels(v, out);
        else if constexpr (is_narrow<T>::value)
            return sys().ilu.llev ? ilu_wide_ool(v, out) : ilu_levels_ool(v, out);
        else return sys().ilu.llev ? ilu_wide(v, out) : ilu_levels(v, out);
    }
    // out = M^{-1} v: L z = v by forward substitution (unit diagonal), then
    // U out = z by backward substitution, in place.  Level scheduling: all
    // rows of one level at once over the team's threads, a team barrier
    // between levels.  Each row is one sequential sum in pattern order, as
    // in the definition; U's diagonal divides.  A thread's first row of the
    // next level (index, entries, right-hand side or diagonal) does not
    // depend on the current level, so it is loaded while the barrier is
    // pending, and only the values of earlier levels are read after it.
    __device__ __forceinline__ bool ilu_levels(const T *v, T *out) {
        const IluView<T> &M = sys().ilu;
        // a level's positions split into one contiguous chunk per CTA of
        // ceil(size / CTAs): every CTA shares each level (a level is a few
        // thousand scattered rows), and a warp reads consecutive positions
        const int64_t G = gs().nblocks, bid = gs().bid;
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
            gs().arrive();
            if (l + 1 < nl) {
                chunk(M.lptr, l + 1, q0, q1);
                ilu_fetch_l(q0 + tid, q1, v, R);
            } else {
                chunk(M.uptr, 0, q0, q1);
                ilu_fetch_u(q0 + tid, q1, R);
            }
            if (!gs().wait(l + 1)) return false;
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
            gs().arrive();
            if (l + 1 < nu) {
                chunk(M.uptr, l + 1, q0, q1);
                ilu_fetch_u(q0 + tid, q1, R);
            }
            if (!gs().wait(nl + l + 1)) return false;
        }
        ilu_count();
        return true;
    }
    // Accounting of one M^{-1}: factors and row data once, v read, out
    // written and re-read.
    __device__ __forceinline__ void ilu_count() {
        if (threadIdx.x == kAcctThread) {
            acct().bytes += sys().ilu.nnz * (int64_t)(sizeof(T) + 4) + sys().N * (int64_t)(8 + 4 + 8 + 3 * sizeof(T));
            acct().flops += (is_cx<T>::value ? 8 : 2) * sys().ilu.nnz;
        }
    }

    // M^{-1} for factors with few levels, as tiles of the ring: each CTA
    // takes a contiguous share of a level's slices; the producer warp streams
    // their values, columns, (row, count) pairs and U's diagonal (constant
    // data, so the next level's tiles arrive during the level's barrier), and
    // warp w takes slice w of each tile, one row per lane.  As in sell_consume
    // the gathers and the right-hand side of tile t+1 are issued among the
    // FMAs of tile t; rows wider than W entries take the rest in batches.
    // What bounds it: one round of gathers per 480 rows and a barrier per
    // level.  (With a row's loads one after another (index, row pointer,
    // entries, values) one M^{-1} at 96^3, four levels, took 95 us, with the
    // slices read by coalesced loads 100 us.)  Each row is one sequential sum
    // in pattern order.
    __device__ __forceinline__ bool ilu_wide(const T *v, T *out) {
        // entries gathered a tile ahead, and at a time after those (the six
        // of a 7-point row's second colour are in flight together with 0 + 6
        // and 2 + 4).  us of 16 iterations, complex, multicolour, 128x128x64:
        // 3 + 2 9025, 3 + 3 8670, 2 + 4 8300, 1 + 5 7970, 0 + 6 7770 (held
        // values spill); of 24 at 96^3, n = 8: 6 + 3 4270, 0 + 6 4180, 2 + 4
        // 4100; refined 6 + 3 2834, 2 + 4 2790; refined complex 6 + 3 2846,
        // 0 + 6 2913.
        constexpr int W = sizeof(T) == 16 ? 0 : is_cx<T>::value ? 6 : 2;
        constexpr int B = sizeof(T) == 16 ? 6 : is_cx<T>::value ? 3 : 4;
        const int lane = threadIdx.x & 31, cw = threadIdx.x >> 5;
        TileRing *const R = the_ring();
        const int nl = sys().ilu.nlev_l, nlev = nl + sys().ilu.nlev_u, spt = sys().ilu.spt;
        unsigned q = gs().seq();
        for (int l = 0; l < nlev; ++l) {
            const bool up = l >= nl;
            const IluLevel L = up ? sys().ilu.ulev[l - nl] : sys().ilu.llev[l];
            const T *const rhs = up ? out : v;
            const int w = L.w;
            int k0, k1;
            ilu_share(L.ns, k0, k1);
            int st = 0, ns = 0;       // stage and slices of the tile at hand
            int row = -1, cnt = 0;
            T t{}, x[W > 0 ? W : 1];
            // stage of tile q; its slices; false when the wait failed
            auto arrived = [&](int k, unsigned tile, int &stage, int &slices) {
                stage = (int)(tile % kStages);
                slices = k1 - k < spt ? k1 - k : spt;
                return mbar_wait_warp(&R->full[stage], (tile / kStages) & 1u, R->timeout_ns);
            };
            auto vals = [&](int stage) {
                return reinterpret_cast<const T *>(the_stages() + stage * kStageBytes) + cw * 32 * w + lane;
            };
            auto cols = [&](int stage, int slices) {
                return reinterpret_cast<const int32_t *>(the_stages() + stage * kStageBytes +
                                                         slices * 32 * w * (int)sizeof(T)) + cw * 32 * w + lane;
            };
            auto meta = [&](int stage, int slices) {
                return reinterpret_cast<const int2 *>(the_stages() + stage * kStageBytes +
                                                      slices * 32 * w * (int)(sizeof(T) + 4))[cw * 32 + lane];
            };
            auto diag = [&](int stage, int slices) {
                return reinterpret_cast<const T *>(the_stages() + stage * kStageBytes +
                                                   slices * 32 * (w * (int)(sizeof(T) + 4) + 8))[cw * 32 + lane];
            };
            bool ok = k0 >= k1 || arrived(k0, q, st, ns);
            if (k0 < k1 && ok && cw < ns) {
                const int2 m = meta(st, ns);
                row = m.x;
                cnt = m.y;
                if (row >= 0) t = ldcg_val(rhs + row);
                const int32_t *c = cols(st, ns);
#pragma unroll
                for (int e = 0; e < W; ++e)
                    if (e < cnt) x[e] = out[c[32 * e]];
            }
            for (int k = k0; ok && k < k1; k += spt, ++q) {
                int st1 = 0, ns1 = 0, row1 = -1, cnt1 = 0;
                T t1{};
                if (k + spt < k1) {
                    if (!arrived(k + spt, q + 1, st1, ns1)) {
                        ok = false;
                        break;
                    }
                    if (cw < ns1) {
                        const int2 m = meta(st1, ns1);
                        row1 = m.x;
                        cnt1 = m.y;
                        if (row1 >= 0) t1 = ldcg_val(rhs + row1);
                    }
                }
                const T *a = vals(st);
                const int32_t *c = cols(st, ns), *c1 = cols(st1, ns1);
#pragma unroll
                for (int e = 0; e < W; ++e) {
                    if (e < cnt) t = efma(-a[32 * e], x[e], t);
                    if (e < cnt1) x[e] = out[c1[32 * e]];
                }
                for (int e0 = W; e0 < cnt; e0 += B) {
                    T xw[B];
#pragma unroll
                    for (int u = 0; u < B; ++u)
                        if (e0 + u < cnt) xw[u] = out[c[32 * (e0 + u)]];
#pragma unroll
                    for (int u = 0; u < B; ++u)
                        if (e0 + u < cnt) t = efma(-a[32 * (e0 + u)], xw[u], t);
                }
                if (row >= 0) {
                    if (up) t = t / diag(st, ns);
                    out[row] = t;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&R->empty[st]);
                st = st1;
                ns = ns1;
                row = row1;
                cnt = cnt1;
                t = t1;
            }
            if (!ok) tile_lost(l + 1);
            if (!gs().sync(l + 1)) {
                gs().seq() = q;
                return false;
            }
        }
        gs().seq() = q;
        ilu_count();
        return true;
    }
    // This CTA's share [k0, k1) of a level's slices.
    __device__ __forceinline__ static void ilu_share(int ns, int &k0, int &k1) {
        const int G = (int)gs().nblocks, ch = (ns + G - 1) / G;
        k0 = (int)gs().bid * ch;
        k1 = k0 + ch < ns ? k0 + ch : ns;
    }
    // Producer warp: the tiles of ilu_wide (lane 0 the values, 1 the columns,
    // 2 the (row, count) pairs, 3 U's diagonal).
    __device__ __forceinline__ int issue_ilu(unsigned &sq) {
        if constexpr (PC != kIluWide && PC != kIluAny) {
            return 0;
        } else {
            if (!sys().ilu.llev) return 0;
            const int lane = threadIdx.x & 31;
            const int nl = sys().ilu.nlev_l, nlev = nl + sys().ilu.nlev_u, spt = sys().ilu.spt;
            TileRing *const R = the_ring();
            for (int l = 0; l < nlev; ++l) {
                const bool up = l >= nl;
                const IluLevel L = up ? sys().ilu.ulev[l - nl] : sys().ilu.llev[l];
                int k0, k1;
                ilu_share(L.ns, k0, k1);
                const unsigned ev = 32u * (unsigned)L.w;   // entries of a slice
                // bytes of a slice of each lane's part, and where the parts
                // of the share start
                const unsigned b0 = ev * (unsigned)sizeof(T), b1 = ev * 4u, b2 = 256u,
                               b3 = up ? 32u * (unsigned)sizeof(T) : 0u;
                const unsigned mine = lane == 0 ? b0 : lane == 1 ? b1 : lane == 2 ? b2 : lane == 3 ? b3 : 0u;
                const unsigned before = lane == 0 ? 0u : lane == 1 ? b0 : lane == 2 ? b0 + b1 : b0 + b1 + b2;
                const unsigned char *src;
                if (lane == 0) src = (const unsigned char *)((up ? sys().ilu.uell_a : sys().ilu.lell_a) + L.e0);
                else if (lane == 1) src = (const unsigned char *)((up ? sys().ilu.uell_c : sys().ilu.lell_c) + L.e0);
                else if (lane == 2) src = (const unsigned char *)((up ? sys().ilu.umeta : sys().ilu.lmeta) + 32 * (int64_t)L.m0);
                else src = (const unsigned char *)(sys().ilu.udiag + 32 * (int64_t)L.m0);
                for (int k = k0; k < k1; k += spt, ++sq) {
                    const int s = (int)(sq % kStages);
                    const unsigned use = sq / kStages;
                    int st = 0;
                    if (lane == 0 && use > 0) st = producer_wait(R, &R->empty[s], (use - 1) & 1u, false);
                    st = __shfl_sync(0xffffffffu, st, 0);
                    if (st) return st;
                    const unsigned n = (unsigned)(k1 - k < spt ? k1 - k : spt);
                    if (lane == 0) mbar_arrive_expect_tx(&R->full[s], n * (b0 + b1 + b2 + b3));
                    __syncwarp();
                    if (mine)
                        bulk_g2s(the_stages() + s * kStageBytes + n * before, src + (size_t)k * mine, n * mine,
                                 &R->full[s]);
                }
            }
            return 0;
        }
    }

    // Out of line, for the refined mode's residual replacement; the
    // iteration's own M^{-1} is inlined in inner().
    __device__ __noinline__ bool ilu_solve(const T *v, T *out) {
        if (sys().ilu.llev) gs().post(kCmdIlu);
        const bool good = ilu_solve_body(v, out);
        consumer_sync();   // the next team barrier may have any turn
        return good;
    }

    // y_0 = M x_0 = L (U x_0), in place on x: t = U x, then x = L t (two
    // row-parallel products).
    __device__ __forceinline__ bool ilu_to_y() {
        const IluView<T> &M = sys().ilu;
        const int64_t nth = (int64_t)gs().nblocks * kConsumers;
        const int64_t me = (int64_t)gs().bid * kConsumers + threadIdx.x;
        T *const x = sys().x, *const t = M.t;
        for (int64_t i = me; i < sys().N; i += nth) {
            const int64_t kd = M.rp[i] + M.dpos[i], k1 = M.rp[i + 1];
            T s{};
            for (int64_t k = kd; k < k1; ++k) s = efma(M.lu[k], x[M.ci[k]], s);
            t[i] = s;
        }
        if (!gs().sync(1)) return false;
        for (int64_t i = me; i < sys().N; i += nth) {
            const int64_t k0 = M.rp[i], kd = k0 + M.dpos[i];
            T s = ldcg_val(t + i);
            for (int64_t k = k0; k < kd; ++k) s = efma(M.lu[k], ldcg_val(t + M.ci[k]), s);
            x[i] = s;
        }
        return gs().sync();
    }

    // x = M^{-1} y once the final residual pass has formed t = M^{-1} y.
    __device__ __forceinline__ bool ilu_to_x() {
        const int64_t nth = (int64_t)gs().nblocks * kConsumers;
        const int64_t me = (int64_t)gs().bid * kConsumers + threadIdx.x;
        T *const x = sys().x;
        const T *t = sys().ilu.t;
        for (int64_t i = me; i < sys().N; i += nth) x[i] = ldcg_val(t + i);
        return gs().sync();
    }

    // ------------------------------------------------------------------
    // passes
    // ------------------------------------------------------------------
    // Those of the iteration leave this thread's share of their sums in
    // sums.v[0, K) and return what ends them (inner() does it, in one place
    // for all of them).
    struct Sums {
        double v[kMaxSums];
        int K;        // sums; 0: a team barrier (the next pass gathers)
        bool fence;   // the next pass gathers
    };
    template <int K>
    __device__ __forceinline__ static void take(Sums &r, const ACC (&acc)[K], int used, bool fence) {
#pragma unroll
        for (int k = 0; k < K; ++k) r.v[k] = (double)acc[k];
        r.K = used;
        r.fence = fence;
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
        T *const bq = sys().b;
        T *const rq = sys().r;
        T *const xq = sys().x;
        const int64_t clo = c_lo(), chi = c_hi();
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
        if (!gs().template reduce<K>(v, true)) return false;
        bb = the_red().total[0];
        rr = the_red().total[1];
        qr = mk_coef<T>(the_red().total + 2);
        if (threadIdx.x == kAcctThread) acct().bytes += sys().N * (int64_t)(sizeof(TW) + 5 * sizeof(T));
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
        T *const rq = sys().r;
        const int64_t clo = c_lo(), chi = c_hi();
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
        if (!gs().template reduce<K>(v, true)) return false;
        rr = the_red().total[0];
        qr = mk_coef<T>(the_red().total + 1);
        fr = mk_coef<T>(the_red().total + 1 + DS);
        if (threadIdx.x == kAcctThread)
            acct().bytes += sys().N * (int64_t)(sizeof(TW) + (1 + (qv ? 1 : 0) + (fv ? 1 : 0)) * sizeof(T));
        return true;
    }

    // The products, one copy of the code (several crowd each other out of
    // the registers): P_SPMV_C: w_i = A g_i, sum q_i^H w.  P_SPMV_Z: z = A u
    // (u held in r), sums z^H z, z^H u.  P_RESIDUAL: r = b - A x, g_0 = r
    // (write_g0), sums ||b||^2, ||r||^2, q_1^H r (q_1 by direct loads: one
    // such pass per call of the method).
    __device__ __forceinline__ void ph_product(int what, int i, bool write_g0, unsigned &sq, Sums &sums) {
        constexpr int K = 2 + DS;
        ACC acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = ACC(0);
        const bool az = what == P_SPMV_Z, res = what == P_RESIDUAL;
        T *const out = az ? sys().z : res ? sys().r : Wc(i);
        T *const g0 = Gc(0);
        const T *const q1 = sys().Q;
        const T *epi[1] = {az ? sys().r : res ? sys().b : Qc(i)};
        // epilogues capture by value: a captured reference would keep the
        // pointer in memory, reloaded after every store of the loop
        spmv_rows(az ? sys().r : res ? sys().x : Gc(i), epi, sys().spt[res ? 2 : 1], sq,
                  [=](int64_t row, T y, const T (&e)[1], ACC(&a)[K]) {
            if (res) {
                const T rv = subT(e[0], y);
                out[row] = rv;
                if (write_g0) g0[row] = rv;
                acc_nrm(&a[0], e[0]);
                acc_nrm(&a[1], rv);
                acc_dot(&a[2], ldg_val(q1 + row), rv);
            } else {
                out[row] = y;
                if (az) {
                    acc_nrm(&a[1], y);
                    acc_dot(&a[2], y, e[0]);
                } else {
                    acc_dot(&a[2], e[0], y);
                }
            }
        }, acc);
        sbytes(res ? (write_g0 ? 4 : 3) : 1);
        // the sums are the last ones of acc
        const int drop = res ? 0 : az ? 1 : 2;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            ACC v = acc[k];
            if (drop == 1) v = acc[k + 1 < K ? k + 1 : k];
            if (drop == 2) v = acc[k + 2 < K ? k + 2 : k];
            sums.v[k] = (double)v;
        }
        sums.K = K - drop;
        sums.fence = res;
    }

    // x += alpha g_sl, r -= alpha w_sl; sums ||r||^2, q_qcol^H r (hq) and
    // (when f0) f_1^H r.
    __device__ __forceinline__ void ph_alpha(S alpha, bool hq, bool f0, unsigned &sq, Sums &sums) {
        constexpr int K = 1 + 2 * DS;
        const T a = to_t<T>(alpha), na = to_t<T>(-alpha);
        const int ni = 4 + (hq ? 1 : 0) + (f0 ? 1 : 0), iff = hq ? 5 : 4;
        T *const xo = sys().x;
        T *const ro = sys().r;
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
        // without f the sums are ||r||^2 and q^H r, at the block's end (u in
        // r, which the next pass gathers) ||u||^2 alone
        take<K>(sums, acc, f0 ? K : hq ? 1 + DS : 1, !hq);
    }

    // x += omega u, r = u - omega z (u in r); sums ||r||^2, q_1^H r.
    __device__ __forceinline__ void ph_omega(S omega, unsigned &sq, Sums &sums) {
        constexpr int K = 1 + DS;
        const T om = to_t<T>(omega), nom = to_t<T>(-omega);
        T *const xo = sys().x;
        T *const ro = sys().r;
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
        take<K>(sums, acc, K, false);
    }

    // z_w = r + bt0 w_i (first) or z_w += bts w_s, in place; sum q^H z_w.
    __device__ __forceinline__ void ph_w(bool first, S coef, int i, unsigned &sq, Sums &sums) {
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
        take<DS>(sums, acc, DS, false);
    }

    // Last pass of the z_w sweep, fused with every deferred g-update of the
    // sweep and the omega-correction:
    //   first=true : z_w = r + bt()[sl] w_sl                (empty s-loop)
    //   first=false: z_w += bt()[last] w_last
    //   g = bt()[sl] g_sl;  g += bt()[t] g_t for t = sl+1..n-1;  g = z_w - g/omega
    // sums f_1^H g when with_f.  The first kMaxInputs-4 columns g_t come
    // through the tile pipeline, any further ones by direct loads.
    __device__ __forceinline__ void ph_w_last(int sl, unsigned &sq, Sums &sums) {
        const int n = sys().n;
        const int last = n - 1;
        const bool first = sl == last, with_f = sl > 0;
        T *wp = Wc(sl);
        T *gp = Gc(sl);
        const T bl = to_t<T>(bt()[first ? sl : last]);
        const T b0 = to_t<T>(bt()[sl]);
        const T nio = to_t<T>(-sc().inv_omega);
        const int t0 = sl + 1;
        const int nt = n - t0;                                     // g_t columns
        const int ntile = nt < kMaxInputs - 4 ? nt : kMaxInputs - 4;
        const int i_t = with_f ? 4 : 3;
        const T *const Gb = sys().G;
        const int64_t ldv = sys().ld;
        const S *const btl = bt();
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
        take<DS>(sums, acc, with_f ? DS : 0, !with_f);   // without f the next pass gathers g
    }

    // g_i += beta g_s, or (block 0's first) g_i = r + beta g_0; sums f^H g_i, or, at the sweep's end (the next pass gathers g_i), a team
    // barrier.
    __device__ __forceinline__ void ph_g(S beta, int i, bool with_f, unsigned &sq, Sums &sums) {
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
        take<DS>(sums, acc, with_f ? DS : 0, !with_f);
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
        if (rec && ctl().err_hist && iter < ctl().hist_cap && gs().bid == 0) ctl().err_hist[iter] = err;
    }
    __device__ __forceinline__ S total(int k) const { return mk_coef<T>(the_red().total + k); }

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
    // last: only the residual pass (after the last iteration; ||b||^2 and
    // ||r||^2 are then in the_red().total).  One call site per kernel, inlined:
    // this is the kernel's loop, and a call in it costs every pass registers.
    //
    // After inner() returns, x and r are visible to their own CTA only: a
    // team barrier comes before any pass that gathers them.
    template <typename Hook = NoHook>
    __device__ __forceinline__ Out inner(bool last, int64_t maxit, bool rec, double tol,
                                         const typename wide_of<T>::type *init = nullptr, double scale = 1.0,
                                         Hook *hook = nullptr) {
        const int tid = threadIdx.x;
        Out o{1, 0, 0, 0, 0.0};
        if (tid == kAcctThread && !last)
            for (int q = 0; q < 5; ++q) acct().ops[q] = 0;
        if (tid == 0) {
            sc().tol = tol;
            sc().maxit = maxit;
            sc().rec = rec && ctl().err_hist != nullptr;
        }

        Step st;
        if constexpr (is_narrow<T>::value) {
            double bb, rr;
            S e;
            if (!ph_init_narrow(init, scale, bb, rr, e)) return o;
            op(OP_NORM, 2);
            if (tid == 0) start();
            if (tid == 0 && Hook::kActive) hook->reset(sc().err);
            consumer_sync();
            o.err = sc().err;
            if (sc().exit) {
                o.flag = sc().flag;
                return o;
            }
            gs().post(kCmdInner);   // from the product w_0 = A g_0 on
        } else {
            // r_0 = b - A x_0 (step 2) with the stopping-rule denominator
            st.op = P_RESIDUAL;
        }
        unsigned sq = gs().seq();

        // what lives from pass to pass is in shared memory: the registers
        // belong to the pass
        for (;; st.advance(sys().n)) {
            const int i = st.i, n = sys().n;
            // which of its two forms a sweep's pass has (see the cases)
            const bool hq = i < n;                      // P_ALPHA: not the block's end
            const bool f0 = st.first && hq;             // P_ALPHA: block 0's f_1^H r
            const int s1 = st.op == P_F_ROUND ? st.s + 1 : 1;
            const bool more = s1 <= i - 1;              // P_F_ROUND, P_G_J0: another f follows
            if (!is_narrow<T>::value && st.op == P_RESIDUAL) gs().post(kCmdResidual);
            if constexpr (PC != kNoIlu) {
                if ((st.op == P_SPMV_C || st.op == P_SPMV_Z || st.op == P_RESIDUAL) && sys().ilu.lu) {
                    gs().seq() = sq;
                    const bool good = ilu_solve_body(
                        st.op == P_SPMV_C ? Gc(i) : st.op == P_SPMV_Z ? sys().r : sys().x, sys().ilu.t);
                    sq = gs().seq();
                    if (!good) {
                        // no product: the ring may still hold M^{-1}'s tiles
                        if (st.op == P_RESIDUAL) return o;
                        break;
                    }
                }
            }
            Sums sums;
            switch (st.op) {
            case P_RESIDUAL:
            case P_SPMV_C:   // steps 31-32, 51 (and w_0 = A g_0): w = A g, c = q_{i+1}^H w
            case P_SPMV_Z:   // step 38
                ph_product(st.op, i, !last, sq, sums);
                break;
            case P_ALPHA:
                // steps 5-8: alpha, x, r, e (and f_1^H r in block 0); steps
                // 34-36 at the block's end (u kept in r)
                ph_alpha(sc().coef, hq, f0, sq, sums);
                break;
            case P_OMEGA:    // steps 39-41: x += omega u, r = u - omega A u, e = q_1^H r
                ph_omega(sc().coef, sq, sums);
                break;
            case P_W_FIRST:  // steps 10-17, 42-48: sweep the rest of block j-1 with q's
            case P_W_ROUND:
                ph_w(st.op == P_W_FIRST, sc().coef, i, sq, sums);
                break;
            case P_W_LAST:   // its end, with the omega-correction (steps 18, 50)
                ph_w_last(i, sq, sums);
                break;
            default:         // steps 19-22 (24-28 in block 0): sweep block j with f's
                ph_g(sc().coef, i, more, sq, sums);
                break;
            }
            bool good = sums.K ? gs().reduce_k(sums.v, sums.K, sums.fence) : gs().sync();
            // the scalars of the next pass, the stopping rule and the
            // accounting, each on a thread of its own warp
            if (tid == 0) {
                switch (st.op) {
                case P_RESIDUAL:
                    if (!last) start();
                    break;
                case P_SPMV_C: {
                    const S cv = total(0);
                    c()[i] = cv;
                    if (is_zero(cv) || !finite_of(cv)) {
                        sc().flag = -1;
                        sc().exit = 1;
                    }
                    sc().coef = sc().e / cv;
                    break;
                }
                case P_ALPHA:
                    if (hq) alpha_coef(i, f0);
                    break;
                case P_SPMV_Z: {
                    // omega = (A u)^H u / ||A u||^2, Eq. 5.1 guard
                    const double zz = the_red().total[0];
                    const S zu = total(1);
                    const bool bad = zz == 0.0 || !isfinite(zz);
                    S om = zu / zz;
                    if (ctl().kappa > 0.0) {
                        const double arho = abs_of(zu) / (sqrt(zz) * sqrt(sc().rr));
                        if (arho < ctl().kappa && arho != 0.0) om = (ctl().kappa * om) / arho;
                    }
                    if (bad || is_zero(om) || !finite_of(om)) {
                        sc().flag = -1;
                        sc().exit = 1;
                    }
                    sc().bad = bad;
                    sc().coef = om;
                    sc().omega = om;
                    break;
                }
                case P_OMEGA:
                    omega_coef();
                    break;
                case P_W_FIRST:
                case P_W_ROUND: {
                    const int s = st.op == P_W_FIRST ? i + 1 : st.s + 1;
                    const S b = -(total(0) / c()[s]);
                    bt()[s] = b;
                    sc().coef = b;
                    break;
                }
                case P_W_LAST:
                    if (i > 0) sc().coef = -(total(0) / c()[0]);
                    break;
                default:
                    if (more) sc().coef = -(total(0) / c()[s1]);
                    break;
                }
            } else if (tid == kErrThread) {
                if (st.op == P_ALPHA) {
                    sc().j = sc().block;
                    sc().i = i;
                }
                if (st.op == P_OMEGA) sc().block += 1;
                if (st.op == P_ALPHA || st.op == P_OMEGA)
                    residual_norm<Hook>(the_red().total[0], st.op == P_OMEGA || hq, st.op == P_OMEGA, hook);
            } else if (tid == kAcctThread) {
                if (st.op == P_OMEGA) sc().inv_omega = recip(sc().omega);
                if (!last) count(st, n);
            }
            consumer_sync();
            if (st.op == P_RESIDUAL) {
                if (!good || last || sc().exit) {
                    gs().seq() = sq;
                    if (!last) {
                        o.err = sc().err;
                        if (good) o.flag = sc().flag;
                    }
                    return o;
                }
                gs().post(kCmdInner);   // from the product w_0 = A g_0 on
                continue;
            }
            if (!good) break;
            if (st.op == P_SPMV_Z && !sc().bad) {
                op(OP_DOT);
                if (ctl().kappa > 0.0) op(OP_NORM, 2);
            }
            if constexpr (Hook::kActive) {
                if (st.op == P_ALPHA || st.op == P_OMEGA) {
                    if (sc().exit) break;
                    const bool whole = st.op == P_OMEGA || hq;   // not the half step u
                    const bool f1 = st.op == P_ALPHA && f0;
                    if (sc().act) {
                        gs().seq() = sq;
                        double rr;
                        S qr, fr;
                        bool conv;
                        good = hook->replace(st.op == P_OMEGA ? 0 : hq ? i : -1, f1, rr, qr, fr, conv);
                        sq = gs().seq();
                        if (!good) break;
                        if (tid == kErrThread) replaced<Hook>(rr, conv, st.op, whole, hook);
                        if (tid == 0 && whole) {
                            if (st.op == P_OMEGA) omega_coef();
                            else alpha_coef(i, f1);
                        }
                        consumer_sync();
                        if (sc().exit) break;
                    }
                    gs().post(kCmdGo);
                }
            }
            if (sc().exit) break;
            if (st.op == P_ALPHA && hq) op(OP_DOT);
            if (st.op == P_OMEGA) op(OP_DOT);
        }
        gs().end(kCmdStop, sq);
        gs().seq() = sq;
        o.flag = gs().ok ? sc().flag : 1;
        o.iter = sc().iter;
        o.j = sc().j;
        o.i = sc().i;
        o.err = sqrt(sc().rr) / sc().bnrm2;
        return o;
    }

    // Thread 0: the scalars of a start, from ||b||^2, ||r||^2, q_1^H r.
    __device__ __forceinline__ void start() {
        sc().e = total(2);
        const double t0 = sqrt(the_red().total[0]);
        const double bn = t0 == 0.0 ? 1.0 : t0, rr = the_red().total[1], e0 = sqrt(rr) / bn;
        sc().bnrm2 = bn;
        sc().rr = rr;
        sc().err = e0;
        // sqrt(rr) / bn < tol is impossible above this (1e-12 covers the
        // roundings; below 1e-290 the exact test decides)
        const double t = sc().tol * bn, f = t * t * (1.0 + 1e-12);
        sc().far = f > 1e-290 ? f : 1e-290;
        sc().iter = 0;
        sc().flag = 1;
        sc().exit = 0;
        sc().j = sc().i = sc().block = 0;
        sc().act = sc().conv = 0;
        record(sc().rec != 0, 0, e0);
        if (e0 < sc().tol) {
            sc().flag = 0;
            sc().exit = 1;
        }
    }
    // Thread kAcctThread: the operations of a pass that are counted before
    // its exits.
    __device__ __forceinline__ void count(const Step &st, int n) {
        const int i = st.i;
        switch (st.op) {
        case P_RESIDUAL:
            op(OP_NORM, 2);
            op(OP_MATVEC);
            break;
        case P_SPMV_C:
        case P_SPMV_Z:
            op(OP_MATVEC);
            op(OP_DOT);
            break;
        case P_ALPHA:
            // the inner product of c_0 belongs to the first block's start
            if (st.first && i == 1) op(OP_DOT);
            op(OP_SAXPY, 2);
            op(OP_NORM);
            break;
        case P_OMEGA:
            op(OP_SAXPY, 2);
            op(OP_NORM);
            break;
        case P_W_LAST:
            op(OP_SAXPY);   // omega-correction (steps 18, 50)
            if (i == n - 1) {
                op(OP_SAXPY);
                op(OP_SCALE);
            } else {
                op(OP_DOT);
                op(OP_SAXPY, 2);
            }
            break;
        case P_W_FIRST:
            op(OP_SAXPY);
            op(OP_SCALE);
            break;
        case P_W_ROUND:
            op(OP_DOT);
            op(OP_SAXPY, 2);
            break;
        default:
            op(OP_DOT);
            op(OP_SAXPY);
            break;
        }
    }
    // Thread 0: the coefficient after an update of r within a block
    // (i: the step's slot): e, then beta~ of the sweep with q's (bt()[i]) or,
    // in block 0, beta of the one with f's.
    __device__ __forceinline__ void alpha_coef(int i, bool f0) {
        const S e = total(1);
        sc().e = e;
        if (f0) {
            sc().coef = -(total(1 + DS) / c()[0]);
        } else {
            const S b = -(e / c()[i]);
            bt()[i] = b;
            sc().coef = b;
        }
    }
    // Thread 0: the coefficient after the omega step.
    __device__ __forceinline__ void omega_coef() {
        const S e = total(1);
        sc().e = e;
        const S b = -(e / c()[0]);
        bt()[0] = b;
        sc().coef = b;
    }
    // Thread kErrThread, after an update of r (or of u at the block's end,
    // counts = false): iteration count, stopping rule, iteration limit.
    // The division and the square root of ||r|| / ||b|| are only taken where
    // the value is recorded or can decide.
    template <typename Hook>
    __device__ __forceinline__ void residual_norm(double rr, bool counts, bool block_end, Hook *hook) {
        const bool rec = sc().rec != 0;
        sc().rr = rr;
        int64_t iter = sc().iter + (counts ? 1 : 0);
        sc().iter = iter;
        bool conv = false;
        if (Hook::kActive || rec || !(rr > sc().far)) {
            const double err = sqrt(rr) / sc().bnrm2;
            conv = err < sc().tol;
            if constexpr (Hook::kActive) {
                hook->track(err);
                sc().act = conv || (block_end && hook->want(err));
                if (!sc().act) after_norm(err, counts, block_end, hook);
                return;
            }
            if (conv && !counts) {
                iter++;
                sc().iter = iter;
            }
            if (counts || conv) record(rec, iter, err);
        }
        if (conv) {
            sc().flag = 0;
            sc().exit = 1;
        } else if (counts && iter >= sc().maxit) {
            sc().exit = 1;
        }
    }
    // Refined mode: the tests that follow the (possibly replaced) residual.
    template <typename Hook>
    __device__ __forceinline__ void after_norm(double err, bool counts, bool block_end, Hook *hook) {
        if constexpr (Hook::kActive) {
            if (block_end && hook->stalled(sc().iter, err)) sc().exit = 1;
            else if (counts && sc().iter >= sc().maxit) sc().exit = 1;
        }
    }
    template <typename Hook>
    __device__ __forceinline__ void replaced(double rr, bool conv, int op_, bool hq, Hook *hook) {
        if constexpr (Hook::kActive) {
            sc().rr = rr;
            const double err = sqrt(rr) / sc().bnrm2;
            hook->reset(err);
            if (conv) {
                if (!hq) sc().iter += 1;   // the converged half step counts
                sc().flag = 0;
                sc().exit = 1;
            } else {
                after_norm(err, hq, op_ == P_OMEGA, hook);
            }
        }
    }
};

}  // namespace mlb
