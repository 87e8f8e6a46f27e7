// Allocation-free fused y = A x, d = Q^H y for callers that cannot
// allocate device memory (see mlbicgstab_spmv_qdot_noalloc in the header).
//
// The per-CTA partial sums live in one fixed array of this library's own
// device memory instead of caller or library allocations.  Every GPU that
// loads the library holds this array until the process exits.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "../../include/mlbicgstab.h"
#include "mlb_device.cuh"

namespace mlb {
namespace {

constexpr int kNaThreads = 256;
constexpr int kNaWarps = kNaThreads / 32;
constexpr int kNaMaxN = 64;
constexpr int kNaStages = 3;   // groups of 32 rows in a warp's shared memory
// Scratch: the CTAs' sums, value by value (value v of CTA b at v * grid + b).
constexpr int64_t kNaScratchDoubles = 65536;  // 512 KiB

static __device__ __align__(256) double g_noalloc_scratch[kNaScratchDoubles];

// Device address of g_noalloc_scratch, looked up once per device.
std::mutex g_mu;
double *g_addr[256];
bool g_done[256];

int scratch_address(int dev, double **out) {
    if (dev < 0 || dev >= 256) return MLB_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_done[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || p == nullptr) {
            cudaGetLastError();
            return MLB_ERR_CUDA;
        }
        g_addr[dev] = (double *)p;
        g_done[dev] = true;
    }
    *out = g_addr[dev];
    return MLB_OK;
}

__device__ __forceinline__ double ldv(const double *p) { return __ldg(p); }
__device__ __forceinline__ cdouble ldv(const cdouble *p) {
    double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    return {v.x, v.y};
}

__device__ __forceinline__ void cp_async(void *dst, const double *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async(void *dst, const cdouble *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async(void *dst, const int32_t *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// Sums of V values (a power of two, at most 8) over a warp: lane l returns
// the sum of value l / (32 / V).  Each of the first steps halves the values a
// lane still holds, so it takes V + 1 adds where V trees take 5 V (an FP64
// instruction occupies the SM's pipe for ~15 cycles).  Fixed order.
template <int V>
__device__ __forceinline__ double warp_sums(double (&a)[V]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int h = V / 2; h > 0; h /= 2, o /= 2) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const double keep = up ? a[k + h] : a[k], give = up ? a[k] : a[k + h];
            a[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    for (; o > 0; o /= 2) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    return a[0];
}

// The CTA's sums of the threads' values, one per value and CTA, to `part`.
template <typename T, int NB>
__device__ __forceinline__ void cta_parts(const typename real_of<T>::type *acc, int n, double *part) {
    constexpr int DS = dslots<T>(), V = NB * DS;
    constexpr int GV = V < 8 ? V : 8;                // sums taken together
    __shared__ double red[kNaWarps][V];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // GV values at a time (every index into acc a constant: a run-time index
    // would put acc in local memory)
#pragma unroll
    for (int v0 = 0; v0 < V; v0 += GV) {
        if (v0 < n * DS) {
            double a[GV];
#pragma unroll
            for (int k = 0; k < GV; ++k) a[k] = (double)acc[v0 + k];
            const double t = warp_sums<GV>(a);
            if (lane % (32 / GV) == 0) red[warp][v0 + lane / (32 / GV)] = t;
        }
    }
    __syncthreads();
    for (int v = threadIdx.x; v < n * DS; v += kNaThreads) {
        double t[kNaWarps];
#pragma unroll
        for (int w = 0; w < kNaWarps; ++w) t[w] = red[w][v];
#pragma unroll
        for (int h = kNaWarps / 2; h > 0; h /= 2)
#pragma unroll
            for (int w = 0; w < h; ++w) t[w] += t[w + h];
        part[(size_t)v * gridDim.x + blockIdx.x] = t[0];
    }
}

// CTAs an SM holds: as many as the accumulators (NB * DS doubles a thread)
// and the loads in flight leave registers for.
template <typename T, int NB>
constexpr int na_ctas() {
    return NB * dslots<T>() > 16 ? 1 : 2;
}
// Entries of 32 rows that a warp stages (9 a row, complex 7): others are
// read directly.
template <typename T>
constexpr int na_cap() {
    return 32 * (dslots<T>() == 1 ? 9 : 7);
}
template <typename T>
constexpr size_t na_smem() {
    return (size_t)kNaWarps * kNaStages * na_cap<T>() * (sizeof(T) + 4);
}

// One row per lane, 32 rows per warp at a time; each thread keeps NB running
// inner products conj(q_k) y over its rows.  What bounds it at 1e6 rows of 7
// entries: HBM (177 MB for n = 8, 26 us) and the FP64 pipe (15 multiply-adds
// a row, 25 us).  So the warp's entries, which lie one after another, come by
// coalesced asynchronous copies into its own shared memory, 32 rows ahead
// (a lane that walks its row itself touches 14 lines per load instruction,
// and its loads wait for one another), and a row's gathers of x and its
// entries of Q are in flight together.  us a call, before -> now: 101^3, n = 8:
// 65 -> 46 (3.8 TB/s), n = 4: 48 -> 44; 40^3: 25 -> 10.  It is as fast with 2 as
// with 3 CTAs per SM, and a third stage gives 1 us.
// Rows too long for the staging are read directly (where they are so long on
// average the kernel below may run instead).  Each row is one sequential sum in
// the order of its entries.
template <typename T, int NB>
__global__ void __launch_bounds__(kNaThreads, na_ctas<T, NB>())
    spmv_qdot_csr_kernel(int64_t N, const int64_t *rp, const int32_t *ci, const T *av, const T *x,
                         const T *Q, int64_t ldq, int n, T *y, double *part) {
    constexpr int DS = dslots<T>(), V = NB * DS, CAP = na_cap<T>(), ST = kNaStages;
    constexpr int B = DS == 1 ? 7 : 4;               // gathers of x in flight (8: 47 for 46 us)
    constexpr int NQ = V <= 8 ? NB : 0;              // entries of Q loaded ahead
    using ACC = typename real_of<T>::type;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T *const vbuf = reinterpret_cast<T *>(smem) + (size_t)warp * ST * CAP;
    int32_t *const cbuf = reinterpret_cast<int32_t *>(smem + (size_t)kNaWarps * ST * CAP * sizeof(T)) +
                          (size_t)warp * ST * CAP;
    ACC acc[V];
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] = ACC(0);
    const int64_t ng = (N + 31) / 32, step = (int64_t)gridDim.x * kNaWarps;
    // the entries [b, e) of this lane's row of group g (empty past the end)
    auto bounds = [&](int64_t g, int64_t &b, int64_t &e) {
        const int64_t row = g * 32 + lane;
        b = g < ng ? __ldg(rp + (row < N ? row : N)) : 0;
        e = g < ng ? __ldg(rp + (row + 1 < N ? row + 1 : N)) : 0;
    };
    // copies of a group into stage st; the first of its entries, or -1 when
    // it is read directly
    auto stage = [&](int st, int64_t b, int64_t e) -> int64_t {
        const int64_t e0 = __shfl_sync(0xffffffffu, b, 0), e1 = __shfl_sync(0xffffffffu, e, 31);
        const bool fits = __all_sync(0xffffffffu, e1 - e0 <= CAP && b >= e0 && b <= e && e <= e1);
        if (fits)
            for (int64_t t = e0 + lane; t < e1; t += 32) {
                cp_async(vbuf + st * CAP + (t - e0), av + t);
                cp_async(cbuf + st * CAP + (t - e0), ci + t);
            }
        cp_async_commit();
        return fits ? e0 : -1;
    };
    int64_t g = (int64_t)blockIdx.x * kNaWarps + warp;
    // bounds and first entry of the groups g, g + step, ... in flight, and the
    // bounds of the one to be copied next
    int64_t b[ST], e[ST], at[ST];
#pragma unroll
    for (int u = 0; u + 1 < ST; ++u) bounds(g + u * step, b[u], e[u]);
#pragma unroll
    for (int u = 0; u + 1 < ST; ++u) at[u] = stage(u, b[u], e[u]);
    bounds(g + (ST - 1) * step, b[ST - 1], e[ST - 1]);
    for (int st = 0; g < ng; g += step, st = st + 1 < ST ? st + 1 : 0) {
        at[ST - 1] = stage(st > 0 ? st - 1 : ST - 1, b[ST - 1], e[ST - 1]);
        int64_t b2, e2;
        bounds(g + ST * step, b2, e2);
        const int64_t row = g * 32 + lane;
        const bool in = row < N;
        T qv[NQ > 0 ? NQ : 1];
#pragma unroll
        for (int q = 0; q < NQ; ++q) qv[q] = in && q < n ? ldv(Q + (int64_t)q * ldq + row) : T{};
        cp_async_wait<ST - 1>();
        __syncwarp();
        T sum{};
        if (at[0] >= 0) {
            const T *vp = vbuf + st * CAP + (int)(b[0] - at[0]);
            const int32_t *cp = cbuf + st * CAP + (int)(b[0] - at[0]);
            const int len = (int)(e[0] - b[0]);
            for (int k = 0; k < len; k += B) {
                T xv[B];
#pragma unroll
                for (int u = 0; u < B; ++u)
                    if (k + u < len) xv[u] = ldv(x + cp[k + u]);
#pragma unroll
                for (int u = 0; u < B; ++u)
                    if (k + u < len) sum = efma(vp[k + u], xv[u], sum);
            }
        } else {
            for (int64_t k = b[0]; k < e[0]; ++k) sum = efma(ldv(av + k), ldv(x + __ldg(ci + k)), sum);
        }
        if (in) {
            y[row] = sum;
            if constexpr (NQ > 0) {
#pragma unroll
                for (int q = 0; q < NB; ++q)
                    if (q < n) acc_dot(&acc[q * DS], qv[q], sum);
            } else {
#pragma unroll
                for (int q = 0; q < NB; ++q)
                    if (q < n) acc_dot(&acc[q * DS], ldv(Q + (int64_t)q * ldq + row), sum);
            }
        }
        __syncwarp();   // the stage is free
#pragma unroll
        for (int u = 0; u + 1 < ST; ++u) {
            at[u] = at[u + 1];
            b[u] = b[u + 1];
            e[u] = e[u + 1];
        }
        b[ST - 1] = b2;
        e[ST - 1] = e2;
    }
    asm volatile("griddepcontrol.launch_dependents;");
    cta_parts<T, NB>(acc, n, part);
}

// The same for long rows and few sums: each lane walks its row.  A row's loads
// wait for one another, so the threads hide the latency: no staging, 40 to 74
// registers, as many CTAs as an SM holds (6 of n <= 4; the kernel above holds
// 2).  us a call, that kernel -> this one: 64x64x32 reservoir matrix (21 entries
// a row) n = 1 44 -> 39, n = 4 49 -> 41; 27-point 64^3 n = 4 40 -> 37; 30,000
// rows of 130 39 -> 33; complex, 27-point 48^3 n = 1 41 -> 35, n = 8 47 -> 41,
// 60 entries a row 39 -> 26.  With more sums the registers take the CTAs away
// again (real, 130 entries, n = 8 37 -> 41, n = 16 39 -> 54).
template <typename T, int NB>
__global__ void __launch_bounds__(kNaThreads)
    spmv_qdot_csr_long_kernel(int64_t N, const int64_t *rp, const int32_t *ci, const T *av, const T *x,
                              const T *Q, int64_t ldq, int n, T *y, double *part) {
    constexpr int DS = dslots<T>(), V = NB * DS;
    using ACC = typename real_of<T>::type;
    ACC acc[V];
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] = ACC(0);
    for (int64_t row = (int64_t)blockIdx.x * kNaThreads + threadIdx.x; row < N;
         row += (int64_t)gridDim.x * kNaThreads) {
        T sum{};
        for (int64_t k = __ldg(rp + row), k1 = __ldg(rp + row + 1); k < k1; ++k)
            sum = efma(ldv(av + k), ldv(x + __ldg(ci + k)), sum);
        y[row] = sum;
#pragma unroll
        for (int q = 0; q < NB; ++q)
            if (q < n) acc_dot(&acc[q * DS], ldv(Q + (int64_t)q * ldq + row), sum);
    }
    asm volatile("griddepcontrol.launch_dependents;");
    cta_parts<T, NB>(acc, n, part);
}

// d from the CTAs' sums: one warp per value, lanes over the CTAs in index
// order, then the warp's tree.  Launched so that it may start as the product
// ends; in place of a counter that the CTAs take a ticket from (zeroed by a
// launch of its own on every call, a fence and an atomic per CTA).
__global__ void __launch_bounds__(1024) sum_parts_kernel(const double *part, int grid, int nv, double *d) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31;
    for (int v = threadIdx.x >> 5; v < nv; v += blockDim.x >> 5) {
        constexpr int M = 16;   // CTA sums in flight per lane
        double s = 0.0;
        for (int b = lane; b < grid; b += 32 * M) {
            double t[M];
#pragma unroll
            for (int m = 0; m < M; ++m)
                t[m] = b + 32 * m < grid ? __ldcg(part + (size_t)v * grid + b + 32 * m) : 0.0;
#pragma unroll
            for (int h = M / 2; h > 0; h /= 2)
#pragma unroll
                for (int m = 0; m < h; ++m) t[m] += t[m + h];
            s += t[0];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) d[v] = s;
    }
}

// CTAs that device `dev` holds of a kernel with `smem` bytes of dynamic shared
// memory, 0 on failure; asked for once per device (`ctas`: zeroed, one set per
// kernel).
template <typename Kernel>
int device_ctas(int dev, Kernel kernel, size_t smem, std::atomic<int> (&ctas)[256]) {
    int c = ctas[dev].load(std::memory_order_acquire);
    if (c > 0) return c;
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kNaThreads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    c = sms * std::max(per_sm, 1);
    ctas[dev].store(c, std::memory_order_release);
    return c;
}

template <typename T, int NB>
int launch(int dev, int64_t N, int64_t nnz, const int64_t *rp, const int32_t *ci, const T *av, const T *x, const T *Q,
           int64_t ldq, int n, T *y, T *d, double *scratch, cudaStream_t st) {
    constexpr int DS = dslots<T>();
    auto *kernel = spmv_qdot_csr_kernel<T, NB>;
    size_t smem = na_smem<T>();
    static std::atomic<int> staged[256], walked[256];
    auto *held = &staged;
    // the line: rows that on average do not fit the staging, and as many sums
    // as the other kernel has registers for (see there)
    if constexpr (NB <= (DS == 1 ? 4 : 8)) {
        if (nnz > N * (na_cap<T>() / 32)) {
            kernel = spmv_qdot_csr_long_kernel<T, NB>;
            smem = 0;
            held = &walked;
        }
    }
    const int ctas = device_ctas(dev, kernel, smem, *held);
    if (ctas == 0) return MLB_ERR_CUDA;
    const int64_t fit = kNaScratchDoubles / ((int64_t)NB * DS);
    const int64_t need = (N + kNaThreads - 1) / kNaThreads;
    const int64_t grid = std::min<int64_t>(ctas, std::min(fit, need));
    kernel<<<(int)grid, kNaThreads, smem, st>>>(N, rp, ci, av, x, Q, ldq, n, y, scratch);
    if (cudaGetLastError() != cudaSuccess) return MLB_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(std::min(32 * n * DS, 1024));
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, sum_parts_kernel, (const double *)scratch, (int)grid, n * DS,
                           reinterpret_cast<double *>(d)) != cudaSuccess) {
        cudaGetLastError();
        return MLB_ERR_CUDA;
    }
    return MLB_OK;
}

template <typename T>
int dispatch(int dev, int64_t N, int64_t nnz, const int64_t *rp, const int32_t *ci, const T *av, const T *x,
             const T *Q, int64_t ldq, int n, T *y, T *d, double *scratch, cudaStream_t st) {
    if (n <= 4) return launch<T, 4>(dev, N, nnz, rp, ci, av, x, Q, ldq, n, y, d, scratch, st);
    if (n <= 8) return launch<T, 8>(dev, N, nnz, rp, ci, av, x, Q, ldq, n, y, d, scratch, st);
    if (n <= 16) return launch<T, 16>(dev, N, nnz, rp, ci, av, x, Q, ldq, n, y, d, scratch, st);
    if (n <= 32) return launch<T, 32>(dev, N, nnz, rp, ci, av, x, Q, ldq, n, y, d, scratch, st);
    return launch<T, kNaMaxN>(dev, N, nnz, rp, ci, av, x, Q, ldq, n, y, d, scratch, st);
}

// Device memory of the current device `dev`, or managed memory.  Memory of
// another GPU is refused: the kernel runs on `dev`, where such a pointer
// is either unmapped (without peer access) or read over NVLink.
bool on_device(const void *p, int dev) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (at.type == cudaMemoryTypeManaged) return true;
    return at.type == cudaMemoryTypeDevice && at.device == dev;
}

}  // namespace
}  // namespace mlb

extern "C" int mlbicgstab_spmv_qdot_noalloc(int64_t nrows, int64_t nnz, const int64_t *row_ptr,
                                            const int32_t *col_idx, const void *values, int32_t dtype,
                                            const void *x, const void *Q, int64_t ldq, int32_t n, void *y,
                                            void *d, void *stream) {
    using namespace mlb;
    if (nrows <= 0 || nrows > (int64_t)INT32_MAX || nnz < 0 || n < 1 || n > kNaMaxN || ldq < nrows)
        return MLB_ERR_ARG;
    if (dtype != MLB_F64 && dtype != MLB_C128) return MLB_ERR_ARG;
    if (!row_ptr || !x || !Q || !y || !d || (nnz > 0 && (!col_idx || !values))) return MLB_ERR_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return MLB_ERR_CUDA;
    }
    if (!on_device(row_ptr, dev) || !on_device(x, dev) || !on_device(Q, dev) || !on_device(y, dev) ||
        !on_device(d, dev) || (nnz > 0 && (!on_device(col_idx, dev) || !on_device(values, dev))))
        return MLB_ERR_ARG;
    double *scratch = nullptr;
    int rc = scratch_address(dev, &scratch);
    if (rc != MLB_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    if (dtype == MLB_C128)
        return dispatch<cdouble>(dev, nrows, nnz, row_ptr, col_idx, (const cdouble *)values, (const cdouble *)x,
                                 (const cdouble *)Q, ldq, n, (cdouble *)y, (cdouble *)d, scratch, st);
    return dispatch<double>(dev, nrows, nnz, row_ptr, col_idx, (const double *)values, (const double *)x,
                            (const double *)Q, ldq, n, (double *)y, (double *)d, scratch, st);
}
