// Device building blocks of the ML(n)BiCGStab library (sm_103a):
// scalar types, 16-byte vector packs, a bounded grid barrier and the exchange
// of values between CTAs by tagged slots.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace mlb {

// ---------------------------------------------------------------------------
// complex numbers (interleaved re, im; 8- or 16-byte aligned like C99)
// ---------------------------------------------------------------------------
template <typename R>
struct alignas(2 * sizeof(R)) cx {
    R re, im;
};

using cdouble = cx<double>;
using cfloat = cx<float>;

template <typename T> struct is_cx { static constexpr bool value = false; };
template <typename R> struct is_cx<cx<R>> { static constexpr bool value = true; };

// Real part type.
template <typename T> struct real_of { using type = T; };
template <typename R> struct real_of<cx<R>> { using type = R; };

// Scalar type of the recurrence coefficients: always FP64 (the small
// coefficient arithmetic stays FP64 even when vectors are FP32).
template <typename T> struct coef_of { using type = double; };
template <typename R> struct coef_of<cx<R>> { using type = cdouble; };

__host__ __device__ __forceinline__ double re_of(double a) { return a; }
__host__ __device__ __forceinline__ double re_of(cdouble a) { return a.re; }
__host__ __device__ __forceinline__ double im_of(double) { return 0.0; }
__host__ __device__ __forceinline__ double im_of(cdouble a) { return a.im; }

__host__ __device__ __forceinline__ cdouble operator+(cdouble a, cdouble b) { return {a.re + b.re, a.im + b.im}; }
__host__ __device__ __forceinline__ cdouble operator-(cdouble a, cdouble b) { return {a.re - b.re, a.im - b.im}; }
__host__ __device__ __forceinline__ cdouble operator-(cdouble a) { return {-a.re, -a.im}; }
__host__ __device__ __forceinline__ cdouble operator*(cdouble a, cdouble b) {
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__host__ __device__ __forceinline__ cdouble operator*(double s, cdouble b) { return {s * b.re, s * b.im}; }
__host__ __device__ __forceinline__ cdouble operator/(cdouble a, cdouble b) {
    double d = b.re * b.re + b.im * b.im;
    return {(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}
__host__ __device__ __forceinline__ cdouble operator/(cdouble a, double s) { return {a.re / s, a.im / s}; }
// FP32 complex (the ILU(0) triangular solves of the refined mode)
__host__ __device__ __forceinline__ cfloat operator-(cfloat a) { return {-a.re, -a.im}; }
__host__ __device__ __forceinline__ cfloat operator/(cfloat a, cfloat b) {
    float d = b.re * b.re + b.im * b.im;
    return {(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}
__host__ __device__ __forceinline__ bool is_zero(double a) { return a == 0.0; }
__host__ __device__ __forceinline__ bool is_zero(cdouble a) { return a.re == 0.0 && a.im == 0.0; }
__host__ __device__ __forceinline__ double abs_of(double a) { return fabs(a); }
__host__ __device__ __forceinline__ double abs_of(cdouble a) { return hypot(a.re, a.im); }
__host__ __device__ __forceinline__ bool finite_of(double a) { return isfinite(a); }
__host__ __device__ __forceinline__ bool finite_of(cdouble a) { return isfinite(a.re) && isfinite(a.im); }
__host__ __device__ __forceinline__ double recip(double a) { return 1.0 / a; }
__host__ __device__ __forceinline__ cdouble recip(cdouble a) { return cdouble{1.0, 0.0} / a; }

// Make a coefficient of compute type T from an FP64 coefficient.
template <typename T> __device__ __forceinline__ T to_t(double a) { return (T)a; }
template <typename T> __device__ __forceinline__ T to_t(cdouble a);
template <> __device__ __forceinline__ cdouble to_t<cdouble>(cdouble a) { return a; }
template <> __device__ __forceinline__ cfloat to_t<cfloat>(cdouble a) { return {(float)a.re, (float)a.im}; }
template <> __device__ __forceinline__ double to_t<double>(double a) { return a; }
template <> __device__ __forceinline__ float to_t<float>(double a) { return (float)a; }

// ---------------------------------------------------------------------------
// element arithmetic: y = a*x + y as fused multiply-adds
// ---------------------------------------------------------------------------
__device__ __forceinline__ double fmaR(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fmaR(float a, float b, float c) { return fmaf(a, b, c); }

__device__ __forceinline__ double efma(double a, double x, double y) { return fma(a, x, y); }
__device__ __forceinline__ float efma(float a, float x, float y) { return fmaf(a, x, y); }
template <typename R>
__device__ __forceinline__ cx<R> efma(cx<R> a, cx<R> x, cx<R> y) {
    cx<R> o;
    o.re = fmaR(a.re, x.re, fmaR(-a.im, x.im, y.re));
    o.im = fmaR(a.re, x.im, fmaR(a.im, x.re, y.im));
    return o;
}
__device__ __forceinline__ double emul(double a, double x) { return a * x; }
__device__ __forceinline__ float emul(float a, float x) { return a * x; }
template <typename R>
__device__ __forceinline__ cx<R> emul(cx<R> a, cx<R> x) {
    return {fmaR(a.re, x.re, -a.im * x.im), fmaR(a.re, x.im, a.im * x.re)};
}

// Accumulators of inner products: conj(u) v added into acc (re[, im]).
__device__ __forceinline__ void acc_dot(double *a, double u, double v) { a[0] = fma(u, v, a[0]); }
__device__ __forceinline__ void acc_dot(float *a, float u, float v) { a[0] = fmaf(u, v, a[0]); }
template <typename R>
__device__ __forceinline__ void acc_dot(R *a, cx<R> u, cx<R> v) {
    a[0] = fmaR(u.re, v.re, fmaR(u.im, v.im, a[0]));
    a[1] = fmaR(u.re, v.im, fmaR(-u.im, v.re, a[1]));
}
// |v|^2 added into a[0]
__device__ __forceinline__ void acc_nrm(double *a, double v) { a[0] = fma(v, v, a[0]); }
__device__ __forceinline__ void acc_nrm(float *a, float v) { a[0] = fmaf(v, v, a[0]); }
template <typename R>
__device__ __forceinline__ void acc_nrm(R *a, cx<R> v) { a[0] = fmaR(v.re, v.re, fmaR(v.im, v.im, a[0])); }

// Number of accumulator slots one inner product takes.
template <typename T> constexpr int dslots() { return is_cx<T>::value ? 2 : 1; }

// ---------------------------------------------------------------------------
// 16-byte packs of vector elements
// ---------------------------------------------------------------------------
template <typename T>
struct alignas(16) Pack {
    static constexpr int W = 16 / sizeof(T);
    T e[W];
};

template <typename T>
__device__ __forceinline__ Pack<T> ldp(const T *base, int64_t c) {
    // coherent load (data may have been written earlier in the same launch)
    uint4 u = reinterpret_cast<const uint4 *>(base)[c];
    Pack<T> p;
    *reinterpret_cast<uint4 *>(&p) = u;
    return p;
}
template <typename T>
__device__ __forceinline__ Pack<T> ldp_ro(const T *base, int64_t c) {
    // read-only for the lifetime of the kernel (Q, F, matrix)
    uint4 u = __ldg(reinterpret_cast<const uint4 *>(base) + c);
    Pack<T> p;
    *reinterpret_cast<uint4 *>(&p) = u;
    return p;
}
template <typename T>
__device__ __forceinline__ void stp(T *base, int64_t c, const Pack<T> &p) {
    reinterpret_cast<uint4 *>(base)[c] = *reinterpret_cast<const uint4 *>(&p);
}

// ---------------------------------------------------------------------------
// memory-model helpers and the bounded grid barrier
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned ld_relaxed_u32(const unsigned *p) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_relaxed_i32(const int *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u32(unsigned *p, unsigned v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void red_release_add_u32(unsigned *p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Barrier state in global memory (zeroed before every launch).
struct BarrierState {
    unsigned count;   // arrivals since the launch began (monotonic; grid_barrier)
    unsigned progress;   // changes while a triangular solve moves (Engine::ilu_flow)
    int status;       // 0, or an MLB_ERR_* code set by a CTA that gave up
    int pad1;
};

constexpr int kStatusTimeout = 4;  // == MLB_ERR_TIMEOUT

// Arrive-and-wait of one CTA, executed by thread 0 only, after the CTA's
// writes have been ordered before it (a __syncthreads, or thread 0's own
// writes).  `epoch` counts the barriers this CTA has passed; all CTAs pass
// the same sequence, so barrier e completes when the counter reaches
// e * expected.  The spin is bounded by timeout_ns (%globaltimer) without
// progress of a triangular solve and gives up early when another CTA has already recorded a failure.
// grid_arrive and grid_wait are its two halves, for callers with work to
// overlap with the wait.  Polls are relaxed loads and one fence orders what
// follows them.
__device__ __forceinline__ void grid_arrive(BarrierState *bs, unsigned &epoch) {
    epoch += 1;
    red_release_add_u32(&bs->count, 1u);
}
__device__ __forceinline__ bool grid_wait(BarrierState *bs, unsigned epoch, unsigned expected,
                                          uint64_t timeout_ns) {
    const unsigned target = epoch * expected;
    uint64_t t0 = 0;
    unsigned spins = 0, seen = 0;
    while ((int)(ld_relaxed_u32(&bs->count) - target) < 0) {
        if ((++spins & 31u) == 0) {
            if (ld_relaxed_i32(&bs->status) != 0) return false;
            const uint64_t t = globaltimer_ns();
            const unsigned at = ld_relaxed_u32(&bs->progress);
            if (t0 == 0 || at != seen) {
                t0 = t;
                seen = at;
            } else if (t - t0 > timeout_ns) {
                atomicCAS(&bs->status, 0, kStatusTimeout);
                return false;
            }
        }
        __nanosleep(16);
    }
    fence_acq_rel_gpu();
    return true;
}
__device__ __forceinline__ bool grid_arrive_wait(BarrierState *bs, unsigned &epoch, unsigned expected,
                                                 uint64_t timeout_ns) {
    grid_arrive(bs, epoch);
    return grid_wait(bs, epoch, expected, timeout_ns);
}

// ---------------------------------------------------------------------------
// team exchange: tagged slots
// ---------------------------------------------------------------------------
// A team's barrier and its sums in one step: every CTA puts one 16-byte
// slot per sum, its value and the number of the exchange (epoch), and every
// CTA polls all slots until they carry that epoch.  Against a counter (an
// atomic per CTA, a poll of the counter, then a load of the partial sums)
// this saves the loads after the poll and, where only the CTA's own rows
// follow, the release and acquire.  A slot is put with an atomic exchange: a
// plain store reaches the other SMs later (152 CTAs, one sum, exchange with
// the CTA's two barriers: 1.12 us, with stores 1.59 us, counter and partial
// sums 1.67 us), and a round of polls loads all its slots before it looks at
// the first (one at a time: 2.2 us).  Slots are zeroed before a launch;
// epochs count from 1.  A slot's value and epoch belong together only while
// the load stays one access of 16 bytes, so a reader uses all of its words
// (the epoch is compared whole): of a load with unused words the compiler may
// keep the others as accesses of their own.
struct alignas(16) Slot {
    double v;
    unsigned long long epoch;
};

__device__ __forceinline__ void slot_put(Slot *p, double v, unsigned epoch) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v), ep = epoch;
    asm volatile("{ .reg .b128 q, o; mov.b128 q, {%1, %2}; atom.exch.relaxed.gpu.global.b128 o, [%0], q; }" ::"l"(p),
                 "l"(b), "l"(ep)
                 : "memory");
}
__device__ __forceinline__ Slot slot_load(const Slot *p) {
    unsigned long long b, ep;
    asm volatile("{ .reg .b128 q; ld.relaxed.gpu.global.b128 q, [%2]; mov.b128 {%0, %1}, q; }"
                 : "=l"(b), "=l"(ep)
                 : "l"(p)
                 : "memory");
    return Slot{__longlong_as_double((long long)b), ep};
}
// Slots of one value each (Engine::ilu_flow): a float and its epoch in 8
// bytes, a double in a Slot.
template <int BYTES>
struct ValueSlot {
    using type = Slot;
};
template <>
struct ValueSlot<4> {
    using type = unsigned long long;
};
__device__ __forceinline__ void value_put(Slot *p, double v, unsigned epoch) { slot_put(p, v, epoch); }
__device__ __forceinline__ void value_put(unsigned long long *p, float v, unsigned epoch) {
    const unsigned long long b = (unsigned long long)epoch << 32 | __float_as_uint(v);
    asm volatile("{ .reg .b64 o; atom.exch.relaxed.gpu.global.b64 o, [%0], %1; }" ::"l"(p), "l"(b) : "memory");
}
__device__ __forceinline__ Slot value_load(const Slot *p) { return slot_load(p); }
__device__ __forceinline__ unsigned long long value_load(const unsigned long long *p) {
    unsigned long long b;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(b) : "l"(p) : "memory");
    return b;
}
__device__ __forceinline__ bool value_of(Slot s, unsigned epoch, double &v) {
    v = s.v;
    return s.epoch == epoch;
}
__device__ __forceinline__ bool value_of(unsigned long long s, unsigned epoch, float &v) {
    v = __uint_as_float((unsigned)s);
    return (unsigned)(s >> 32) == epoch;
}

// Limit of a warp's polls in a triangular solve by value slots: `limit_ns`
// without any warp's progress (one may wait for a whole triangle).
struct SlotWait {
    uint64_t t0 = 0;
    unsigned spins = 0, seen = 0;
    // After each round of polls: false (uniformly in the warp) when the wait is
    // over, or another CTA has recorded a failure in bs.  Looks every 32nd time.
    __device__ __forceinline__ bool go_on(BarrierState *bs, uint64_t limit_ns) {
        if ((++spins & 31u) != 0) return true;
        int stop = 0;
        if ((threadIdx.x & 31) == 0) {
            const uint64_t now = globaltimer_ns();
            const unsigned at = ld_relaxed_u32(&bs->progress);
            if (ld_relaxed_i32(&bs->status) != 0) stop = 1;
            else if (t0 == 0 || at != seen) {
                t0 = now;
                seen = at;
            } else if (now - t0 > limit_ns) {
                atomicCAS(&bs->status, 0, kStatusTimeout);
                stop = 1;
            }
        }
        return __shfl_sync(0xffffffffu, stop, 0) == 0;
    }
};

// One warp waits until all G slots at p carry `epoch` and adds their values:
// lane l those of CTAs l, l + 32, ... as a pair tree, then an xor tree over
// the lanes (every lane receives the sum).  The wait is bounded by
// timeout_ns (%globaltimer) and gives up early when another CTA has
// recorded a failure in bs.  Returns false (uniformly in the warp) then.
__device__ __forceinline__ bool slots_sum(const Slot *p, unsigned G, unsigned epoch, BarrierState *bs,
                                          uint64_t timeout_ns, double &sum) {
    constexpr int M = 5;   // slots per lane of one round (160 CTAs: every SM of this GPU)
    const unsigned lane = threadIdx.x & 31;
    double total = 0.0;
    for (unsigned b0 = 0; b0 < G; b0 += 32 * M) {
        const unsigned left = G - b0;
        double x[M];
        unsigned need = 0;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            x[m] = 0.0;
            if (lane + 32 * m < left) need |= 1u << m;
        }
        uint64_t t0 = 0;
        unsigned spins = 0;
        for (;;) {
            Slot s[M];
#pragma unroll
            for (int m = 0; m < M; ++m)
                if (32 * m < left) s[m] = slot_load(p + b0 + (lane + 32 * m < left ? lane + 32 * m : 0));
#pragma unroll
            for (int m = 0; m < M; ++m)
                if ((need >> m & 1u) && s[m].epoch == epoch) {
                    x[m] = s[m].v;
                    need &= ~(1u << m);
                }
            if (__all_sync(0xffffffffu, need == 0)) break;
            if ((++spins & 31u) == 0) {
                int stop = 0;
                if (lane == 0) {
                    const uint64_t now = globaltimer_ns();
                    if (ld_relaxed_i32(&bs->status) != 0) stop = 1;
                    else if (t0 == 0) t0 = now;
                    else if (now - t0 > timeout_ns) {
                        atomicCAS(&bs->status, 0, kStatusTimeout);
                        stop = 1;
                    }
                }
                if (__shfl_sync(0xffffffffu, stop, 0)) return false;
            }
        }
        // the pair tree over 5 terms; terms past the team are zero, so the
        // adds that cannot change the sum are left out
        double part = x[0];
        if (left > 32) part = part + x[1];
        if (left > 64) part = part + (x[2] + x[3]);
        if (left > 128) part = part + x[4];
        total = b0 == 0 ? part : total + part;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    sum = total;
    return true;
}

// Whole-CTA grid barrier: every thread calls it; returns false (uniformly
// in the CTA) when the wait failed, and the caller must then return.
__device__ __forceinline__ bool grid_barrier(BarrierState *bs, unsigned &epoch, unsigned expected,
                                             uint64_t timeout_ns, int *s_flag) {
    __syncthreads();
    if (threadIdx.x == 0) *s_flag = grid_arrive_wait(bs, epoch, expected, timeout_ns) ? 1 : 0;
    __syncthreads();
    return *s_flag != 0;
}

}  // namespace mlb
