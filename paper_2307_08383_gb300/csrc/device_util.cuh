// Device helpers shared by the libba kernels.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "ba_internal.h"

namespace ba {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum NV doubles over the CTA; the result is valid in every lane of warp 0.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double *sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = warp_sum(v[i]);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < NV; ++i) sh[w * NV + i] = v[i];
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = warp_sum(lane < nw ? sh[lane * NV + i] : 0.0);
    }
    __syncthreads();
}

// Deterministic grid-wide sum: every CTA stores its partial, the last CTA to
// arrive (a counter, no waiting) adds the partials in CTA order and thread 0
// runs fin(totals).  Must be the last thing a kernel does; every thread of
// every CTA must call it.
template <int NV, class Fin>
__device__ __forceinline__ void grid_sum(double (&v)[NV], double *part, unsigned *counter, Fin fin) {
    __shared__ double sh[32 * NV];
    __shared__ bool last;
    block_sum<NV>(v, sh);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) part[blockIdx.x * NV + i] = v[i];
        __threadfence();
        const unsigned t = atomicAdd(counter, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = 0.0;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x)
#pragma unroll
        for (int i = 0; i < NV; ++i) acc[i] += __ldcg(part + b * NV + i);
    block_sum<NV>(acc, sh);
    if (threadIdx.x == 0) {
        fin(acc);
        *counter = 0;
        __threadfence();
    }
}


__device__ __forceinline__ double clampd(double x) { return x < 1e-6 ? 1e-6 : (x > 1e32 ? 1e32 : x); }
template <typename T> __device__ __forceinline__ T clampT(T x) { return x < T(1e-6) ? T(1e-6) : (x > T(1e32) ? T(1e32) : x); }

// Per-thread running sum in the mode precision.  FP32: compensated
// (Knuth TwoSum, error-free per step), so a thread's partial keeps about
// twice FP32 precision without touching GB300's slow FP64 pipe; the
// partials are then added across threads in FP64.  FP64: plain.
template <typename T> struct RunSum;
template <> struct RunSum<float> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x, z = t - s;
        c += (s - (t - z)) + (x - z);
        s = t;
    }
    __device__ __forceinline__ double get() const { return (double)s + (double)c; }
};
template <> struct RunSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ double get() const { return s; }
};

// FP32 to FP64 without the FP64 pipe's conversion (16 cycles per warp, as much as
// a multiply-add there; this is about six on the integer pipe): the exponent
// rebiased, the mantissa shifted.  Exact; denormals, infinities and NaN take
// the conversion.
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), m = u << 1;
    if (m != 0u && m - 0x01000000u >= 0xfe000000u) return (double)f;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (m ? 0x38000000u : 0u))),
                            (int)(u << 29));
}
__device__ __forceinline__ double widen(double d) { return d; }

// a / b in two steps after the reciprocal inv = 1 / b (correctly rounded, formed
// before a is known or for several a): the quotient's remainder is exact and the
// correction leaves it correctly rounded (Markstein, IBM J. Res. Dev. 34, 1990).
// Where the reciprocal or the remainder leaves the normal range, the division.
__device__ __forceinline__ double quotient(double a, double b, double inv) {
    const double q = a * inv, r = fma(-q, b, a);
    const double m = fabs(b);
    if (!(m > 1e-150 && m < 1e150 && ((fabs(q) > 1e-100 && fabs(q) < 1e100) || a == 0.0))) return a / b;
    return fma(r, inv, q);
}

// Cholesky of symmetric 6x6 matrices, eight lanes each (lane r < 6 of a group
// holds row r in a; lanes 6 and 7 hold zeros): on return a holds row r of L
// (columns k <= r), x column r of L^-1 (rows k >= r, zeros above), and the
// result is false in the whole group if a pivot is not positive.  One thread
// per matrix ran some 450 FP64 instructions of 64 cycles each; a group runs
// about 170, its pivots' one division per column.  STORED: the factor is used in
// its own precision, and its entries are quotients; else (FP64, rounded to FP32
// afterwards) products with the pivot's reciprocal, 2 us less for 200 cameras.
template <typename T, bool STORED = true>
__device__ __forceinline__ bool chol6_lanes(T (&a)[6], T (&x)[6]) {
    constexpr unsigned FULL = 0xffffffffu;
    const int r = threadIdx.x & 7;
    bool ok = true;
    T invd = T(1);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        T p = __shfl_sync(FULL, a[q], q, 8);
        if (!(p > T(0))) {
            ok = false;
            p = T(1);
        }
        const T s = sqrt(p);
        if constexpr (sizeof(T) == 4) {  // one division for the column and for the pivot's reciprocal
            const T v = (r == q ? T(1) : a[q]) / s;
            if (r == q) invd = v;
            a[q] = r == q ? s : v;
        } else {
            const T inv = T(1) / s;
            if (r == q) invd = inv;
            a[q] = r == q ? s : (STORED ? quotient(a[q], s, inv) : a[q] * inv);
        }
#pragma unroll
        for (int k = q + 1; k < 6; ++k) a[k] -= a[q] * __shfl_sync(FULL, a[q], k, 8);  // rows r >= k are meant
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const T dq = __shfl_sync(FULL, invd, q, 8);
        T s = T(0);
#pragma unroll
        for (int k = 0; k < q; ++k) s += __shfl_sync(FULL, a[k], q, 8) * x[k];
        x[q] = q < r ? T(0) : (q == r ? dq : -s * dq);
    }
    return ok;
}
// Row r of the inverse, from chol6_lanes' x: (L^-1)^T L^-1.
template <typename T>
__device__ __forceinline__ void inv6_row(const T (&x)[6], T (&out)[6]) {
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        T s = T(0);
#pragma unroll
        for (int k = c; k < 6; ++k) s += x[k] * __shfl_sync(0xffffffffu, x[k], c, 8);
        out[c] = s;
    }
}
// A lane's row of six values to an 8-byte aligned address.
__device__ __forceinline__ void store6(float *p, const float (&v)[6]) {
    float2 *q = reinterpret_cast<float2 *>(p);
#pragma unroll
    for (int k = 0; k < 3; ++k) q[k] = make_float2(v[2 * k], v[2 * k + 1]);
}
__device__ __forceinline__ void store6(double *p, const double (&v)[6]) {
    double2 *q = reinterpret_cast<double2 *>(p);
#pragma unroll
    for (int k = 0; k < 3; ++k) q[k] = make_double2(v[2 * k], v[2 * k + 1]);
}

// Quaternion (w, x, y, z) of the rotation vector v.
__device__ __forceinline__ void quat_exp(const double *v, double *q) {
    const double th2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    const double th = sqrt(th2);
    double s, c;
    if (th < 1e-8) {
        s = 0.5 - th2 / 48.0;
        c = 1.0 - th2 / 8.0;
    } else {
        s = sin(0.5 * th) / th;
        c = cos(0.5 * th);
    }
    q[0] = c;
    q[1] = s * v[0];
    q[2] = s * v[1];
    q[3] = s * v[2];
}

// Rotation vector of a unit quaternion (shortest rotation).
__device__ __forceinline__ void quat_log(const double *qin, double *v) {
    double q[4] = {qin[0], qin[1], qin[2], qin[3]};
    if (q[0] < 0) { q[0] = -q[0]; q[1] = -q[1]; q[2] = -q[2]; q[3] = -q[3]; }
    const double s = sqrt(q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
    double f;
    if (s < 1e-8) {
        f = 2.0 / q[0] * (1.0 - s * s / (3.0 * q[0] * q[0]));
    } else {
        f = 2.0 * atan2(s, q[0]) / s;
    }
    v[0] = f * q[1];
    v[1] = f * q[2];
    v[2] = f * q[3];
}

__device__ __forceinline__ void quat_mul(const double *a, const double *b, double *o) {
    o[0] = a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3];
    o[1] = a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2];
    o[2] = a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1];
    o[3] = a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0];
}

// Row-major rotation matrix of a unit quaternion.
__device__ __forceinline__ void quat_to_R(const double *q, double *R) {
    const double w = q[0], x = q[1], y = q[2], z = q[3];
    R[0] = 1 - 2 * (y * y + z * z); R[1] = 2 * (x * y - w * z);     R[2] = 2 * (x * z + w * y);
    R[3] = 2 * (x * y + w * z);     R[4] = 1 - 2 * (x * x + z * z); R[5] = 2 * (y * z - w * x);
    R[6] = 2 * (x * z - w * y);     R[7] = 2 * (y * z + w * x);     R[8] = 1 - 2 * (x * x + y * y);
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_add_release(unsigned *p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Symmetric deterministic grid all-reduce for persistent cooperative kernels.
// `bar` is an arrival counter that starts at 0 for the launch and only grows;
// `gen` numbers this kernel's calls 0, 1, 2, ...  Each CTA stores its NV
// partials (v, valid in warp 0 as block_sum leaves them) in half (gen & 1)
// of `part` (2 * gridDim.x * AR_NV_MAX doubles), announces itself with a release
// add and waits (bounded) until (gen + 1) * gridDim.x arrivals.  Then every
// thread loads the partials of CTAs threadIdx.x, threadIdx.x + blockDim.x, ...
// (its loads issued together: one L2 round trip) and a block sum joins them,
// an order fixed by the launch shape, so every CTA obtains the same bits
// without a broadcast round trip.  A half is written again only two calls
// later, by a CTA that has passed call gen + 1, which every CTA enters after
// reading the partials of call gen.  On return every thread holds the totals;
// false on timeout.  The shared totals are rewritten by the next call only
// after its first barrier, which every thread reaches after reading them.
constexpr int AR_NV_MAX = 4;
template <int NV>
__device__ __forceinline__ bool grid_allreduce_sym(double (&v)[NV], double *part, unsigned gen, unsigned *bar,
                                                   int *err, long long limit_cycles) {
    static_assert(NV <= AR_NV_MAX, "too many values");
    __shared__ double s_tot[NV];
    __shared__ double s_red[NV * 32];
    __shared__ int s_ok;
    double *half = part + (size_t)(gen & 1u) * gridDim.x * AR_NV_MAX;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) __stcg(half + blockIdx.x * AR_NV_MAX + k, v[k]);
        red_add_release(bar, 1u);
        const unsigned target = (gen + 1u) * gridDim.x;
        const long long t0 = clock64();
        int ok = 1;
        while (ld_acquire(bar) < target) {
            if (clock64() - t0 > limit_cycles || *(volatile int *)err == (int)BA_ERR_TIMEOUT) {
                atomicExch(err, (int)BA_ERR_TIMEOUT);
                ok = 0;
                break;
            }
        }
        s_ok = ok;
    }
    __syncthreads();  // thread 0's acquire orders every thread's partial reads
    const bool ok = s_ok != 0;
    double acc[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = 0.0;
    if (ok) {
        const unsigned b0 = threadIdx.x, b1 = threadIdx.x + blockDim.x;
        double t0[NV], t1[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            t0[k] = b0 < gridDim.x ? __ldcg(half + b0 * AR_NV_MAX + k) : 0.0;
            t1[k] = b1 < gridDim.x ? __ldcg(half + b1 * AR_NV_MAX + k) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = t0[k] + t1[k];
        for (unsigned b = threadIdx.x + 2 * blockDim.x; b < gridDim.x; b += blockDim.x)
#pragma unroll
            for (int k = 0; k < NV; ++k) acc[k] += __ldcg(half + b * AR_NV_MAX + k);
    }
    block_sum<NV>(acc, s_red);
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) s_tot[k] = acc[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = s_tot[k];
    return ok;
}

// Totals over the warp of one or two doubles per lane, with half the adds of
// two butterflies: the two values are folded onto the warp's halves first.
// Lanes 0..15 return the total of v[0], lanes 16..31 that of v[NV - 1].
// (FP64 adds issue at 1/64 of the FP32 rate on GB300: 16 cycles per warp.)
template <int NV>
__device__ __forceinline__ double warp_fold(const double (&v)[NV]) {
    static_assert(NV == 1 || NV == 2, "one or two values");
    const bool up = (threadIdx.x & 16) != 0;
    const double send = NV == 2 && !up ? v[NV - 1] : v[0];
    double keep = NV == 2 && up ? v[NV - 1] : v[0];
    keep += __shfl_xor_sync(0xffffffffu, send, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, o);
    return keep;
}

// The exchange of a grid all-reduce, run by one warp per CTA of a cooperative
// launch: v holds the CTA's partials in lane 0; they are published, the CTA
// announces itself (arrivals spread over AR_SUB counters on lines of their own
// as in grid_allreduce_df, the wait bounded), and the warp adds all CTAs'
// partials, each lane's loads issued together.  Totals in every lane, the same
// bits in every CTA; false on timeout (the error word is set).  `bar` holds
// AR_SUB * 32 words, zero at launch; `gen` numbers the launch's calls.
constexpr int AR_SUB = 16;
template <int NV>
__device__ __forceinline__ bool grid_exchange(double (&v)[NV], double *part, unsigned gen, unsigned *bar, int *err,
                                              long long limit_cycles) {
    const int lane = threadIdx.x & 31;
    double2 *half = reinterpret_cast<double2 *>(part + (size_t)(gen & 1u) * gridDim.x * AR_NV_MAX);
    if (lane == 0) {
        __stcg(half + blockIdx.x, make_double2(v[0], v[NV - 1]));
        red_add_release(bar + 32 * (blockIdx.x % AR_SUB), 1u);
    }
    int lane_ok = 1;
    if (lane < AR_SUB) {
        const unsigned per = gridDim.x / AR_SUB + ((unsigned)lane < gridDim.x % AR_SUB ? 1u : 0u);
        const unsigned target = (gen + 1u) * per;
        const long long t0 = clock64();
        while (ld_acquire(bar + 32 * lane) < target) {
            if (clock64() - t0 > limit_cycles || *(volatile int *)err == (int)BA_ERR_TIMEOUT) {
                lane_ok = 0;
                break;
            }
        }
    }
    const bool ok = __all_sync(0xffffffffu, lane_ok) != 0;  // orders the other lanes' partial reads too
    __syncwarp();
    double acc[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = 0.0;
    if (ok) {
        double2 u[5];
#pragma unroll
        for (int q = 0; q < 5; ++q)
            u[q] = lane + 32 * q < (int)gridDim.x ? __ldcg(half + lane + 32 * q) : make_double2(0.0, 0.0);
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            acc[0] += u[q].x;
            if (NV == 2) acc[NV - 1] += u[q].y;
        }
        for (unsigned b0 = lane + 160; b0 < gridDim.x; b0 += 160) {
#pragma unroll
            for (int q = 0; q < 5; ++q)
                u[q] = b0 + 32 * q < gridDim.x ? __ldcg(half + b0 + 32 * q) : make_double2(0.0, 0.0);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                acc[0] += u[q].x;
                if (NV == 2) acc[NV - 1] += u[q].y;
            }
        }
    } else if (lane == 0) {
        atomicExch(err, (int)BA_ERR_TIMEOUT);
    }
    const double tot = warp_fold<NV>(acc);
    v[0] = __shfl_sync(0xffffffffu, tot, 0);
    if (NV == 2) v[NV - 1] = __shfl_sync(0xffffffffu, tot, 16);
    return ok;
}

// A 16-byte slot of payload and tag, moved by one 128-bit access: a reader
// that sees the tag has the payload, with no flag to wait for and no second
// round trip.  (Relaxed: acquiring polls would not overlap one another.)
__device__ __forceinline__ void st_slot(void *p, unsigned long long a, unsigned long long b) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p), "l"(a),
                 "l"(b)
                 : "memory");
}
__device__ __forceinline__ void ld_slot(const void *p, unsigned long long &a, unsigned long long &b) {
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(a), "=l"(b)
                 : "l"(p)
                 : "memory");
}
// Whether a bounded poll gives up: its cycles are used up, or (looked at every
// 64th time) another wait of the launch has timed out.
__device__ __forceinline__ bool poll_over(long long t0, long long limit_cycles, unsigned n, int *err) {
    return clock64() - t0 > limit_cycles || ((n & 63u) == 63u && *(volatile int *)err == (int)BA_ERR_TIMEOUT);
}

// The exchange of a grid all-reduce by mailboxes, run by one warp per CTA of a
// cooperative launch; the totals alone cross, nothing else is ordered.  Post:
// every lane stores the CTA's partials (v, the same in all lanes) with the
// call's tag into the mailboxes of CTAs lane, lane + 32, ...  Wait: every lane
// polls the CTA's own mailbox for the partials of the same CTAs (bounded) and
// the warp adds them.  Totals in every lane, the same bits in every CTA; false
// on timeout (the error word is set).  `mail` holds mail_bytes(gridDim.x)
// bytes; `epoch` numbers the launches that use it from 1 on, `gen` the launch's
// calls (two sets in turn: a set is written again only two calls later, by a
// CTA that has every CTA's partials of call gen + 1, sent after reading call
// gen).  All accesses are relaxed; what orders that reuse is dependence: a post
// of call gen + 1 is computed from the totals of call gen, so after the reads of
// that call, and a post of gen + 2 from those of every gen + 1.  A slot written
// too early would carry a tag that its reader does not take: the wait would end
// by its limit, never with another call's value.
// miss: 0 (set, the tag waited for is one that nobody posts).
// Against grid_exchange: a store and a poll instead of a store, its
// acknowledged release, an atomic, a poll and a read.  One slot per CTA that
// all the others poll was slower than either at 100 CTAs and more (its few
// lines are read by every SM while they are written).
__host__ __device__ constexpr size_t mail_bytes(int grid) { return (size_t)2 * 2 * 16 * grid * grid; }
struct Mail {
    unsigned char *box;
    unsigned epoch, miss;
};
template <int NV>
__device__ __forceinline__ void mail_post(const double (&v)[NV], const Mail &m, unsigned gen) {
    const unsigned G = gridDim.x;
    const unsigned long long tag = ((unsigned long long)m.epoch << 32) | gen;
    unsigned char *o = m.box + ((size_t)(gen & 1u) * G * 2 * G + blockIdx.x) * 16;
    for (unsigned b = threadIdx.x & 31; b < G; b += 32) {
#pragma unroll
        for (int k = 0; k < NV; ++k)
            st_slot(o + ((size_t)b * 2 + k) * G * 16, (unsigned long long)__double_as_longlong(v[k]), tag);
    }
}
template <int NV>
__device__ __forceinline__ bool mail_wait(double (&v)[NV], const Mail &m, unsigned gen, int *err,
                                          long long limit_cycles) {
    const unsigned G = gridDim.x, lane = threadIdx.x & 31;
    const unsigned long long tag = ((unsigned long long)(m.epoch + m.miss) << 32) | gen;
    const unsigned char *in = m.box + ((size_t)(gen & 1u) * G + blockIdx.x) * 2 * G * 16;
    double acc[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = 0.0;
    bool ok = true;
    const long long t0 = clock64();
    for (unsigned b0 = 0; b0 < G && ok; b0 += 160) {
        unsigned long long u[NV][5], t[NV][5];
#pragma unroll
        for (int k = 0; k < NV; ++k)
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                u[k][q] = 0ull;
                t[k][q] = tag;
            }
        for (unsigned n = 0;; ++n) {
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    const unsigned b = b0 + lane + 32 * q;
                    if (b < G) ld_slot(in + ((size_t)k * G + b) * 16, u[k][q], t[k][q]);
                }
            bool all = true;
#pragma unroll
            for (int q = 0; q < 5; ++q) all = all && t[0][q] == tag && t[NV - 1][q] == tag;
            if (all) break;
            if (poll_over(t0, limit_cycles, n, err)) {
                ok = false;
                break;
            }
        }
        __syncwarp();
        ok = __all_sync(0xffffffffu, ok) != 0;
        // (64 cycles an add: none for the stretches that the grid does not reach)
#pragma unroll
        for (int q = 0; q < 5; ++q)
            if (b0 + 32 * q < G) {
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    const double x = __longlong_as_double((long long)u[k][q]);
                    acc[k] = b0 + q == 0 ? x : acc[k] + x;
                }
            }
    }
    if (!ok && lane == 0) atomicExch(err, (int)BA_ERR_TIMEOUT);
    const double tot = warp_fold<NV>(acc);
    v[0] = __shfl_sync(0xffffffffu, tot, 0);
    if (NV == 2) v[NV - 1] = __shfl_sync(0xffffffffu, tot, 16);
    return ok;
}

// grid_allreduce_sym for kernels of few warps per CTA: v holds the own
// partials of every thread of the first nwv warps (at most 16 warps per CTA),
// and warp 0 alone runs the exchange, so that a call costs one warp-wide fold
// of FP64 adds per such warp and two in warp 0.  Warp 0 then runs
// fin(totals, ok) (for what only one warp needs to compute) before the CTA's
// other warps go on.  Totals in every thread; false on timeout.
template <int NV, class F>
__device__ __forceinline__ bool grid_allreduce_w0(double (&v)[NV], double *part, unsigned gen, unsigned *bar,
                                                  int *err, long long limit_cycles, int nwv, F &&fin) {
    __shared__ double s_w[NV * 16];
    __shared__ double s_tot[NV];
    __shared__ int s_ok;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w < nwv) {
        const double t = warp_fold<NV>(v);
        if (lane == 0) s_w[w] = t;
        if (NV == 2 && lane == 16) s_w[16 * (NV - 1) + w] = t;
    }
    if (nwv > 1) __syncthreads();
    else __syncwarp();
    if (w == 0) {
        const int l = lane & 15;
        double t = l < nwv ? s_w[(NV == 2 ? lane & 16 : 0) + l] : 0.0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
            if (o < nwv) t += __shfl_xor_sync(0xffffffffu, t, o);
        double x[NV];
        x[NV - 1] = __shfl_sync(0xffffffffu, t, 16);
        x[0] = __shfl_sync(0xffffffffu, t, 0);
        const bool ok = grid_exchange<NV>(x, part, gen, bar, err, limit_cycles);
        fin(x, ok);
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < NV; ++k) s_tot[k] = x[k];
            s_ok = ok ? 1 : 0;
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = s_tot[k];
    return s_ok != 0;
}
template <int NV>
__device__ __forceinline__ bool grid_allreduce_w0(double (&v)[NV], double *part, unsigned gen, unsigned *bar,
                                                  int *err, long long limit_cycles) {
    return grid_allreduce_w0<NV>(v, part, gen, bar, err, limit_cycles, (int)(blockDim.x >> 5),
                                 [](const double (&)[NV], bool) {});
}

// ---- 6x6 block SpMV helpers (BSMC and the full-block formats) ----

// One 6x6 block (16-byte aligned) into registers, read-only path.
template <typename TS, typename TV>
__device__ __forceinline__ void load_block(const TS *__restrict__ Sb, TV (&v)[36]) {
    if constexpr (sizeof(TS) == 4) {
        const float4 *s4 = reinterpret_cast<const float4 *>(Sb);
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float4 t = __ldg(s4 + q);
            v[4 * q] = (TV)t.x; v[4 * q + 1] = (TV)t.y; v[4 * q + 2] = (TV)t.z; v[4 * q + 3] = (TV)t.w;
        }
    } else {
        const double2 *s2 = reinterpret_cast<const double2 *>(Sb);
#pragma unroll
        for (int q = 0; q < 18; ++q) {
            const double2 t = __ldg(s2 + q);
            v[2 * q] = (TV)t.x; v[2 * q + 1] = (TV)t.y;
        }
    }
}

// Six entries of a camera vector (24 B for FP32, 8-byte aligned; 48 B for FP64).
__device__ __forceinline__ void load6(const float *p, float (&v)[6]) {
    const float2 *p2 = reinterpret_cast<const float2 *>(p);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float2 t = __ldcg(p2 + k);
        v[2 * k] = t.x;
        v[2 * k + 1] = t.y;
    }
}
__device__ __forceinline__ void load6(const double *p, double (&v)[6]) {
    const double2 *p2 = reinterpret_cast<const double2 *>(p);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double2 t = __ldcg(p2 + k);
        v[2 * k] = t.x;
        v[2 * k + 1] = t.y;
    }
}

template <typename TV>
__device__ __forceinline__ void block_apply(const TV (&Sv)[36], const TV (&x)[6], bool transposed, TV (&acc)[6]) {
    if constexpr (sizeof(TV) == 8) {
        // a warp whose lanes hold entries of both forms runs one product, not
        // two (36 FP64 instructions of 16-64 cycles against selects on the
        // integer pipe); same sums in the same order
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int c = 0; c < 6; ++c) acc[r] += (transposed ? Sv[6 * c + r] : Sv[6 * r + c]) * x[c];
    } else if (!transposed) {
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int c = 0; c < 6; ++c) acc[r] += Sv[6 * r + c] * x[c];
    } else {
#pragma unroll
        for (int c = 0; c < 6; ++c)
#pragma unroll
            for (int r = 0; r < 6; ++r) acc[c] += Sv[6 * r + c] * x[r];
    }
}

// Sums of six values over the warp by recursive halving (eight adds per lane
// instead of thirty: the adds of an FP64 row sum took as long as a quarter of
// its products).  Lane l ends with the total of component fold6_comp(l); the
// additions pair the lanes as the xor butterfly 16, 8, 4, 2, 1 does, so the
// totals are its bits.
__device__ __forceinline__ int fold6_comp(int lane) {
    return ((lane & 16) ? 3 : 0) + ((lane & 8) ? 2 : ((lane & 4) ? 1 : 0));
}
__device__ __forceinline__ bool fold6_owner(int lane) { return (lane & 3) == 0 && (lane & 12) != 12; }
template <typename TV>
__device__ __forceinline__ TV warp_fold6(const TV (&a)[6], int lane) {
    const unsigned M = 0xffffffffu;
    const bool b16 = lane & 16, b8 = lane & 8, b4 = lane & 4;
    TV k[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) k[c] = (b16 ? a[3 + c] : a[c]) + __shfl_xor_sync(M, b16 ? a[c] : a[3 + c], 16);
    const TV r0 = __shfl_xor_sync(M, b8 ? k[0] : k[2], 8), r1 = __shfl_xor_sync(M, k[1], 8);
    const TV u = (b8 ? k[2] : k[0]) + r0, v = k[1] + r1;
    TV t = (b8 || !b4) ? u : v;
    t += __shfl_xor_sync(M, (b8 || b4) ? u : v, 4);
    t += __shfl_xor_sync(M, t, 2);
    t += __shfl_xor_sync(M, t, 1);
    return t;
}

// Six FP32 reductions into a camera vector (24 B, 8-byte aligned).
__device__ __forceinline__ void red_add2_f(float *a, float u, float v) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(a), "f"(u), "f"(v) : "memory");
}
__device__ __forceinline__ void red_add4_f(float *a, float u0, float u1, float u2, float u3) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(a), "f"(u0), "f"(u1), "f"(u2), "f"(u3)
                 : "memory");
}
__device__ __forceinline__ void red_add6_f(float *qj, const float (&t)[6]) {
    if ((reinterpret_cast<uintptr_t>(qj) & 15u) == 0) {
        red_add4_f(qj, t[0], t[1], t[2], t[3]);
        red_add2_f(qj + 4, t[4], t[5]);
    } else {
        red_add2_f(qj, t[0], t[1]);
        red_add4_f(qj + 2, t[2], t[3], t[4], t[5]);
    }
}
// One stored linearization row (JW values, 16-byte aligned, read-only) into
// registers with vector loads.
__device__ __forceinline__ void load_jrow(const float *__restrict__ s, float (&v)[JW]) {
    const float4 *s4 = reinterpret_cast<const float4 *>(s);
#pragma unroll
    for (int q = 0; q < JW / 4; ++q) {
        const float4 t = __ldg(s4 + q);
        v[4 * q] = t.x; v[4 * q + 1] = t.y; v[4 * q + 2] = t.z; v[4 * q + 3] = t.w;
    }
}
__device__ __forceinline__ void load_jrow(const double *__restrict__ s, double (&v)[JW]) {
    const double2 *s2 = reinterpret_cast<const double2 *>(s);
#pragma unroll
    for (int q = 0; q < JW / 2; ++q) {
        const double2 t = __ldg(s2 + q);
        v[2 * q] = t.x; v[2 * q + 1] = t.y;
    }
}

// Double-float (hi + lo, both FP32) values for reductions on the FP32 pipe:
// the sum of two is formed with an error-free TwoSum, so it is exact to about
// 2^-44 relative and, TwoSum being symmetric, a xor-butterfly gives every lane
// the same bits.
struct df32 {
    float hi, lo;
};
__device__ __forceinline__ df32 df_add(df32 a, df32 b) {
    const float s = a.hi + b.hi, bb = s - a.hi;
    float e = (a.hi - (s - bb)) + (b.hi - bb);
    e += a.lo + b.lo;
    const float hi = s + e;
    return {hi, e - (hi - s)};
}
// Products and quotients of double-floats (Dekker's two-product by FMA, one
// Newton correction of the FP32 quotient): about 2^-44 relative, within the
// FP32 exponent range.
__device__ __forceinline__ df32 df_fast_norm(float s, float e) {
    const float hi = s + e;
    return {hi, e - (hi - s)};
}
__device__ __forceinline__ df32 df_sub(df32 a, df32 b) { return df_add(a, df32{-b.hi, -b.lo}); }
__device__ __forceinline__ df32 df_mul(df32 a, df32 b) {
    const float p = a.hi * b.hi;
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
    return df_fast_norm(p, e);
}
__device__ __forceinline__ df32 df_mulf(df32 a, float b) {
    const float p = a.hi * b;
    const float e = __fmaf_rn(a.lo, b, __fmaf_rn(a.hi, b, -p));
    return df_fast_norm(p, e);
}
__device__ __forceinline__ df32 df_div(df32 a, df32 b) {
    const float q1 = a.hi / b.hi;
    float r = __fmaf_rn(-q1, b.hi, a.hi);  // exact: a.hi - q1 b.hi
    r = __fmaf_rn(-q1, b.lo, r + a.lo);
    return df_fast_norm(q1, r / b.hi);
}
__device__ __forceinline__ double df_to_double(df32 a) { return (double)a.hi + (double)a.lo; }

__device__ __forceinline__ df32 warp_sum_df(df32 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const df32 u = {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
        v = df_add(v, u);
    }
    return v;
}

// warp_fold6 for double-floats: component fold6_comp(lane) of the six sums.
__device__ __forceinline__ df32 shfl_xor_df(df32 v, int o) {
    return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ df32 warp_fold6_df(const df32 (&a)[6], int lane) {
    const bool b16 = lane & 16, b8 = lane & 8, b4 = lane & 4;
    df32 k[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) k[c] = df_add(b16 ? a[3 + c] : a[c], shfl_xor_df(b16 ? a[c] : a[3 + c], 16));
    const df32 r0 = shfl_xor_df(b8 ? k[0] : k[2], 8), r1 = shfl_xor_df(k[1], 8);
    const df32 u = df_add(b8 ? k[2] : k[0], r0), v = df_add(k[1], r1);
    df32 t = (b8 || !b4) ? u : v;
    t = df_add(t, shfl_xor_df((b8 || b4) ? u : v, 4));
    t = df_add(t, shfl_xor_df(t, 2));
    return df_add(t, shfl_xor_df(t, 1));
}

// Sum over the warp's first N lanes (a power of two), valid in lane 0.
template <int N>
__device__ __forceinline__ df32 warp_sum_df_n(df32 v) {
#pragma unroll
    for (int o = N / 2; o > 0; o >>= 1) {
        const df32 u = {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
        v = df_add(v, u);
    }
    return v;
}

// Block sum of NV double-floats over NW warps (a power of two, the whole CTA);
// the totals are valid in lane 0 of warp 0.
template <int NV, int NW>
__device__ __forceinline__ void block_sum_df(df32 (&v)[NV], float2 *sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = warp_sum_df(v[i]);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < NV; ++i) sh[w * NV + i] = make_float2(v[i].hi, v[i].lo);
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const float2 t = lane < NW ? sh[lane * NV + i] : make_float2(0.f, 0.f);
            v[i] = warp_sum_df_n<NW>(df32{t.x, t.y});
        }
    }
    __syncthreads();
}

// grid_allreduce_sym for double-floats (partials stored as float2 in the same
// slots): every CTA adds all partials itself in CTA order.  Arrivals are
// spread over AR_SUB counters, one per 128-byte line (CTA c announces itself
// on counter c % AR_SUB), so the release adds of a large grid do not queue on
// one address; lanes 0..AR_SUB-1 of warp 0 each poll one counter.  Once all
// have arrived, every thread of the CTA loads the partials of CTAs
// threadIdx.x, threadIdx.x + blockDim.x, ... (all loads of a thread issued
// before its adds, so the grid's partials cost one L2 round trip instead of
// gridDim.x / 32 dependent ones), and a block sum joins them: a fixed order
// for a given launch shape, so every CTA gets the same bits.  `bar` holds
// AR_SUB * 32 words, zero at launch; `sh` holds NV * warps float2, `s_ok` is
// shared.  Every thread of the CTA calls this (it holds __syncthreads); the
// CTA's own partial is v as left by block_sum_df (valid in thread 0).  Once
// every CTA has arrived, every thread runs after_wait() (what the grid wrote
// before arriving is visible to it) right after issuing its partial reads;
// meant for asynchronous copies that overlap the rest.  On return the
// totals are valid in thread 0 only (as double-floats); false on timeout.
template <int NV, int NW, class F>
__device__ __forceinline__ bool grid_allreduce_df(df32 (&v)[NV], double *part, unsigned gen, unsigned *bar,
                                                  int *err, long long limit_cycles, df32 (&tot)[NV], float2 *sh,
                                                  int *s_ok, F &&after_wait) {
    static_assert(NV <= AR_NV_MAX, "too many values");
    float2 *half = reinterpret_cast<float2 *>(part + (size_t)(gen & 1u) * gridDim.x * AR_NV_MAX);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) __stcg(half + blockIdx.x * AR_NV_MAX + k, make_float2(v[k].hi, v[k].lo));
        red_add_release(bar + 32 * (blockIdx.x % AR_SUB), 1u);
    }
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int lane_ok = 1;
        if (lane < AR_SUB) {
            // CTAs that announce themselves on this lane's counter
            const unsigned per = gridDim.x / AR_SUB + ((unsigned)lane < gridDim.x % AR_SUB ? 1u : 0u);
            const unsigned target = (gen + 1u) * per;
            const long long t0 = clock64();
            while (ld_acquire(bar + 32 * lane) < target) {
                if (clock64() - t0 > limit_cycles || *(volatile int *)err == (int)BA_ERR_TIMEOUT) {
                    lane_ok = 0;
                    break;
                }
            }
        }
        const bool ok = __all_sync(0xffffffffu, lane_ok) != 0;
        if (lane == 0) {
            *s_ok = ok ? 1 : 0;
            if (!ok) atomicExch(err, (int)BA_ERR_TIMEOUT);
        }
    }
    __syncthreads();  // the pollers' acquires order every thread's partial reads
    const bool ok = *s_ok != 0;
    df32 acc[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = df32{0.f, 0.f};
    if (ok) {
        const unsigned b0 = threadIdx.x, b1 = threadIdx.x + blockDim.x;
        float2 t0[NV], t1[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            t0[k] = b0 < gridDim.x ? __ldcg(half + b0 * AR_NV_MAX + k) : make_float2(0.f, 0.f);
            t1[k] = b1 < gridDim.x ? __ldcg(half + b1 * AR_NV_MAX + k) : make_float2(0.f, 0.f);
        }
        after_wait();  // issued behind the partial reads, overlapping their use
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            acc[k] = df_add(df32{t0[k].x, t0[k].y}, df32{t1[k].x, t1[k].y});
        }
        for (unsigned b = threadIdx.x + 2 * blockDim.x; b < gridDim.x; b += blockDim.x)
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const float2 u = __ldcg(half + b * AR_NV_MAX + k);
                acc[k] = df_add(acc[k], df32{u.x, u.y});
            }
    }
    block_sum_df<NV, NW>(acc, sh);
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) tot[k] = acc[k];
    return ok;
}

}  // namespace ba
