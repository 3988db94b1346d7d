// Variable-size BSMC (Sec. 4, Fig. 4: block (i, j) is c_i x c_j; c = 11 with
// five interior unknowns in Sec. 4.1): storage, the two-sided product of
// Sec. 6.2 (Fig. 13) and the block-Jacobi PCG of Sec. 3.2 (Eqs. 6-7), behind
// the ba_vbsmc_* calls of ba_vbsmc.h.
//
// Device layout: the upper blocks packed in row order (block k at value
// offset boff[k], row-major c_row x c_col), a column per block, row starts,
// block sizes cdim and vector offsets off (camera i's entries are
// off[i] .. off[i] + c_i - 1).  The product runs from two-sided entry lists
// built on the host: row i lists its stored blocks, then the blocks of its
// column in the rows above it, flagged "transposed" (one 16-byte record per
// entry); so every row is summed by one warp with no atomics, in a fixed
// order.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "device_util.cuh"
#include "vbsmc_internal.h"

namespace ba {

// One part of a row's product.  The warp's lanes form G groups of c_i lanes
// (at most min(32 / c_i, 5)); group g takes entries e0 + g, e0 + g + step, ... below
// e1, its lane a component a of the row.  The group stages the entry's c_j
// values of x (each formed once, gx(index)) in the warp's shared memory sx and
// holds the lane's row (or column) of the block in registers, so an entry
// costs c_j multiply-adds per lane and one evaluation of x per value.  An
// entry's record rec[e] is (value offset lo / hi, vector offset of j,
// c_j << 1 | transposed).  Lanes 0 .. c_i - 1 return the part's sum.
// (The first version gave every entry 16 lanes, evaluated x in each of them
// and ran 16 columns whatever c_j: in FP64, where a warp instruction takes 16
// cycles of its SM, 32 per pair of entries instead of 12 at c = 11.)
constexpr int VB_GROUPS = 5;
// The row products of the owning PCG (k_vb_pcg_own): FP32 always in two groups (every c_i <= 16 allows
// them), so that the order of a row's additions does not depend on c_i and an
// FP32 system with six-unknown cameras keeps the bits of its iterates, on which
// an LM trajectory rests (1,984 cameras, half of them c = 6: 24.1 us per iteration,
// 22.8 with as many groups as fit; nothing to lose at c = 11); FP64 in as many as
// fit (its issue rate is the limit).  k_vb_pcg, for larger systems, takes as many
// as fit in both (20,000 cameras of c = 6, FP32: 460 us for four iterations, 884
// with two).
template <typename T>
__host__ __device__ constexpr int vb_pcg_groups(int ci) {
    return 32 / ci < (sizeof(T) == 4 ? 2 : VB_GROUPS) ? 32 / ci : (sizeof(T) == 4 ? 2 : VB_GROUPS);
}
// One entry's row (or column) of values in registers, zero beyond c_j.
template <typename T>
__device__ __forceinline__ void vb_load(int ci, int a, const int4 in, const T *__restrict__ val, T (&bv)[BA_VB_CMAX]) {
    const int cj = in.w >> 1;
    const T *Bp = val + ((int64_t)(uint32_t)in.x | ((int64_t)in.y << 32)) + ((in.w & 1) ? a : a * cj);
    const int stride = (in.w & 1) ? ci : 1;
#pragma unroll
    for (int c = 0; c < BA_VB_CMAX; ++c) {
        bv[c] = T(0);
        if (c < cj) bv[c] = __ldg(Bp + c * stride);
    }
}
// The groups' sums joined: lanes 0 .. c_i - 1 return the part's sum.
template <typename T>
__device__ __forceinline__ T vb_join(T acc, int ci, int G, int a) {
    T tot = acc;
    for (int h = 1; h < G; ++h) tot += __shfl_sync(0xffffffffu, acc, (a + h * ci) & 31);
    return tot;
}
template <typename T, class GX>
__device__ __forceinline__ T vb_part(int ci, int G, int e0, int e1, int step, const int4 *__restrict__ rec,
                                     const T *__restrict__ val, T *sx, GX gx) {
    const int lane = threadIdx.x & 31;
    const int g = lane / ci, a = lane - g * ci;
    T acc = T(0);
    for (int t = e0; t < e1; t += step) {
        const int e = t + g;
        int4 in = make_int4(0, 0, 0, 0);
        if (g < G && e < e1) in = __ldg(rec + e);
        const int cj = in.w >> 1;
        T bv[BA_VB_CMAX];
        vb_load<T>(ci, a, in, val, bv);
        for (int c = a; c < cj; c += ci) sx[BA_VB_CMAX * g + c] = gx(in.z + c);
        const int cm = (int)__reduce_max_sync(0xffffffffu, (unsigned)cj);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < BA_VB_CMAX; ++c) {
            if (c >= cm) break;
            acc = fma(bv[c], c < cj ? sx[BA_VB_CMAX * g + c] : T(0), acc);
        }
        __syncwarp();
    }
    return vb_join<T>(acc, ci, G, a);
}
// The same with every entry's x already in shared memory (sx, 16 values per
// entry).  PACKED: the values too, each block by columns of this row's form
// (element (a, c) at in.x + c c_i + a); otherwise the next pass's values are
// loaded while this one's are used.
template <typename T, bool PACKED>
__device__ __forceinline__ T vb_own_part(int ci, int e0, int e1, int step, const int4 *rec, const T *val,
                                         const T *sx) {
    const int lane = threadIdx.x & 31;
    const int G = vb_pcg_groups<T>(ci), g = lane / ci, a = lane - g * ci;
    T acc = T(0);
    // all of a pass's loads are issued before its multiply-adds (columns beyond
    // c_j read as zeros; FP32 multiplies them, FP64 stops at the warp's
    // largest c_j)
    auto apply = [&](const T(&bv)[BA_VB_CMAX], const T(&xv)[BA_VB_CMAX], int cj) {
        if constexpr (sizeof(T) == 8) {
            const int cm = (int)__reduce_max_sync(0xffffffffu, (unsigned)cj);
#pragma unroll
            for (int c = 0; c < BA_VB_CMAX; ++c) {
                if (c >= cm) break;
                acc = fma(bv[c], xv[c], acc);
            }
        } else {
#pragma unroll
            for (int c = 0; c < BA_VB_CMAX; ++c) acc = fma(bv[c], xv[c], acc);
        }
    };
    auto load_x = [&](bool on, int e, T(&xv)[BA_VB_CMAX]) {
        using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
        constexpr int N = 16 / (int)sizeof(T);
        const V *xp = reinterpret_cast<const V *>(sx + BA_VB_CMAX * e);
#pragma unroll
        for (int k = 0; k < BA_VB_CMAX / N; ++k) {
            V v;
            memset(&v, 0, sizeof(V));
            if (on) v = xp[k];
            memcpy(&xv[N * k], &v, sizeof(V));
        }
    };
    if (PACKED) {
        for (int t = e0; t < e1; t += step) {
            const int e = t + g;
            const bool on = g < G && e < e1;
            int4 in = make_int4(0, 0, 0, 0);
            if (on) in = rec[e];
            const int cj = in.w >> 1;
            const T *Bp = val + in.x + a;
            T bv[BA_VB_CMAX], xv[BA_VB_CMAX];
#pragma unroll
            for (int c = 0; c < BA_VB_CMAX; ++c) {
                bv[c] = T(0);
                if (c < cj) bv[c] = Bp[c * ci];
            }
            load_x(on, e, xv);
            apply(bv, xv, cj);
        }
    } else {
        T bn[BA_VB_CMAX];
        int4 in = make_int4(0, 0, 0, 0);
        if (g < G && e0 + g < e1) in = rec[e0 + g];
        vb_load<T>(ci, a, in, val, bn);
        for (int t = e0; t < e1; t += step) {
            T bv[BA_VB_CMAX], xv[BA_VB_CMAX];
#pragma unroll
            for (int c = 0; c < BA_VB_CMAX; ++c) bv[c] = bn[c];
            const int cj = in.w >> 1;
            const bool on = g < G && t + g < e1;
            in = make_int4(0, 0, 0, 0);
            if (g < G && t + step + g < e1) in = rec[t + step + g];
            vb_load<T>(ci, a, in, val, bn);
            load_x(on, t + g, xv);
            apply(bv, xv, cj);
        }
    }
    return vb_join<T>(acc, ci, G, a);
}

// y = S x: `wpr` warps of the CTA's eight to a row, so that systems of few
// rows still fill the SMs with loads in flight; the parts of a row are added
// in order.
template <typename T>
__global__ void __launch_bounds__(256) k_vb_spmv(int n, int wpr, const int *__restrict__ cdim,
                                                 const int *__restrict__ off, const int *__restrict__ tw_ptr,
                                                 const int4 *__restrict__ tw_info, const T *__restrict__ val,
                                                 const T *__restrict__ x, T *__restrict__ y) {
    __shared__ T s_x[8][VB_GROUPS * BA_VB_CMAX];
    __shared__ T s_part[8][BA_VB_CMAX];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int rows = 8 / wpr, lr = w / wpr, part = w - lr * wpr;
    for (int base = blockIdx.x * rows; base < n; base += gridDim.x * rows) {
        const int i = base + lr;
        int ci = 1;
        if (i < n) {
            ci = __ldg(cdim + i);
            const int G = min(32 / ci, VB_GROUPS), e0 = __ldg(tw_ptr + i), e1 = __ldg(tw_ptr + i + 1);
            const T t = vb_part<T>(ci, G, e0 + part * G, e1, wpr * G, tw_info, val, s_x[w],
                                          [&](int k) { return __ldg(x + k); });
            if (wpr == 1) {
                if (lane < ci) y[__ldg(off + i) + lane] = t;
            } else if (lane < ci) {
                s_part[w][lane] = t;
            }
        }
        if (wpr > 1) {
            __syncthreads();
            if (part == 0 && i < n && lane < ci) {
                T t = s_part[w][lane];
                for (int q = 1; q < wpr; ++q) t += s_part[w + q][lane];
                y[__ldg(off + i) + lane] = t;
            }
            __syncthreads();
        }
    }
}

// M^-1 per camera, sixteen lanes each, in FP64: lane r holds row r of the
// (symmetrised) diagonal block, the Cholesky factor is formed column by column
// (right-looking, the pivot column passed by shuffles), then lane q solves for
// column q of the inverse.  A block that is not positive definite sets
// BA_ERR_NOT_SPD and leaves zeros.  (A thread per camera, its factor in local
// memory, was one serial FP64 chain: 260 us at 990 and at 120 cameras of c =
// 11, against 21 us.)
template <typename T>
__global__ void __launch_bounds__(64) k_vb_minv(int n, const int *__restrict__ cdim, const int *__restrict__ row_ptr,
                                                const int64_t *__restrict__ boff, const T *__restrict__ val,
                                                const int64_t *__restrict__ moff, T *__restrict__ Minv, int *err) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int CM = BA_VB_CMAX;
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 4, r = threadIdx.x & 15;
    const int c = i < n ? cdim[i] : 0;
    const int cm = (int)__reduce_max_sync(FULL, (unsigned)c);
    const T *D = val + (i < n ? boff[row_ptr[i]] : 0);
    // a / b with inv = 1 / b: the quotient for FP64; for values stored in FP32
    // the product, whose one rounding of 2^-53 more is not seen there (5,000
    // cameras of c = 11: 43 us less)
    auto over = [](double a, double b, double inv) { return sizeof(T) == 4 ? a * inv : quotient(a, b, inv); };
    double A[CM], invd = 1.0;
#pragma unroll
    for (int q = 0; q < CM; ++q)
        A[q] = r < c && q < c ? 0.5 * ((double)D[r * c + q] + (double)D[q * c + r]) : 0.0;
    bool ok = true;
#pragma unroll
    for (int q = 0; q < CM; ++q) {
        if (q >= cm) break;
        double p = __shfl_sync(FULL, A[q], q, 16);
        if (!(p > 0.0)) {
            ok = ok && q >= c;
            p = 1.0;
        }
        const double d = sqrt(p), inv = 1.0 / d;
        if (r == q) invd = inv;
        A[q] = r == q ? d : over(A[q], d, inv);
#pragma unroll
        for (int k = q + 1; k < CM; ++k) {
            if (k >= cm) break;
            A[k] -= A[q] * __shfl_sync(FULL, A[q], k, 16);  // rows r >= k of column k are meant
        }
    }
    // column r of (L L^T)^-1: forward, then backward substitution on e_r
    double x[CM];
#pragma unroll
    for (int q = 0; q < CM; ++q) {
        x[q] = 0.0;
        if (q < cm) {
            double s = r == q ? 1.0 : 0.0;
#pragma unroll
            for (int k = 0; k < q; ++k) s -= __shfl_sync(FULL, A[k], q, 16) * x[k];
            x[q] = over(s, __shfl_sync(FULL, A[q], q, 16), __shfl_sync(FULL, invd, q, 16));
        }
    }
#pragma unroll
    for (int q = CM - 1; q >= 0; --q) {
        if (q < cm) {
            double s = x[q];
#pragma unroll
            for (int k = q + 1; k < CM; ++k)
                if (k < cm) s -= __shfl_sync(FULL, A[q], k, 16) * x[k];
            x[q] = over(s, __shfl_sync(FULL, A[q], q, 16), __shfl_sync(FULL, invd, q, 16));
        }
    }
    if (!ok && r == 0) atomicExch(err, (int)BA_ERR_NOT_SPD);
    if (r < c) {
        T *M = Minv + moff[i];
#pragma unroll
        for (int q = 0; q < CM; ++q)
            if (q < c) M[q * c + r] = ok ? (T)x[q] : T(0);
    }
}

// The PCG of Sec. 3.2 with a CTA owning a contiguous run of block rows: `wpr`
// warps share a row's product (units of row and part, taken round-robin by the
// CTA's warps), and thread t keeps y, r, z, d and its row of M^-1 of the CTA's
// t-th vector entry in registers for the whole solve; only z and d pass
// through memory; the neighbours' d is gathered once per iteration into shared
// memory.  The entries' records, and with PACKED the values too (by columns, so
// the lanes of a group read consecutive words), are copied there once.  Two
// grid exchanges per iteration, run by one warp, which also forms alpha and
// beta; every wait is bounded (BA_ERR_TIMEOUT).
// What bounds it: in FP64 the SM's FP64 issue (one warp instruction per 16
// cycles), spread over every SM and its four schedulers; in FP32 the two
// exchanges and the reads of S.  Against one warp per row on n / 8 SMs and
// vectors in memory, c = 11, us per iteration: FP64 61.7 -> 10.9 at 120 cameras,
// 115 -> 50 at 1,984 (values in L2); FP32 32 -> 10.3 at 120, 33.4 -> 13.7 at
// 990 (22 with the neighbours' values gathered pass by pass), 38.7 -> 22.5 at
// 1,984 (values in L2).
template <typename T>
__host__ __device__ constexpr size_t vb_own_smem(int rows, int wpr, int max_ent, int64_t max_val, int threads) {
    return (size_t)max_ent * sizeof(int4) +
           ((size_t)max_val + (size_t)rows * wpr * BA_VB_CMAX + (size_t)max_ent * BA_VB_CMAX + threads) * sizeof(T) +
           (size_t)(2 * rows + 2) * sizeof(int);
}
template <typename T>
__host__ __device__ constexpr int vb_own_threads() {
    return sizeof(T) == 4 ? 512 : 256;
}
template <typename T, bool PACKED>
__global__ void __launch_bounds__(vb_own_threads<T>(), 1)
    k_vb_pcg_own(int n, VbPlan pl, const int *__restrict__ cdim, const int *__restrict__ off,
                 const int *__restrict__ ent_cam, const int *__restrict__ tw_ptr, const int4 *__restrict__ tw_info,
                 const T *__restrict__ val, const int64_t *__restrict__ moff, const T *__restrict__ Minv,
                 const T *__restrict__ b, T *y, T *z, T *d0, T *d1, VbScalars *sc, double *red, unsigned *bar,
                 long long limit_cycles) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ double s_ab;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int row0 = blockIdx.x * pl.rows, R = min(pl.rows, n - row0);
    int4 *s_rec = reinterpret_cast<int4 *>(sm_raw);
    // s_x is read by 16-byte loads: it follows the 16-byte records, and its
    // stride of BA_VB_CMAX values is a multiple of 16 bytes; the rest is read
    // by single values
    T *s_x = reinterpret_cast<T *>(s_rec + pl.max_ent);
    T *s_part = s_x + (size_t)pl.max_ent * BA_VB_CMAX;
    T *s_r = s_part + (size_t)pl.rows * pl.wpr * BA_VB_CMAX;
    T *s_val = s_r + blockDim.x;
    int *s_e = reinterpret_cast<int *>(s_val + pl.max_val), *s_c = s_e + pl.rows + 1;
    const int t0 = __ldg(tw_ptr + row0), ne = __ldg(tw_ptr + row0 + R) - t0;
    for (int q = threadIdx.x; q <= R; q += blockDim.x) {
        s_e[q] = __ldg(tw_ptr + row0 + q) - t0;
        if (q < R) s_c[q] = __ldg(cdim + row0 + q);
    }
    for (int q = threadIdx.x; q < ne; q += blockDim.x) s_rec[q] = __ldg(tw_info + t0 + q);
    __syncthreads();
    if (PACKED) {
        // packed offsets (warp 0, running sum of the blocks' sizes), then the
        // values by columns, a warp per entry
        if (w == 0) {
            int base = 0, lr = 0;
            for (int q0 = 0; q0 < ne; q0 += 32) {
                const int q = q0 + lane;
                int sz = 0;
                if (q < ne) {
                    while (q >= s_e[lr + 1]) ++lr;
                    sz = s_c[lr] * (s_rec[q].w >> 1);
                }
                int inc = sz;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += u;
                }
                // the offset rides in w's upper bits until the values are copied
                if (q < ne) s_rec[q].w |= (base + inc - sz) << 8;
                base += __shfl_sync(0xffffffffu, inc, 31);
            }
        }
        __syncthreads();
        for (int q = w; q < ne; q += W) {
            int lr = 0;
            while (q >= s_e[lr + 1]) ++lr;
            const int ci = s_c[lr];
            const int4 in = s_rec[q];
            const int cj = (in.w & 0xff) >> 1, po = in.w >> 8;
            const T *B = val + ((int64_t)(uint32_t)in.x | ((int64_t)in.y << 32));
            for (int k = lane; k < ci * cj; k += 32) {
                const int c = k / ci, a = k - c * ci;
                s_val[po + k] = (in.w & 1) ? __ldg(B + k) : __ldg(B + a * cj + c);
            }
            __syncwarp();
            if (lane == 0) s_rec[q] = make_int4(po, 0, in.z, in.w & 0xff);
        }
        __syncthreads();
    }
    // this thread's vector entry
    const int v0 = __ldg(off + row0), NE = __ldg(off + row0 + R) - v0;
    const int nwv = (NE + 31) >> 5;
    const bool own = (int)threadIdx.x < NE;
    const int e = v0 + threadIdx.x;
    int lrow = 0, comp = 0, cown = 0;
    T Mr[BA_VB_CMAX], rv = T(0), yv = T(0), zv = T(0), dv = T(0);
#pragma unroll
    for (int k = 0; k < BA_VB_CMAX; ++k) Mr[k] = T(0);
    if (own) {
        const int i = __ldg(ent_cam + e);
        lrow = i - row0;
        comp = e - __ldg(off + i);
        cown = __ldg(cdim + i);
        const T *M = Minv + __ldg(moff + i) + (int64_t)comp * cown;
#pragma unroll
        for (int k = 0; k < BA_VB_CMAX; ++k)
            if (k < cown) Mr[k] = __ldg(M + k);
        rv = __ldg(b + e);
        s_r[threadIdx.x] = rv;
        d0[e] = T(0);
    }
    __syncthreads();
    const T *r6 = s_r + threadIdx.x - comp;  // the camera's residual entries
    auto precond = [&]() {
        T s = T(0);
#pragma unroll
        for (int k = 0; k < BA_VB_CMAX; ++k)
            if (k < cown) s = fma(Mr[k], r6[k], s);
        return s;
    };
    const double tol2 = sc->tol2;
    const int max_iters = sc->max_iters;
    unsigned gen = 0;
    double v2[2] = {0.0, 0.0};
    if (own) {
        zv = precond();
        z[e] = zv;
        v2[0] = (double)(rv * zv);
        v2[1] = (double)(rv * rv);
    }
    auto none = [](const double (&)[2], bool) {};
    if (!grid_allreduce_w0<2>(v2, red, gen++, bar, &sc->err, limit_cycles, nwv, none)) return;
    double rz = v2[0];
    const double rr0 = v2[1];
    if (!(rr0 > 0.0) || max_iters <= 0) {
        if (own) y[e] = T(0);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            sc->rr0 = rr0;
            sc->rr = rr0;
            sc->iters = 0;
            sc->done = 1;
        }
        return;
    }
    T bt = T(0);
    const int units = R * pl.wpr;
    for (int it = 0;;) {
        const T *dold = (it & 1) ? d1 : d0;
        T *dnew = (it & 1) ? d0 : d1;
        // every entry's x = z + beta d, sixteen lanes to an entry, four entries'
        // loads in flight per lane (their round trips to L2 would otherwise
        // follow one another in the rows' loops)
        for (int q0 = threadIdx.x >> 4; q0 < ne; q0 += 4 * (blockDim.x >> 4)) {
            T zz[4], dd[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int q = q0 + k * (blockDim.x >> 4), c = threadIdx.x & 15;
                zz[k] = dd[k] = T(0);
                if (q < ne) {
                    const int4 in = s_rec[q];
                    if (c < (in.w >> 1)) {
                        zz[k] = __ldcg(z + in.z + c);
                        dd[k] = __ldcg(dold + in.z + c);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int q = q0 + k * (blockDim.x >> 4);
                if (q < ne) s_x[BA_VB_CMAX * q + (threadIdx.x & 15)] = fma(bt, dd[k], zz[k]);
            }
        }
        __syncthreads();
        for (int u = w; u < units; u += W) {
            const int lr = u / pl.wpr, ci = s_c[lr], G = vb_pcg_groups<T>(ci);
            const T t = vb_own_part<T, PACKED>(ci, s_e[lr] + (u - lr * pl.wpr) * G, s_e[lr + 1], pl.wpr * G, s_rec,
                                               PACKED ? s_val : val, s_x);
            if (lane < ci) s_part[u * BA_VB_CMAX + lane] = t;
        }
        __syncthreads();
        T q = T(0);
        double v1[1] = {0.0};
        if (own) {
            const T *sp = s_part + lrow * pl.wpr * BA_VB_CMAX + comp;
            q = sp[0];
            for (int p = 1; p < pl.wpr; ++p) q += sp[p * BA_VB_CMAX];
            dv = fma(bt, dv, zv);
            dnew[e] = dv;
            v1[0] = (double)(dv * q);
        }
        if (!grid_allreduce_w0<1>(v1, red, gen++, bar, &sc->err, limit_cycles, nwv,
                                  [&](const double(&x)[1], bool) { s_ab = rz / x[0]; }))
            return;
        if (!(v1[0] > 0.0)) {
            if (own) y[e] = yv;
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                sc->err = (int)BA_ERR_NOT_SPD;
                sc->done = 1;
                sc->iters = it;
            }
            return;
        }
        const T alpha = (T)s_ab;
        if (own) {
            rv -= alpha * q;
            yv += alpha * dv;
            s_r[threadIdx.x] = rv;
        }
        __syncthreads();
        v2[0] = v2[1] = 0.0;
        if (own) {
            zv = precond();
            z[e] = zv;
            v2[0] = (double)(rv * zv);
            v2[1] = (double)(rv * rv);
        }
        if (!grid_allreduce_w0<2>(v2, red, gen++, bar, &sc->err, limit_cycles, nwv,
                                  [&](const double(&x)[2], bool) { s_ab = x[0] / rz; }))
            return;
        ++it;
        if (v2[1] <= tol2 * rr0 || it >= max_iters) {
            if (own) y[e] = yv;
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                sc->iters = it;
                sc->rr = v2[1];
                sc->rr0 = rr0;
                sc->rz = v2[0];
                sc->done = 1;
            }
            return;
        }
        bt = (T)s_ab;
        rz = v2[0];
    }
}

// z_e = (M^-1_i v_i)[a] for vector entry e = off[i] + a, where v_i[c] = g(off[i] + c).
template <typename T, class G>
__device__ __forceinline__ T vb_precond_entry(int i, int a, const int *__restrict__ cdim, const int *__restrict__ off,
                                              const int64_t *__restrict__ moff, const T *__restrict__ Minv, G g) {
    const int c = __ldg(cdim + i), o = __ldg(off + i);
    const T *M = Minv + __ldg(moff + i) + (int64_t)a * c;
    T z = T(0);
    for (int k = 0; k < c; ++k) z += __ldg(M + k) * g(o + k);
    return z;
}

// The same for systems whose CTAs would own more entries than threads (vectors
// in memory, a warp per row):
// the start (r = b, z = M^-1 b, y = 0) and r^T z, r^T r by one all-reduce;
// then per iteration the product phase (d = z + beta d_old formed on the fly,
// q = S d, d^T S d), its all-reduce, the update phase (y += alpha d,
// r -= alpha q, z = M^-1 r, r^T z, r^T r) and its all-reduce.  Every grid wait
// is bounded (BA_ERR_TIMEOUT).
template <typename T>
__global__ void __launch_bounds__(256) k_vb_pcg(int n, int N, const int *__restrict__ cdim, const int *__restrict__ off,
                                                const int *__restrict__ ent_cam, const int *__restrict__ tw_ptr,
                                                const int4 *__restrict__ tw_info, const T *__restrict__ val,
                                                const int64_t *__restrict__ moff,
                                                const T *__restrict__ Minv, const T *__restrict__ b, T *y, T *r0, T *r1,
                                                T *z, T *d0, T *d1, T *q, VbScalars *sc, double *red, unsigned *bar,
                                                long long limit_cycles) {
    __shared__ T s_x[8][VB_GROUPS * BA_VB_CMAX];
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const double tol2 = sc->tol2;
    const int max_iters = sc->max_iters;
    unsigned gen = 0;
    double v0[2] = {0.0, 0.0};
    for (int e = tid; e < N; e += nth) {
        const int i = __ldg(ent_cam + e);
        const T ze = vb_precond_entry<T>(i, e - __ldg(off + i), cdim, off, moff, Minv, [&](int k) { return __ldg(b + k); });
        const T be = __ldg(b + e);
        r0[e] = be;
        z[e] = ze;
        y[e] = T(0);
        d0[e] = T(0);
        v0[0] += (double)(be * ze);
        v0[1] += (double)(be * be);
    }
    if (!grid_allreduce_w0<2>(v0, red, gen++, bar, &sc->err, limit_cycles)) return;
    double rz = v0[0];
    const double rr0 = v0[1];
    if (!(rr0 > 0.0) || max_iters <= 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            sc->rr0 = rr0;
            sc->rr = rr0;
            sc->iters = 0;
            sc->done = 1;
        }
        return;
    }
    double beta = 0.0;
    int it = 0;
    const int nw = nth >> 5;
    for (;;) {
        const bool odd = it & 1;
        T *dold = odd ? d1 : d0, *dnew = odd ? d0 : d1;
        T *rc = odd ? r1 : r0, *rn = odd ? r0 : r1;
        const T bt = (T)beta;
        auto dir = [&](int k) { return __ldcg(z + k) + bt * __ldcg(dold + k); };
        T pap_t = T(0);
        for (int i = tid >> 5; i < n; i += nw) {
            const int ci = __ldg(cdim + i), lane = threadIdx.x & 31;
            const int G = min(32 / ci, VB_GROUPS);
            const T v = vb_part<T>(ci, G, __ldg(tw_ptr + i), __ldg(tw_ptr + i + 1), G, tw_info, val, s_x[threadIdx.x >> 5], dir);
            if (lane < ci) {
                const int idx = __ldg(off + i) + lane;
                const T dv = dir(idx);
                q[idx] = v;
                dnew[idx] = dv;
                pap_t += dv * v;
            }
        }
        double v1[1] = {(double)pap_t};
        if (!grid_allreduce_w0<1>(v1, red, gen++, bar, &sc->err, limit_cycles)) return;
        const double pAp = v1[0];
        if (!(pAp > 0.0)) {
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                sc->err = (int)BA_ERR_NOT_SPD;
                sc->done = 1;
                sc->iters = it;
            }
            return;
        }
        const T alpha = (T)(rz / pAp);
        double v2[2] = {0.0, 0.0};
        for (int e = tid; e < N; e += nth) {
            const int i = __ldg(ent_cam + e);
            const T ze = vb_precond_entry<T>(i, e - __ldg(off + i), cdim, off, moff, Minv,
                                             [&](int k) { return __ldcg(rc + k) - alpha * __ldcg(q + k); });
            const T ra = __ldcg(rc + e) - alpha * __ldcg(q + e);
            y[e] += alpha * __ldcg(dnew + e);
            rn[e] = ra;
            z[e] = ze;
            v2[0] += (double)(ra * ze);
            v2[1] += (double)(ra * ra);
        }
        if (!grid_allreduce_w0<2>(v2, red, gen++, bar, &sc->err, limit_cycles)) return;
        const double rz_new = v2[0], rr = v2[1];
        ++it;
        if (rr <= tol2 * rr0 || it >= max_iters) {
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                sc->iters = it;
                sc->rr = rr;
                sc->rr0 = rr0;
                sc->rz = rz_new;
                sc->done = 1;
            }
            return;
        }
        beta = rz_new / rz;
        rz = rz_new;
    }
}

}  // namespace ba

using namespace ba;

namespace ba {

ba_status vb_alloc(ba_vbsmc *h, void **d, size_t bytes) {
    bytes = bytes < 16 ? 16 : bytes;
    if (h->cap && h->dev_bytes + bytes > h->cap) return set_error(BA_ERR_OOM, "device_mem_cap reached");
    cudaError_t e = cudaMalloc(d, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return set_error(BA_ERR_OOM, "cudaMalloc failed");
    }
    if (e != cudaSuccess) return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    h->allocs.push_back(*d);
    h->dev_bytes += bytes;
    return BA_OK;
}

ba_status vb_cuda(ba_vbsmc *h, cudaError_t e, const char *what) {
    if (e == cudaSuccess) return BA_OK;
    h->dead = true;
    return set_error(BA_ERR_CUDA, (std::string(what) + ": " + cudaGetErrorString(e)).c_str());
}

}  // namespace ba

namespace {

template <typename T>
ba_status vb_upload(ba_vbsmc *h, void *dst, const double *src, size_t cnt) {
    std::vector<T> tmp(cnt);
    for (size_t k = 0; k < cnt; ++k) tmp[k] = (T)src[k];
    return vb_cuda(h, cudaMemcpy(dst, tmp.data(), cnt * sizeof(T), cudaMemcpyHostToDevice), "upload");
}

template <typename T>
cudaError_t vb_spmv_T(ba_vbsmc *h, const T *x, T *y) {
    int per_sm = 0, n_sm = 0;
    cudaError_t e = occupancy((const void *)k_vb_spmv<T>, 256, 0, &per_sm, &n_sm);
    if (e != cudaSuccess) return e;
    per_sm = std::max(per_sm, 1);
    // warps per row: as many as leave the resident warps one row part each
    int wpr = 1;
    while (wpr < 8 && (int64_t)h->n * wpr * 2 <= (int64_t)per_sm * n_sm * 8) wpr *= 2;
    const int rows = 8 / wpr;
    const int grid = std::min((h->n + rows - 1) / rows, per_sm * n_sm);
    k_vb_spmv<T><<<grid, 256, 0, h->st>>>(h->n, wpr, h->cdim, h->off, h->tw_ptr, h->tw_info, (const T *)h->val, x, y);
    return cudaGetLastError();
}

// The owning kernel's launch shape: rows spread over every SM; 8 warps per CTA
// in FP64 (its FP64 issue is the limit), 16 in FP32.
// Not taken (grid 0) when a CTA would own more entries than threads or its
// records and vectors do not fit in shared memory.
constexpr size_t VB_SMEM_MAX = 225 * 1024;
template <typename T>
VbPlan vb_own_plan(int n, int n_sm, const int32_t *cdim, const std::vector<int32_t> &tw_ptr,
                   const std::vector<int4> &tw_info) {
    const int R = (n + n_sm - 1) / n_sm;
    int max_ent = 0, max_vec = 0, row_ent = 0, max_dim = 1;
    int64_t max_val = 0;
    for (int r0 = 0; r0 < n; r0 += R) {
        int ent = 0, vec = 0;
        int64_t val = 0;
        for (int i = r0; i < std::min(n, r0 + R); ++i) {
            int64_t cols = 0;
            for (int32_t t = tw_ptr[i]; t < tw_ptr[i + 1]; ++t) cols += tw_info[t].w >> 1;
            ent += tw_ptr[i + 1] - tw_ptr[i];
            val += cols * cdim[i];
            vec += cdim[i];
            row_ent = std::max(row_ent, tw_ptr[i + 1] - tw_ptr[i]);
            max_dim = std::max(max_dim, cdim[i]);
        }
        max_ent = std::max(max_ent, ent);
        max_vec = std::max(max_vec, vec);
        max_val = std::max(max_val, val);
    }
    const int nt = vb_own_threads<T>(), W = nt / 32;
    VbPlan pl;
    if (max_vec > nt) return pl;
    const int G = vb_pcg_groups<T>(max_dim);
    // FP32: one warp per row (a row's sum keeps its order, and more warps gained
    // 3 us of 10 at 120 cameras, nothing from 990 on); FP64: the split with the
    // fewest passes (18.3, 13.5, 11.2, 10.9 us per iteration with 1, 2, 4, 8
    // warps per row at 120 cameras)
    int best = 1, best_cost = INT32_MAX;
    for (int wpr = 1; sizeof(T) == 8 && wpr <= W; wpr *= 2) {
        const int cost = ((R * wpr + W - 1) / W) * ((row_ent + wpr * G - 1) / (wpr * G) + 1);
        if (cost < best_cost) {
            best = wpr;
            best_cost = cost;
        }
    }
    pl.packed = max_val < (1 << 22) && vb_own_smem<T>(R, best, max_ent, max_val, nt) <= VB_SMEM_MAX;
    pl.smem = vb_own_smem<T>(R, best, max_ent, pl.packed ? max_val : 0, nt);
    if (pl.smem > VB_SMEM_MAX) return pl;
    pl.rows = R;
    pl.wpr = best;
    pl.max_ent = max_ent;
    pl.max_val = pl.packed ? max_val : 0;
    pl.grid = (n + R - 1) / R;
    pl.threads = nt;
    return pl;
}

template <typename T>
cudaError_t vb_pcg_own(ba_vbsmc *h, long long limit) {
    VbPlan pl = h->plan;
    const void *k = pl.packed ? (const void *)k_vb_pcg_own<T, true> : (const void *)k_vb_pcg_own<T, false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)VB_SMEM_MAX);
    if (e != cudaSuccess) return e;
    int n = h->n;
    const int *cd = h->cdim, *of = h->off, *ec = h->ent_cam, *twp = h->tw_ptr;
    const int4 *twi = h->tw_info;
    const int64_t *mo = h->moff;
    const T *val = (const T *)h->val, *Mi = (const T *)h->Minv, *b = (const T *)h->b;
    T *y = (T *)h->vec[0], *z = (T *)h->vec[3], *d0 = (T *)h->vec[4], *d1 = (T *)h->vec[5];
    VbScalars *sc = h->sc;
    double *red = h->red;
    unsigned *bar = h->bar;
    void *args[] = {&n, &pl, &cd, &of, &ec, &twp, &twi, &val, &mo, &Mi, &b, &y, &z, &d0, &d1, &sc, &red, &bar, &limit};
    return cudaLaunchCooperativeKernel(k, dim3(pl.grid), dim3(pl.threads), args, pl.smem, h->st);
}

template <typename T>
cudaError_t vb_pcg_T(ba_vbsmc *h) {
    int per_sm = 0, n_sm = 0;
    cudaError_t e = occupancy((const void *)k_vb_pcg<T>, 256, 0, &per_sm, &n_sm);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(h->bar, 0, AR_SUB * 32 * sizeof(unsigned), h->st)) != cudaSuccess) return e;
    long long limit = 4000000000LL;  // ~2 s of SM clock per grid wait
    if (h->plan.grid > 0) return vb_pcg_own<T>(h, limit);
    if (per_sm > 2) per_sm = 2;
    if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
    const int64_t want = std::max<int64_t>(((int64_t)h->n * 32 + 255) / 256, (h->N + 255) / 256);
    int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)per_sm * n_sm));
    int n = h->n, N = (int)h->N;
    const int *cd = h->cdim, *of = h->off, *ec = h->ent_cam, *twp = h->tw_ptr;
    const int4 *twi = h->tw_info;
    const int64_t *mo = h->moff;
    const T *val = (const T *)h->val, *Mi = (const T *)h->Minv, *b = (const T *)h->b;
    T *y = (T *)h->vec[0], *r0 = (T *)h->vec[1], *r1 = (T *)h->vec[2], *z = (T *)h->vec[3], *d0 = (T *)h->vec[4],
      *d1 = (T *)h->vec[5], *q = (T *)h->vec[6];
    VbScalars *sc = h->sc;
    double *red = h->red;
    unsigned *bar = h->bar;
    void *args[] = {&n, &N, &cd, &of, &ec, &twp, &twi, &val, &mo, &Mi, &b, &y, &r0, &r1, &z, &d0, &d1, &q,
                    &sc, &red, &bar, &limit};
    return cudaLaunchCooperativeKernel((const void *)k_vb_pcg<T>, dim3(grid), dim3(256), args, 0, h->st);
}

}  // namespace

namespace ba {

ba_status vb_check_pattern(const ba_options &o, int32_t n, const int32_t *cdim, int64_t nnzb, const int32_t *row_ptr,
                           const int32_t *col, int64_t *N_out, int64_t *nval_out) {
    if (o.precision != BA_FP64 && o.precision != BA_FP32) return set_error(BA_ERR_INVALID_ARG, "bad precision");
    if (n <= 0 || n >= (1 << 30) || nnzb < n || nnzb >= (int64_t)INT32_MAX)
        return set_error(BA_ERR_INVALID_ARG, "need 0 < n < 2^30 and n <= nnzb < 2^31");
    if (!cdim || !row_ptr || !col) return set_error(BA_ERR_INVALID_ARG, "null input array");
    if (row_ptr[0] != 0 || row_ptr[n] != nnzb) return set_error(BA_ERR_INVALID_ARG, "row_ptr must run from 0 to nnzb");
    int64_t N = 0, nval = 0;
    for (int32_t i = 0; i < n; ++i) {
        if (cdim[i] < 1 || cdim[i] > BA_VB_CMAX) return set_error(BA_ERR_INVALID_ARG, "block size out of 1..BA_VB_CMAX");
        N += cdim[i];
    }
    if (N >= (int64_t)INT32_MAX) return set_error(BA_ERR_INVALID_ARG, "too many unknowns");
    for (int32_t i = 0; i < n; ++i) {
        if (row_ptr[i + 1] <= row_ptr[i]) return set_error(BA_ERR_INVALID_ARG, "every row needs its diagonal block");
        if (col[row_ptr[i]] != i) return set_error(BA_ERR_INVALID_ARG, "the first block of a row must be its diagonal");
        for (int32_t k = row_ptr[i] + 1; k < row_ptr[i + 1]; ++k)
            if (col[k] <= col[k - 1] || col[k] >= n)
                return set_error(BA_ERR_INVALID_ARG, "columns must increase within a row and stay below n");
        for (int32_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k) nval += (int64_t)cdim[i] * cdim[col[k]];
    }
    *N_out = N;
    *nval_out = nval;
    return BA_OK;
}

ba_status vb_build(const ba_options &o, int32_t n, const int32_t *cdim, int64_t nnzb, const int32_t *row_ptr,
                   const int32_t *col, ba_vbsmc **out) {
    int64_t N = 0, nval = 0, nminv = 0;
    ba_status s = vb_check_pattern(o, n, cdim, nnzb, row_ptr, col, &N, &nval);
    if (s) return s;
    // host-side layout: offsets, two-sided entry lists
    std::vector<int32_t> off(n + 1, 0), ent_cam(N), tw_ptr(n + 1, 0);
    std::vector<int64_t> boff(nnzb + 1, 0), moff(n + 1, 0);
    for (int32_t i = 0; i < n; ++i) {
        off[i + 1] = off[i] + cdim[i];
        moff[i + 1] = moff[i] + (int64_t)cdim[i] * cdim[i];
        for (int32_t a = 0; a < cdim[i]; ++a) ent_cam[off[i] + a] = i;
        for (int32_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k) boff[k + 1] = boff[k] + (int64_t)cdim[i] * cdim[col[k]];
    }
    nminv = moff[n];
    for (int32_t i = 0; i < n; ++i) {
        tw_ptr[i + 1] += row_ptr[i + 1] - row_ptr[i];
        for (int32_t k = row_ptr[i] + 1; k < row_ptr[i + 1]; ++k) tw_ptr[col[k] + 1] += 1;
    }
    for (int32_t i = 0; i < n; ++i) tw_ptr[i + 1] += tw_ptr[i];
    // two-sided entry records: value offset (lo, hi), vector offset of the
    // other camera j, c_j << 1 | transposed
    std::vector<int4> tw_info(tw_ptr[n]);
    {
        auto rec = [&](int32_t k, int32_t j, int tr) {
            return make_int4((int)(uint32_t)(boff[k] & 0xffffffffu), (int)(boff[k] >> 32), off[j], (cdim[j] << 1) | tr);
        };
        std::vector<int32_t> fill(tw_ptr.begin(), tw_ptr.end() - 1);
        for (int32_t i = 0; i < n; ++i)
            for (int32_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k) tw_info[fill[i]++] = rec(k, col[k], 0);
        for (int32_t i = 0; i < n; ++i)
            for (int32_t k = row_ptr[i] + 1; k < row_ptr[i + 1]; ++k) tw_info[fill[col[k]]++] = rec(k, i, 1);
    }
    ba_vbsmc *h = new ba_vbsmc();
    h->n = n;
    h->nnzb = nnzb;
    h->N = N;
    h->nval = nval;
    h->nminv = nminv;
    h->fp32 = o.precision == BA_FP32;
    h->esz = h->fp32 ? 4 : 8;
    h->st = (cudaStream_t)o.cuda_stream;
    h->cap = o.device_mem_cap;
    auto up = [&](void **d, const void *src, size_t bytes) -> ba_status {
        ba_status r = vb_alloc(h, d, bytes);
        if (r) return r;
        return vb_cuda(h, cudaMemcpy(*d, src, bytes, cudaMemcpyHostToDevice), "upload");
    };
    std::vector<int32_t> brow(nnzb);
    for (int32_t i = 0; i < n; ++i)
        for (int32_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k) brow[k] = i;
    int dev = 0, n_sm = 0;
    if (!s) s = vb_cuda(h, cudaGetDevice(&dev), "device");
    if (!s) s = vb_cuda(h, cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev), "device");
    if (!s)
        h->plan = h->fp32 ? vb_own_plan<float>(n, n_sm, cdim, tw_ptr, tw_info)
                          : vb_own_plan<double>(n, n_sm, cdim, tw_ptr, tw_info);
    if (!s) s = up((void **)&h->cdim, cdim, n * sizeof(int32_t));
    if (!s) s = up((void **)&h->off, off.data(), (n + 1) * sizeof(int32_t));
    if (!s) s = up((void **)&h->row_ptr, row_ptr, (n + 1) * sizeof(int32_t));
    if (!s) s = up((void **)&h->col, col, nnzb * sizeof(int32_t));
    if (!s) s = up((void **)&h->brow, brow.data(), nnzb * sizeof(int32_t));
    if (!s) s = up((void **)&h->ent_cam, ent_cam.data(), N * sizeof(int32_t));
    if (!s) s = up((void **)&h->tw_ptr, tw_ptr.data(), (n + 1) * sizeof(int32_t));
    if (!s) s = up((void **)&h->tw_info, tw_info.data(), tw_info.size() * sizeof(int4));
    if (!s) s = up((void **)&h->boff, boff.data(), (nnzb + 1) * sizeof(int64_t));
    if (!s) s = up((void **)&h->moff, moff.data(), (n + 1) * sizeof(int64_t));
    if (!s) s = vb_alloc(h, &h->val, nval * h->esz);
    if (!s) s = vb_alloc(h, &h->b, N * h->esz);
    if (!s) s = vb_alloc(h, &h->Minv, nminv * h->esz);
    for (auto &v : h->vec)
        if (!s) s = vb_alloc(h, &v, N * h->esz);
    if (!s) s = vb_alloc(h, (void **)&h->sc, sizeof(VbScalars));
    if (!s) s = vb_alloc(h, (void **)&h->red, (size_t)RED_SLOTS * sizeof(double));
    if (!s) s = vb_alloc(h, (void **)&h->err, sizeof(int));
    // the arrival counters lie behind the partials (2 grids of AR_NV_MAX doubles
    // each, at most 2 CTAs on every SM)
    if (!s) h->bar = reinterpret_cast<unsigned *>(h->red + RED_SLOTS / 2);
    if (!s) s = vb_cuda(h, cudaEventCreate(&h->ev[0]), "event");
    if (!s) s = vb_cuda(h, cudaEventCreate(&h->ev[1]), "event");
    if (s) {
        ba_vbsmc_destroy(h);
        return s;
    }
    *out = h;
    return BA_OK;
}

ba_status vb_finish(ba_vbsmc *h) {
    ba_status s;
    if ((s = vb_cuda(h, cudaMemsetAsync(h->err, 0, sizeof(int), h->st), "memset"))) return s;
    const int g = (h->n + 3) / 4;  // sixteen lanes per camera, two warps per CTA: spread over the SMs
    if (h->fp32)
        k_vb_minv<float><<<g, 64, 0, h->st>>>(h->n, h->cdim, h->row_ptr, h->boff, (const float *)h->val, h->moff,
                                               (float *)h->Minv, h->err);
    else
        k_vb_minv<double><<<g, 64, 0, h->st>>>(h->n, h->cdim, h->row_ptr, h->boff, (const double *)h->val, h->moff,
                                                (double *)h->Minv, h->err);
    if ((s = vb_cuda(h, cudaGetLastError(), "k_vb_minv"))) return s;
    int err = 0;
    if ((s = vb_cuda(h, cudaMemcpyAsync(&err, h->err, sizeof(int), cudaMemcpyDeviceToHost, h->st), "read flag")))
        return s;
    if ((s = vb_cuda(h, cudaStreamSynchronize(h->st), "sync"))) return s;
    if (err == BA_ERR_NOT_SPD) return set_error(BA_ERR_NOT_SPD, "a diagonal block is not positive definite");
    return BA_OK;
}

}  // namespace ba

extern "C" {

ba_status ba_vbsmc_create(const ba_options *opt, int32_t n, const int32_t *cdim, int64_t nnzb, const int32_t *row_ptr,
                          const int32_t *col, const double *val, const double *b, ba_vbsmc **out) {
    if (!out) return set_error(BA_ERR_INVALID_ARG, "null output pointer");
    *out = nullptr;
    ba_options o;
    if (opt) o = *opt; else ba_options_default(&o);
    if (!val || !b) return set_error(BA_ERR_INVALID_ARG, "null input array");
    int64_t N = 0, nval = 0;
    ba_status s = vb_check_pattern(o, n, cdim, nnzb, row_ptr, col, &N, &nval);
    if (s) return s;
    for (int64_t k = 0; k < nval; ++k)
        if (!std::isfinite(val[k])) return set_error(BA_ERR_NONFINITE, "non-finite block value");
    for (int64_t k = 0; k < N; ++k)
        if (!std::isfinite(b[k])) return set_error(BA_ERR_NONFINITE, "non-finite b");
    ba_vbsmc *h = nullptr;
    if ((s = vb_build(o, n, cdim, nnzb, row_ptr, col, &h))) return s;
    s = h->fp32 ? vb_upload<float>(h, h->val, val, nval) : vb_upload<double>(h, h->val, val, nval);
    if (!s) s = h->fp32 ? vb_upload<float>(h, h->b, b, N) : vb_upload<double>(h, h->b, b, N);
    if (!s) s = vb_finish(h);
    if (s) {
        ba_vbsmc_destroy(h);
        return s;
    }
    *out = h;
    return BA_OK;
}

ba_status ba_vbsmc_get_system(const ba_vbsmc *h, int32_t *row_ptr, int32_t *col, double *val, double *b) {
    if (!h) return set_error(BA_ERR_INVALID_ARG, "null object");
    if (h->dead) return set_error(BA_ERR_STATE, "the object is unusable after an earlier error");
    ba_vbsmc *m = const_cast<ba_vbsmc *>(h);
    ba_status s;
    if (row_ptr && (s = vb_cuda(m, cudaMemcpy(row_ptr, h->row_ptr, (h->n + 1) * sizeof(int32_t), cudaMemcpyDeviceToHost),
                                "read row_ptr")))
        return s;
    if (col && (s = vb_cuda(m, cudaMemcpy(col, h->col, h->nnzb * sizeof(int32_t), cudaMemcpyDeviceToHost), "read col")))
        return s;
    auto rd = [&](double *dst, const void *src, int64_t cnt) -> ba_status {
        std::vector<char> raw(cnt * h->esz);
        ba_status r = vb_cuda(m, cudaMemcpy(raw.data(), src, raw.size(), cudaMemcpyDeviceToHost), "read values");
        if (r) return r;
        for (int64_t k = 0; k < cnt; ++k)
            dst[k] = h->fp32 ? (double)reinterpret_cast<const float *>(raw.data())[k]
                             : reinterpret_cast<const double *>(raw.data())[k];
        return BA_OK;
    };
    if (val && (s = rd(val, h->val, h->nval))) return s;
    if (b && (s = rd(b, h->b, h->N))) return s;
    return BA_OK;
}

ba_status ba_vbsmc_spmv(ba_vbsmc *h, const void *x, void *y) {
    if (!h || !x || !y) return set_error(BA_ERR_INVALID_ARG, "null argument");
    if (h->dead) return set_error(BA_ERR_STATE, "the object is unusable after an earlier error");
    cudaError_t e = h->fp32 ? vb_spmv_T<float>(h, (const float *)x, (float *)y)
                            : vb_spmv_T<double>(h, (const double *)x, (double *)y);
    return vb_cuda(h, e, "k_vb_spmv");
}

ba_status ba_vbsmc_solve(ba_vbsmc *h, double tol, int32_t max_iters, double *x_out, int32_t *iters, double *rel_resid,
                         double *kernel_ms) {
    if (!h) return set_error(BA_ERR_INVALID_ARG, "null object");
    if (h->dead) return set_error(BA_ERR_STATE, "the object is unusable after an earlier error");
    if (!(tol > 0) || max_iters < 0) return set_error(BA_ERR_INVALID_ARG, "need tol > 0 and max_iters >= 0");
    VbScalars init{};
    init.tol2 = tol * tol;
    init.max_iters = max_iters > 0 ? max_iters : std::max(1000, 6 * h->n);
    ba_status s;
    if ((s = vb_cuda(h, cudaMemcpyAsync(h->sc, &init, sizeof(init), cudaMemcpyHostToDevice, h->st), "scalars")))
        return s;
    if ((s = vb_cuda(h, cudaEventRecord(h->ev[0], h->st), "event"))) return s;
    cudaError_t e = h->fp32 ? vb_pcg_T<float>(h) : vb_pcg_T<double>(h);
    if ((s = vb_cuda(h, e, "k_vb_pcg"))) return s;
    if ((s = vb_cuda(h, cudaEventRecord(h->ev[1], h->st), "event"))) return s;
    if ((s = vb_cuda(h, cudaMemcpyAsync(&h->host, h->sc, sizeof(VbScalars), cudaMemcpyDeviceToHost, h->st),
                     "scalars")))
        return s;
    if ((s = vb_cuda(h, cudaStreamSynchronize(h->st), "sync"))) return s;
    if (h->host.err == BA_ERR_TIMEOUT) {
        h->dead = true;
        return set_error(BA_ERR_TIMEOUT, "PCG grid wait timed out");
    }
    if (kernel_ms) {
        float ms = 0.f;
        if ((s = vb_cuda(h, cudaEventElapsedTime(&ms, h->ev[0], h->ev[1]), "event"))) return s;
        *kernel_ms = ms;
    }
    if (x_out) {
        std::vector<char> raw(h->N * h->esz);
        if ((s = vb_cuda(h, cudaMemcpy(raw.data(), h->vec[0], raw.size(), cudaMemcpyDeviceToHost), "read y"))) return s;
        for (int64_t k = 0; k < h->N; ++k)
            x_out[k] = h->fp32 ? (double)reinterpret_cast<const float *>(raw.data())[k]
                               : reinterpret_cast<const double *>(raw.data())[k];
    }
    const double rel = h->host.rr0 > 0 ? std::sqrt(h->host.rr / h->host.rr0) : 0.0;
    if (iters) *iters = h->host.iters;
    if (rel_resid) *rel_resid = rel;
    if (h->host.err == BA_ERR_NOT_SPD) return set_error(BA_ERR_NOT_SPD, "d^T S d <= 0 in PCG");
    if (h->host.rr0 > 0 && !(h->host.rr <= h->host.tol2 * h->host.rr0))
        return set_error(BA_ERR_NO_CONVERGENCE, "PCG reached its iteration cap");
    return BA_OK;
}

ba_status ba_vbsmc_info(const ba_vbsmc *h, int64_t *n_unknowns, int64_t *storage_bytes, int64_t *n_blocks) {
    if (!h) return set_error(BA_ERR_INVALID_ARG, "null object");
    if (n_unknowns) *n_unknowns = h->N;
    if (n_blocks) *n_blocks = h->nnzb;
    if (storage_bytes)
        *storage_bytes = h->nval * (int64_t)h->esz + h->nnzb * (4 + 8) + (int64_t)(h->n + 1) * 4 + (int64_t)h->n * 4;
    return BA_OK;
}

void ba_vbsmc_destroy(ba_vbsmc *h) {
    if (!h) return;
    if (h->st) cudaStreamSynchronize(h->st);
    else cudaDeviceSynchronize();
    for (auto &e : h->ev)
        if (e) cudaEventDestroy(e);
    for (void *d : h->allocs) cudaFree(d);
    delete h;
}

}  // extern "C"
