// The reduced camera system of cameras with interior parameters, formed on
// the device into a variable-size BSMC system (ba_vbsmc_create_interiors).
//
// Sec. 4 gives block (i, j) of the RCS c_i x c_j entries; Sec. 4.1 counts six
// exterior and five interior unknowns per camera.  The interiors are
// [f, cx, cy, k1, k2]: with xh = x/z, yh = y/z, r2 = xh^2 + yh^2 and
// d = 1 + k1 r2 + k2 r2^2 the projection is u = f d xh + cx, v = f d yh + cy.
// A camera has c_i = 6 (interiors fixed) or 11 unknowns.  Four kernels:
//   k_vbi_linearize  e and J of every observation (Eq. 1), rows of
//                    [J_c (11 x 2) | J_p (2 x 3) | e (2)] in the storage
//                    precision (X_cam in FP64, the rest in that precision);
//   k_vbi_factor     per point, in FP64, V_k (damped) and l_p (Eq. 3), the
//                    inverse M = L^-1 of V_k's Cholesky factor and q = M l_p;
//   k_vbi_rows       per observation, in FP64, the factor row P = J_p M^T and
//                    e^ = e + P q;
//   k_vbi_blocks32 / k_vbi_blocks64
//                    a warp per stored block (i, j): the sum over its point
//                    pairs of -J_c,a^T (P_a P_b^T) J_c,b = -W_a V_k^-1 W_b^T
//                    (Eq. 4), plus U_i (damped) and b_i = -sum J_c^T e^ on
//                    the diagonal, in the storage precision.  The pairs of a
//                    block are listed on the host (track order), so the sums
//                    need no atomics and are deterministic.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "device_util.cuh"
#include "tma_util.cuh"
#include "vbsmc_internal.h"

namespace ba {

// J row (T): J_c by columns, the two rows of column c at 2 c, 2 c + 1 (c < 11) |
// pad 22, 23 | J_p 2 x 3 at 24, 27 | e at 30, 31.  A column is one aligned pair
// (the block kernels load the columns they need), J_p and e one aligned
// 32-byte stretch in FP32.
constexpr int VJW = 32, VJP = 24, VJE = 30;
constexpr int VPW = 8;       // factor row (T): P = J_p L^-T (2 x 3) at 0, 3 | e^ = e + P L^-1 l_p at 6, 7
constexpr int VB_CI = 11;    // unknowns of a self-calibrating camera
constexpr int VB_NT = 4;     // block entries per lane: 4 x 32 >= 11 x 11

// Per camera [R (9), t (3)] in FP64, R = Exp(omega).
__device__ __forceinline__ void vbi_camera(const double *cam, double *out) {
    double q[4], R[9];
    quat_exp(cam, q);
    quat_to_R(q, R);
    for (int k = 0; k < 9; ++k) out[k] = R[k];
    for (int k = 0; k < 3; ++k) out[9 + k] = cam[3 + k];
}
__global__ void k_vbi_camcache(int n, const double *__restrict__ cams, double *__restrict__ camc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) vbi_camera(cams + 6 * i, camc + 12 * i);
}

// X_cam = R X + t in FP64 (no cancellation of the large world coordinates),
// then the projection with interiors in T: xh = x/z, yh = y/z,
// r2 = xh^2 + yh^2, d = 1 + k1 r2 + k2 r2^2, e = (f d xh + cx, f d yh + cy) - u.
template <typename T>
struct VbiProj {
    T Xc[3], xh, yh, r2, d, e0, e1;
};
template <typename T>
__device__ __forceinline__ VbiProj<T> vbi_project(const double *__restrict__ camc, const double *__restrict__ intr,
                                                  const double *__restrict__ pts, int i, int64_t k,
                                                  const double *__restrict__ uv) {
    const double *R = camc + 12 * i, *X = pts + 3 * k, *kk = intr + 5 * i;
    VbiProj<T> o;
    for (int r = 0; r < 3; ++r) o.Xc[r] = (T)(R[3 * r] * X[0] + R[3 * r + 1] * X[1] + R[3 * r + 2] * X[2] + R[9 + r]);
    o.xh = o.Xc[0] / o.Xc[2];
    o.yh = o.Xc[1] / o.Xc[2];
    o.r2 = o.xh * o.xh + o.yh * o.yh;
    o.d = T(1) + (T)kk[3] * o.r2 + (T)kk[4] * o.r2 * o.r2;
    o.e0 = (T)kk[0] * o.d * o.xh + (T)(kk[1] - uv[0]);
    o.e1 = (T)kk[0] * o.d * o.yh + (T)(kk[2] - uv[1]);
    return o;
}

// N values from a 16-byte aligned address with 16-byte loads.
template <int N, typename T>
__device__ __forceinline__ void load_vec(const T *__restrict__ p, T (&v)[N]) {
    static_assert(N * sizeof(T) % 16 == 0, "whole 16-byte words");
    if constexpr (sizeof(T) == 4) {
        const float4 *q = reinterpret_cast<const float4 *>(p);
#pragma unroll
        for (int k = 0; k < N / 4; ++k) {
            const float4 t = __ldg(q + k);
            v[4 * k] = t.x; v[4 * k + 1] = t.y; v[4 * k + 2] = t.z; v[4 * k + 3] = t.w;
        }
    } else {
        const double2 *q = reinterpret_cast<const double2 *>(p);
#pragma unroll
        for (int k = 0; k < N / 2; ++k) {
            const double2 t = __ldg(q + k);
            v[2 * k] = t.x; v[2 * k + 1] = t.y;
        }
    }
}

struct VbiScalars {
    double cost, cost_trial, model;
    unsigned long long n_cheir_trial;
};

// A thread per observation; a warp's 32 rows leave through shared memory, so
// that each is written as whole lines.  With sc, also F = 1/2 sum ||e||^2 of the
// stored e (FP64 sum).  (Rows written value by value from the threads, with the
// cost in a pass of its own, took 101 us for 485,000 observations in FP32; this
// takes 47.)
constexpr int VLT = 128;  // threads per CTA
template <typename T>
__global__ void __launch_bounds__(VLT) k_vbi_linearize(int64_t m, const int *__restrict__ ocam,
                                                       const int *__restrict__ opt, const double *__restrict__ uv,
                                                       const double *__restrict__ camc,
                                                       const double *__restrict__ intr,
                                                       const double *__restrict__ pts, T *__restrict__ J,
                                                       VbiScalars *sc, double *red, unsigned *ctr) {
    __shared__ T rows[VLT / 32][32][VJW + 1];
    const int lane = threadIdx.x & 31;
    T(*row)[VJW + 1] = rows[threadIdx.x >> 5];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    double F[1] = {0.0};
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < m; base += stride) {
        const int64_t a = base + lane;
        if (a < m) {
            const int i = ocam[a], k = opt[a];
            const VbiProj<T> pr = vbi_project<T>(camc, intr, pts, i, k, uv + 2 * a);
            const double *R = camc + 12 * i, *kk = intr + 5 * i;
            const T f = (T)kk[0], k1 = (T)kk[3], k2 = (T)kk[4];
            const T z = pr.Xc[2], xh = pr.xh, yh = pr.yh, r2 = pr.r2, d = pr.d;
            const T g = T(2) * (k1 + T(2) * k2 * r2);
            // image-plane Jacobian D of (f d xh, f d yh) w.r.t. (xh, yh), then A = D d(xh, yh)/dX_cam
            const T D00 = f * (d + g * xh * xh), D01 = f * g * xh * yh, D11 = f * (d + g * yh * yh);
            T A[2][3];
            A[0][0] = D00 / z;
            A[0][1] = D01 / z;
            A[0][2] = -(D00 * xh + D01 * yh) / z;
            A[1][0] = D01 / z;
            A[1][1] = D11 / z;
            A[1][2] = -(D01 * xh + D11 * yh) / z;
            // dX_cam/d(d_omega) = -[X_cam]x (camera-frame update), dX_cam/d(dt) = I, dX_cam/dX = R
            const T *Xc = pr.Xc;
            const T Mx[3][3] = {{T(0), Xc[2], -Xc[1]}, {-Xc[2], T(0), Xc[0]}, {Xc[1], -Xc[0], T(0)}};
            T *o = row[lane];
            const T ph[2] = {xh, yh};
            for (int r = 0; r < 2; ++r) {
                T *jc = o + r, *jp = o + VJP + 3 * r;  // column c at jc[2 c]
                for (int c = 0; c < 3; ++c) {
                    jc[2 * c] = A[r][0] * Mx[0][c] + A[r][1] * Mx[1][c] + A[r][2] * Mx[2][c];
                    jc[2 * (3 + c)] = A[r][c];
                    jp[c] = A[r][0] * (T)R[c] + A[r][1] * (T)R[3 + c] + A[r][2] * (T)R[6 + c];
                }
                jc[12] = d * ph[r];                // f
                jc[14] = r == 0 ? T(1) : T(0);     // cx
                jc[16] = r == 0 ? T(0) : T(1);     // cy
                jc[18] = f * ph[r] * r2;           // k1
                jc[20] = f * ph[r] * r2 * r2;      // k2
            }
            o[VJE] = pr.e0;
            o[VJE + 1] = pr.e1;
            o[22] = T(0);
            o[23] = T(0);
            if (sc) {
                const double e0 = widen(pr.e0), e1 = widen(pr.e1);
                F[0] += e0 * e0 + e1 * e1;
            }
        }
        __syncwarp();
        const int nr = (int)min((int64_t)32, m - base);
        T *out = J + base * VJW + lane;
#pragma unroll 8
        for (int r = 0; r < nr; ++r) out[r * VJW] = row[r][lane];
        __syncwarp();
    }
    if (sc) grid_sum<1>(F, red, ctr, [&](double *t) { sc->cost = 0.5 * t[0]; });
}

// Per point, in FP64: V_k = sum J_p^T J_p + lambda clamp(diag), its Cholesky
// factor V_k = L L^T (the three pivots must be positive), l_p = -sum J_p^T e;
// stored per point: M = L^-1 (m00 m10 m11 m20 m21 m22) and q = M l_p, from
// which Eq. 5 and the factor rows follow.  A thread per point, in the order
// `ord` of track lengths, so that the threads of a warp loop alike (bound by
// FP64 issue; in the points' own order a warp runs its longest track, 2.6
// times the mean).  With k_vbi_rows 96 us at 99,000 points, 485,000
// observations, against 275 us for one kernel in the points' own order that
// also formed the factor rows.
template <typename T>
__global__ void __launch_bounds__(128) k_vbi_factor(int64_t P, const int *__restrict__ ord,
                                                    const int *__restrict__ trk_ptr, const T *__restrict__ J,
                                                    double lambda, double *__restrict__ Mq, int *err) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < P; x += (int64_t)gridDim.x * blockDim.x) {
        const int k = __ldg(ord + x);
        double v00 = 0, v01 = 0, v02 = 0, v11 = 0, v12 = 0, v22 = 0, l0 = 0, l1 = 0, l2 = 0;
        const int a1 = __ldg(trk_ptr + k + 1);
        for (int a = __ldg(trk_ptr + k); a < a1; ++a) {
            T s[8];
            load_vec<8>(J + (int64_t)a * VJW + VJP, s);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const double p0 = widen(s[3 * r]), p1 = widen(s[3 * r + 1]), p2 = widen(s[3 * r + 2]);
                const double e = widen(s[6 + r]);
                v00 = fma(p0, p0, v00); v01 = fma(p0, p1, v01); v02 = fma(p0, p2, v02);
                v11 = fma(p1, p1, v11); v12 = fma(p1, p2, v12); v22 = fma(p2, p2, v22);
                l0 = fma(-p0, e, l0); l1 = fma(-p1, e, l1); l2 = fma(-p2, e, l2);
            }
        }
        v00 += lambda * clampT(v00);
        v11 += lambda * clampT(v11);
        v22 += lambda * clampT(v22);
        const double d0 = sqrt(v00), c10 = v01 / d0, c20 = v02 / d0;
        const double s11 = v11 - c10 * c10, d1 = sqrt(s11), c21 = (v12 - c20 * c10) / d1;
        const double s22 = v22 - c20 * c20 - c21 * c21, d2 = sqrt(s22);
        const bool ok = v00 > 0.0 && s11 > 0.0 && s22 > 0.0;
        double m00 = 1.0 / d0, m11 = 1.0 / d1, m22 = 1.0 / d2;
        double m10 = -c10 * m00 * m11, m21 = -c21 * m11 * m22, m20 = -(c20 * m00 + c21 * m10) * m22;
        if (!ok) {
            atomicExch(err, (int)BA_ERR_NOT_SPD);
            m00 = m11 = m22 = m10 = m21 = m20 = 0.0;
        }
        double *o = Mq + 9 * (int64_t)k;
        o[0] = m00; o[1] = m10; o[2] = m11; o[3] = m20; o[4] = m21; o[5] = m22;
        o[6] = m00 * l0;
        o[7] = m10 * l0 + m11 * l1;
        o[8] = m20 * l0 + m21 * l1 + m22 * l2;
    }
}

// Per observation, in FP64, the factor row P = J_p M^T and e^ = e + P q of its
// point, stored in T, so that -W_a V^-1 W_b^T = -J_c,a^T (P_a P_b^T) J_c,b and
// -J_c,a^T e_a - W_a V^-1 l_p = -J_c,a^T e^_a (the block kernels' products).
template <typename T>
__global__ void __launch_bounds__(256) k_vbi_rows(int64_t m, const int *__restrict__ opt, const T *__restrict__ J,
                                                  const double *__restrict__ Mq, T *__restrict__ PE) {
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < m; a += (int64_t)gridDim.x * blockDim.x) {
        T s[8], o[8];
        load_vec<8>(J + a * VJW + VJP, s);
        const double *w = Mq + 9 * (int64_t)__ldg(opt + a);
        const double m00 = __ldg(w), m10 = __ldg(w + 1), m11 = __ldg(w + 2), m20 = __ldg(w + 3), m21 = __ldg(w + 4),
                     m22 = __ldg(w + 5), q0 = __ldg(w + 6), q1 = __ldg(w + 7), q2 = __ldg(w + 8);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const double j0 = widen(s[3 * r]), j1 = widen(s[3 * r + 1]), j2 = widen(s[3 * r + 2]);
            // P = J_p L^-T: P_c = sum_k J_k (L^-1)_ck over k <= c
            const double P0 = j0 * m00, P1 = j0 * m10 + j1 * m11, P2 = j0 * m20 + j1 * m21 + j2 * m22;
            o[3 * r] = (T)P0;
            o[3 * r + 1] = (T)P1;
            o[3 * r + 2] = (T)P2;
            o[6 + r] = (T)(widen(s[6 + r]) + P0 * q0 + P1 * q1 + P2 * q2);
        }
        T *pe = PE + a * VPW;
        if constexpr (sizeof(T) == 4) {
            reinterpret_cast<float4 *>(pe)[0] = make_float4(o[0], o[1], o[2], o[3]);
            reinterpret_cast<float4 *>(pe)[1] = make_float4(o[4], o[5], o[6], o[7]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) reinterpret_cast<double2 *>(pe)[q] = make_double2(o[2 * q], o[2 * q + 1]);
        }
    }
}

// The block kernels: a warp per stored block (beta, gamma) and its list of
// slot pairs (a, b).  A slot is an observation's J_c columns that belong to one
// block: for a block of camera i (c_i = 6 or 11) the first c_i columns, for the
// block of a physical camera whose images share interiors the five interior
// columns; jc0[beta] is the first J_c column of block beta's slots (null: 0).
// The pairs of a block are its slots' pairs within each point (every ordered
// pair, a in beta and b in gamma).  Per pair the 2 x 2 middle factor M is
// -P_a P_b^T, or I - P_a P_a^T when both slots belong to one observation (that
// adds U = J_c^T J_c, the coupling of an image and its physical camera
// included), and the block gains J_c,a^T (M J_c,b).  Summed over a point's slot
// pairs this is U - W_beta V_k^-1 W_gamma^T with W_beta summed over the point's
// slots in beta.  On a diagonal block a slot paired with itself also gives
// b_beta's term -J_c,a^T e^_a and the U diagonal that damps the block at the
// end.  The factors M of 32 pairs are formed at once, one pair to a lane, and
// handed to the warp by shuffles.

// a b + c d with one rounding fewer
template <typename T>
__device__ __forceinline__ T dot2(T a, T b, T c, T d) {
    return fma(a, b, c * d);
}

// One pair's middle factor from the factor rows of its observations (and the
// first row's e^).
template <typename T>
__device__ __forceinline__ void vbi_middle(const T *__restrict__ Pa, const T *__restrict__ Pb, bool same, T (&M)[4],
                                           T (&eh)[2]) {
    T a[8], b[8];
    if constexpr (sizeof(T) == 4) {
        const float4 *p = reinterpret_cast<const float4 *>(Pa), *q = reinterpret_cast<const float4 *>(Pb);
        const float4 a0 = __ldg(p), a1 = __ldg(p + 1), b0 = __ldg(q), b1 = __ldg(q + 1);
        a[0] = a0.x; a[1] = a0.y; a[2] = a0.z; a[3] = a0.w; a[4] = a1.x; a[5] = a1.y; a[6] = a1.z; a[7] = a1.w;
        b[0] = b0.x; b[1] = b0.y; b[2] = b0.z; b[3] = b0.w; b[4] = b1.x; b[5] = b1.y;
    } else {
        const double2 *p = reinterpret_cast<const double2 *>(Pa), *q = reinterpret_cast<const double2 *>(Pb);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double2 u = __ldg(p + k), v = __ldg(q + k);
            a[2 * k] = u.x; a[2 * k + 1] = u.y;
            b[2 * k] = v.x; b[2 * k + 1] = v.y;
        }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v)
            M[2 * u + v] = (same && u == v ? T(1) : T(0)) -
                           fma(a[3 * u + 2], b[3 * v + 2], dot2(a[3 * u], b[3 * v], a[3 * u + 1], b[3 * v + 1]));
    eh[0] = a[6];
    eh[1] = a[7];
}

// FP32: the block as a 4 x 8 grid of lanes, each with up to 3 x 2 entries in
// registers.  The heads of the pairs' J rows (96 bytes: the columns) come eight
// pairs at a time by asynchronous copies into one half of the warp's stage
// while the other half is used, so a pair costs five shared loads, four shuffles
// and about thirty multiply-adds per lane, with no wait of its own.  A block's
// pairs are added in list order, each as acc + (j0 t0 + j1 t1).  Bound by
// instruction issue (57 per pair and warp).  990 cameras of c = 11, 485,000
// observations, 2.1 M pairs: 173 us; 386 with the columns loaded by the lanes
// straight from the rows (waits for L1 and L2), 1031 with both rows passed
// through shared memory pair by pair; the same bits.
constexpr int VB32_FETCH = 8;  // pairs copied at a time: 16 row heads, two halves per warp
static_assert(VB32_FETCH * 12 % 32 == 0, "whole turns of a warp");
// RPL x CPL entries per lane (the lanes beyond the block's edge repeat its last
// row or column, so that the loop has no predicates).
template <int RPL, int CPL, bool DIAG>
__device__ __forceinline__ void vbi32_block(int p0, int p1, int ci, int cj, int ai, int aj,
                                            const int2 *__restrict__ plist, const float *__restrict__ J,
                                            const float *__restrict__ PE, float lambda, float *__restrict__ out,
                                            float *__restrict__ b, float *stage) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, rg = lane >> 3, cg = lane & 7;
    // byte offsets of this lane's columns within a J row
    int ra[RPL], rb[CPL];
#pragma unroll
    for (int u = 0; u < RPL; ++u) ra[u] = 8 * (ai + min(RPL * rg + u, ci - 1));
#pragma unroll
    for (int v = 0; v < CPL; ++v) rb[v] = 8 * (aj + min(CPL * cg + v, cj - 1));
    float acc[RPL][CPL], dU[RPL], bacc[RPL];
#pragma unroll
    for (int u = 0; u < RPL; ++u) {
        dU[u] = bacc[u] = 0.f;
#pragma unroll
        for (int v = 0; v < CPL; ++v) acc[u][v] = 0.f;
    }
    for (; p0 < p1; p0 += 32) {
        const int cnt = min(32, p1 - p0);
        int2 pr = make_int2(0, 0);
        float M[4] = {0.f, 0.f, 0.f, 0.f}, eh[2] = {0.f, 0.f};
        if (lane < cnt) pr = __ldg(plist + p0 + lane);
        // copies of pairs q0 .. q0 + 7 into half `h` of the stage, 16 bytes to a
        // lane and turn: row c / 6 of the sixteen, part c % 6 of its columns
        auto fetch = [&](int q0, int h) {
#pragma unroll
            for (int t = 0; t < VB32_FETCH * 12 / 32; ++t) {
                const int c = lane + 32 * t, row = c / 6, part = c - 6 * row, q = q0 + (row >> 1);
                const int x = __shfl_sync(FULL, pr.x, q & 31), y = __shfl_sync(FULL, pr.y, q & 31);
                if (q < cnt)
                    cp_async16(stage + h * (VB32_FETCH * 48) + row * 24 + 4 * part,
                               J + (int64_t)((row & 1) ? y : x) * VJW + 4 * part);
            }
            cp_async_commit();
        };
        fetch(0, 0);
        if (lane < cnt) vbi_middle<float>(PE + (int64_t)pr.x * VPW, PE + (int64_t)pr.y * VPW, pr.x == pr.y, M, eh);
        for (int q0 = 0, h = 0; q0 < cnt; q0 += VB32_FETCH, h ^= 1) {
            if (q0 + VB32_FETCH < cnt) {
                fetch(q0 + VB32_FETCH, h ^ 1);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncwarp();
            const char *st = reinterpret_cast<const char *>(stage + h * (VB32_FETCH * 48));
            const int nq = min(VB32_FETCH, cnt - q0);
#pragma unroll 4
            for (int qq = 0; qq < nq; ++qq) {
                const int q = q0 + qq;
                const float m00 = __shfl_sync(FULL, M[0], q), m01 = __shfl_sync(FULL, M[1], q),
                            m10 = __shfl_sync(FULL, M[2], q), m11 = __shfl_sync(FULL, M[3], q);
                const char *ja = st + 192 * qq, *jb = ja + 96;
                float2 a[RPL], t[CPL];
#pragma unroll
                for (int u = 0; u < RPL; ++u) a[u] = *reinterpret_cast<const float2 *>(ja + ra[u]);
#pragma unroll
                for (int v = 0; v < CPL; ++v) {
                    const float2 w = *reinterpret_cast<const float2 *>(jb + rb[v]);
                    t[v] = make_float2(dot2(m00, w.x, m01, w.y), dot2(m10, w.x, m11, w.y));
                }
#pragma unroll
                for (int u = 0; u < RPL; ++u)
#pragma unroll
                    for (int v = 0; v < CPL; ++v) acc[u][v] += dot2(a[u].x, t[v].x, a[u].y, t[v].y);
                if (DIAG && __shfl_sync(FULL, pr.x, q) == __shfl_sync(FULL, pr.y, q)) {
                    const float e0 = __shfl_sync(FULL, eh[0], q), e1 = __shfl_sync(FULL, eh[1], q);
#pragma unroll
                    for (int u = 0; u < RPL; ++u) {
                        bacc[u] -= dot2(a[u].x, e0, a[u].y, e1);
                        dU[u] += dot2(a[u].x, a[u].x, a[u].y, a[u].y);
                    }
                }
            }
            __syncwarp();  // this half may be refilled
        }
    }
#pragma unroll
    for (int u = 0; u < RPL; ++u) {
        const int r = RPL * rg + u;
        if (r >= ci) continue;
#pragma unroll
        for (int v = 0; v < CPL; ++v) {
            const int c = CPL * cg + v;
            if (c < cj) out[r * cj + c] = DIAG && r == c ? fmaf(lambda, clampT(dU[u]), acc[u][v]) : acc[u][v];
        }
        if (DIAG && cg == 0) b[r] = bacc[u];
    }
}

constexpr int VB32_WARPS = 1;  // per CTA: a block of many pairs holds back no others (1: 173 us, 2: 184, 4: 178)
__global__ void __launch_bounds__(32 * VB32_WARPS) k_vbi_blocks32(int n, const int *__restrict__ row_ptr,
                                                      int64_t nnzb, const int *__restrict__ brow,
                                                      const int *__restrict__ col, const int *__restrict__ cdim,
                                                      const int *__restrict__ jc0, const int *__restrict__ off,
                                                      const int64_t *__restrict__ boff, const int *__restrict__ pptr,
                                                      const int2 *__restrict__ plist, const float *__restrict__ J,
                                                      const float *__restrict__ PE, double lambda,
                                                      float *__restrict__ val, float *__restrict__ b) {
    __shared__ __align__(16) float stage[VB32_WARPS][2 * VB32_FETCH * 48];
    // the diagonal blocks (every observation of a camera) first: they have the
    // most pairs, and one started last would run alone
    int64_t k = blockIdx.x * (int64_t)VB32_WARPS + (threadIdx.x >> 5);
    const bool first = k < n;
    if (first)
        k = row_ptr[k];
    else
        k -= n;
    if (k >= nnzb) return;
    const int i = brow[k], j = col[k], ci = cdim[i], cj = cdim[j], p0 = pptr[k], p1 = pptr[k + 1];
    if (!first && i == j) return;
    const int ai = jc0 ? jc0[i] : 0, aj = jc0 ? jc0[j] : 0;
    float *out = val + boff[k], *bi = b + off[i];
    const float lam = (float)lambda;
    // up to 4 x 2 = 8 rows and 8 x 1 columns, or 12 rows and 16 columns (c <= 11)
    if (i == j) {
        if (ci <= 8)
            vbi32_block<2, 1, true>(p0, p1, ci, cj, ai, aj, plist, J, PE, lam, out, bi, stage[threadIdx.x >> 5]);
        else
            vbi32_block<3, 2, true>(p0, p1, ci, cj, ai, aj, plist, J, PE, lam, out, bi, stage[threadIdx.x >> 5]);
    } else if (ci <= 8) {
        if (cj <= 8)
            vbi32_block<2, 1, false>(p0, p1, ci, cj, ai, aj, plist, J, PE, lam, out, bi, stage[threadIdx.x >> 5]);
        else
            vbi32_block<2, 2, false>(p0, p1, ci, cj, ai, aj, plist, J, PE, lam, out, bi, stage[threadIdx.x >> 5]);
    } else {
        if (cj <= 8)
            vbi32_block<3, 1, false>(p0, p1, ci, cj, ai, aj, plist, J, PE, lam, out, bi, stage[threadIdx.x >> 5]);
        else
            vbi32_block<3, 2, false>(p0, p1, ci, cj, ai, aj, plist, J, PE, lam, out, bi, stage[threadIdx.x >> 5]);
    }
}

// FP64: an SM issues one FP64 warp instruction per 16 cycles, so the pairs are
// staged four at a time (J_c,a and M J_c,b in the warp's shared memory, 6 FP64
// instructions per four pairs) and every lane adds its four entries of the
// block with 8 per pair (32 before, M and the products formed pair by pair).
// A block of more than VB64_SPLIT pairs (a diagonal block, mostly) is shared by
// the CTA's VB64_WARPS warps, which take batches of 32 pairs in turn and join their
// sums in shared memory.  1778 -> 297 us at 120 cameras (half of them c = 11),
// 58,000 observations.
constexpr int VB64_SPLIT = 96;
constexpr int VB64_WARPS = 8;
struct Vbi64Sums {
    double acc[VB_NT], du, bacc;  // entries lane + 32 t; row `lane`'s U diagonal and b
};
// pairs p0 + 32 (first + k step), ... of a block into s
__device__ __forceinline__ void vbi64_pairs(int p0, int p1, int first, int step, int ci, int cj, int ai, int aj,
                                            bool diag, const int2 *__restrict__ plist, const double2 *__restrict__ J2,
                                            const double *__restrict__ PE, double *sm, Vbi64Sums &s) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int SP = 4;  // pairs staged at a time
    const int lane = threadIdx.x & 31, nel = ci * cj;
    double *sA = sm, *sT = sm + SP * 2 * VB_CI;  // [pair][row][column]
    int er[VB_NT], ec[VB_NT];
#pragma unroll
    for (int t = 0; t < VB_NT; ++t) {
        const int E = lane + 32 * t;
        er[t] = E < nel ? E / cj : 0;
        ec[t] = E < nel ? E - er[t] * cj : 0;
    }
    for (int pb = p0 + 32 * first; pb < p1; pb += 32 * step) {
        const int cnt = min(32, p1 - pb);
        int2 pr = make_int2(0, 0);
        double M[4] = {0.0, 0.0, 0.0, 0.0}, eh[2] = {0.0, 0.0};
        if (lane < cnt) {
            pr = __ldg(plist + pb + lane);
            vbi_middle<double>(PE + (int64_t)pr.x * VPW, PE + (int64_t)pr.y * VPW, pr.x == pr.y, M, eh);
        }
        for (int q0 = 0; q0 < cnt; q0 += SP) {
            // stage: item (pair, row, column) over the lanes
            double av[3], tv[3];
#pragma unroll
            for (int h = 0; h < 3; ++h) {
                const int it = lane + 32 * h, qq = it / (2 * VB_CI), rem = it - qq * 2 * VB_CI;
                const int u = rem >= VB_CI ? 1 : 0, c = rem - u * VB_CI, q = min(q0 + qq, 31);
                const int x = __shfl_sync(FULL, pr.x, q), y = __shfl_sync(FULL, pr.y, q);
                const double m0 = __shfl_sync(FULL, M[0], q), m1 = __shfl_sync(FULL, M[1], q),
                             m2 = __shfl_sync(FULL, M[2], q), m3 = __shfl_sync(FULL, M[3], q);
                const bool on = qq < SP && q0 + qq < cnt;
                double2 a = make_double2(0.0, 0.0), w = a;
                if (on && c < ci) a = __ldg(J2 + (int64_t)x * (VJW / 2) + ai + c);
                if (on && c < cj) w = __ldg(J2 + (int64_t)y * (VJW / 2) + aj + c);
                av[h] = u ? a.y : a.x;
                tv[h] = (u ? m2 : m0) * w.x + (u ? m3 : m1) * w.y;
            }
            __syncwarp();
#pragma unroll
            for (int h = 0; h < 3; ++h) {
                const int it = lane + 32 * h;
                if (it < SP * 2 * VB_CI) {
                    sA[it] = av[h];
                    sT[it] = tv[h];
                }
            }
            __syncwarp();
#pragma unroll
            for (int qq = 0; qq < SP; ++qq) {
                const double *A = sA + qq * 2 * VB_CI, *Tq = sT + qq * 2 * VB_CI;
#pragma unroll
                for (int t = 0; t < VB_NT; ++t) {
                    if (32 * t >= nel) break;
                    s.acc[t] = fma(A[er[t]], Tq[ec[t]], s.acc[t]);
                    s.acc[t] = fma(A[VB_CI + er[t]], Tq[VB_CI + ec[t]], s.acc[t]);
                }
                if (diag) {
                    const int q = min(q0 + qq, 31);
                    const bool same = q0 + qq < cnt && __shfl_sync(FULL, pr.x, q) == __shfl_sync(FULL, pr.y, q);
                    const double e0 = __shfl_sync(FULL, eh[0], q), e1 = __shfl_sync(FULL, eh[1], q);
                    if (same && lane < ci) {
                        const double j0 = A[lane], j1 = A[VB_CI + lane];
                        s.du = fma(j0, j0, s.du);
                        s.du = fma(j1, j1, s.du);
                        s.bacc = fma(-j0, e0, s.bacc);
                        s.bacc = fma(-j1, e1, s.bacc);
                    }
                }
            }
        }
    }
}
__global__ void __launch_bounds__(32 * VB64_WARPS) k_vbi_blocks64(int64_t nnzb, const int *__restrict__ brow,
                                                      const int *__restrict__ col, const int *__restrict__ cdim,
                                                      const int *__restrict__ jc0, const int *__restrict__ off,
                                                      const int64_t *__restrict__ boff, const int *__restrict__ pptr,
                                                      const int2 *__restrict__ plist, const double *__restrict__ J,
                                                      const double *__restrict__ PE, double lambda,
                                                      double *__restrict__ val, double *__restrict__ b) {
    __shared__ double sm[VB64_WARPS][2 * 4 * 2 * VB_CI];     // staging per warp
    __shared__ double join[VB64_WARPS][(VB_NT + 2) * 32];    // a shared block's sums per warp
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double2 *J2 = reinterpret_cast<const double2 *>(J);
    auto finish = [&](int64_t k, int i, int cj, int nel, int ci, bool diag, const Vbi64Sums &s) {
#pragma unroll
        for (int t = 0; t < VB_NT; ++t) {
            const int E = lane + 32 * t, r = E / cj, c = E - r * cj;
            const double d = __shfl_sync(0xffffffffu, s.du, min(r, 31));
            if (E < nel) val[boff[k] + E] = diag && r == c ? fma(lambda, clampT(d), s.acc[t]) : s.acc[t];
        }
        if (diag && lane < ci) b[off[i] + lane] = s.bacc;
    };
    {
        const int64_t k0 = blockIdx.x * (int64_t)VB64_WARPS;
        const int nb = (int)min((int64_t)VB64_WARPS, nnzb - k0);
        // blocks of few pairs: one to a warp
        if (w < nb) {
            const int64_t k = k0 + w;
            const int p0 = pptr[k], p1 = pptr[k + 1];
            if (p1 - p0 <= VB64_SPLIT) {
                const int i = brow[k], j = col[k], ci = cdim[i], cj = cdim[j];
                Vbi64Sums s = {};
                vbi64_pairs(p0, p1, 0, 1, ci, cj, jc0 ? jc0[i] : 0, jc0 ? jc0[j] : 0, i == j, plist, J2, PE, sm[w], s);
                finish(k, i, cj, ci * cj, ci, i == j, s);
            }
        }
        // the others: the CTA's warps together
        for (int q = 0; q < nb; ++q) {
            const int64_t k = k0 + q;
            const int p0 = pptr[k], p1 = pptr[k + 1];
            if (p1 - p0 <= VB64_SPLIT) continue;  // CTA-uniform
            const int i = brow[k], j = col[k], ci = cdim[i], cj = cdim[j];
            Vbi64Sums s = {};
            vbi64_pairs(p0, p1, w, VB64_WARPS, ci, cj, jc0 ? jc0[i] : 0, jc0 ? jc0[j] : 0, i == j, plist, J2, PE, sm[w], s);
            __syncthreads();  // the previous block's sums have been read
#pragma unroll
            for (int t = 0; t < VB_NT; ++t) join[w][32 * t + lane] = s.acc[t];
            join[w][32 * VB_NT + lane] = s.du;
            join[w][32 * (VB_NT + 1) + lane] = s.bacc;
            __syncthreads();
            if (w == q % VB64_WARPS) {
                s = {};
                for (int h = 0; h < VB64_WARPS; ++h) {
#pragma unroll
                    for (int t = 0; t < VB_NT; ++t) s.acc[t] += join[h][32 * t + lane];
                    s.du += join[h][32 * VB_NT + lane];
                    s.bacc += join[h][32 * (VB_NT + 1) + lane];
                }
                finish(k, i, cj, ci * cj, ci, i == j, s);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// LM iteration with interiors: Eq. 5, the trial state and its cost, and the
// model decrease of the gain ratio (all FP64)
// ---------------------------------------------------------------------------

// Eq. 5, first half: per observation J_p,a^T (J_c,a dx_c) in FP64 (the sum over
// the camera's c_i columns; dxc is the solve's vector, c_i entries per camera at
// off[i]) into `g`, three doubles at the start of the observation's factor row
// (rewritten by the next formation).  A thread per observation, so that no
// thread waits for a longer track.
template <typename T>
__global__ void __launch_bounds__(256) k_vbi_jdx(int64_t m, const int *__restrict__ ocam, const T *__restrict__ J,
                                                 const int *__restrict__ cdim, const int *__restrict__ off,
                                                 const T *__restrict__ dxc, T *__restrict__ g) {
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < m; a += (int64_t)gridDim.x * blockDim.x) {
        const int i = __ldg(ocam + a), ci = __ldg(cdim + i);
        const T *dc = dxc + __ldg(off + i);
        T o[VJW];
        load_vec<VJW>(J + a * VJW, o);
        double t0 = 0.0, t1 = 0.0;
#pragma unroll
        for (int c = 0; c < VB_CI; ++c) {
            if (c >= ci) break;
            const double d = widen(__ldg(dc + c));
            t0 = fma(widen(o[2 * c]), d, t0);
            t1 = fma(widen(o[2 * c + 1]), d, t1);
        }
        double *w = reinterpret_cast<double *>(g + a * VPW);
        double c3[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) c3[q] = fma(widen(o[VJP + q]), t0, widen(o[VJP + 3 + q]) * t1);
        *reinterpret_cast<double2 *>(w) = make_double2(c3[0], c3[1]);
        w[2] = c3[2];
    }
}

// Eq. 5, second half, per point (in the order of track lengths): with V^-1 =
// M^T M and q = M l_p, dx_p = M^T (q - M sum_a J_p,a^T J_c,a dx_c), and the
// trial point X + dx_p.  One pass over tracks and FP64 conversions of every J_c
// value by a thread per point took 261 us at 485,000 observations; the two
// kernels take 56.
template <typename T>
__global__ void __launch_bounds__(128) k_vbi_dxp(int64_t P, const int *__restrict__ ord,
                                                 const int *__restrict__ trk_ptr, const T *__restrict__ g,
                                                 const double *__restrict__ Mq, const double *__restrict__ pts,
                                                 double *__restrict__ dxp, double *__restrict__ pts_t) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < P; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = __ldg(ord + x);
        double s0 = 0.0, s1 = 0.0, s2 = 0.0;
        const int a1 = __ldg(trk_ptr + k + 1);
        for (int a = __ldg(trk_ptr + k); a < a1; ++a) {
            const double *w = reinterpret_cast<const double *>(g + (int64_t)a * VPW);
            const double2 u = *reinterpret_cast<const double2 *>(w);
            s0 += u.x;
            s1 += u.y;
            s2 += w[2];
        }
        const double *w = Mq + 9 * k;
        const double m00 = w[0], m10 = w[1], m11 = w[2], m20 = w[3], m21 = w[4], m22 = w[5];
        const double u0 = w[6] - m00 * s0, u1 = w[7] - (m10 * s0 + m11 * s1),
                     u2 = w[8] - (m20 * s0 + m21 * s1 + m22 * s2);
        const double d[3] = {m00 * u0 + m10 * u1 + m20 * u2, m11 * u1 + m21 * u2, m22 * u2};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            dxp[3 * k + q] = d[q];
            pts_t[3 * k + q] = pts[3 * k + q] + d[q];
        }
    }
}

// The trial cameras: the pose perturbed in the camera frame,
// R <- Exp(d_omega) R, t <- Exp(d_omega) t + dt (unit quaternions), and the
// interiors of a self-calibrating camera (c_i = 11) moved additively; also the
// trial cameras' [R, t].
template <typename T>
__global__ void k_vbi_update_cams(int n, const double *__restrict__ cams, const double *__restrict__ intr,
                                  const int *__restrict__ cdim, const int *__restrict__ off, const T *__restrict__ dxc,
                                  double *__restrict__ cams_t, double *__restrict__ intr_t,
                                  double *__restrict__ camc_t) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const T *dc = dxc + off[i];
    double w[3], q[4], qd[4], qn[4], Rd[9];
    const double dw[3] = {(double)dc[0], (double)dc[1], (double)dc[2]};
    quat_exp(cams + 6 * i, q);
    quat_exp(dw, qd);
    quat_mul(qd, q, qn);
    const double nn = rsqrt(qn[0] * qn[0] + qn[1] * qn[1] + qn[2] * qn[2] + qn[3] * qn[3]);
    for (int k = 0; k < 4; ++k) qn[k] *= nn;
    quat_log(qn, w);
    quat_to_R(qd, Rd);
    const double *t = cams + 6 * i + 3;
    for (int r = 0; r < 3; ++r) {
        cams_t[6 * i + r] = w[r];
        cams_t[6 * i + 3 + r] = Rd[3 * r] * t[0] + Rd[3 * r + 1] * t[1] + Rd[3 * r + 2] * t[2] + (double)dc[3 + r];
    }
    vbi_camera(cams_t + 6 * i, camc_t + 12 * i);
    const bool self_cal = cdim[i] == VB_CI;
    for (int r = 0; r < 5; ++r) intr_t[5 * i + r] = intr[5 * i + r] + (self_cal ? (double)dc[6 + r] : 0.0);
}

// Per observation the trial residual (trial cost, camc_t the trial cameras'
// [R, t]) and the model decrease term -(2 e^T J dx + ||J dx||^2),
// J dx = J_c dx_c (c_i columns) + J_p dx_p; both summed in FP64, plus the
// trial cheirality count.
template <typename T>
__global__ void __launch_bounds__(256) k_vbi_trial(int64_t m, const int *__restrict__ ocam,
                                                   const int *__restrict__ opt, const double *__restrict__ uv,
                                                   const T *__restrict__ J, const int *__restrict__ cdim,
                                                   const int *__restrict__ off, const T *__restrict__ dxc,
                                                   const double *__restrict__ dxp, const double *__restrict__ camc_t,
                                                   const double *__restrict__ intr_t, const double *__restrict__ pts_t,
                                                   VbiScalars *sc, double *red, unsigned *ctr) {
    double v[3] = {0.0, 0.0, 0.0};
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < m; a += (int64_t)gridDim.x * blockDim.x) {
        const int i = ocam[a], k = opt[a], ci = cdim[i];
        const VbiProj<T> pr = vbi_project<T>(camc_t, intr_t, pts_t, i, k, uv + 2 * a);
        const double e0 = widen(pr.e0), e1 = widen(pr.e1);
        v[0] += e0 * e0 + e1 * e1;
        v[2] += pr.Xc[2] <= T(1e-6) ? 1.0 : 0.0;
        T o[VJW];
        load_vec<VJW>(J + a * VJW, o);
        const T *dc = dxc + off[i];
        T t0 = T(0), t1 = T(0);
#pragma unroll
        for (int c = 0; c < VB_CI; ++c) {
            if (c >= ci) break;
            const T d = __ldg(dc + c);
            t0 = fma(o[2 * c], d, t0);
            t1 = fma(o[2 * c + 1], d, t1);
        }
        for (int c = 0; c < 3; ++c) {
            t0 += o[VJP + c] * (T)dxp[3 * (int64_t)k + c];
            t1 += o[VJP + 3 + c] * (T)dxp[3 * (int64_t)k + c];
        }
        v[1] -= widen(t0 * (T(2) * o[VJE] + t0) + t1 * (T(2) * o[VJE + 1] + t1));
    }
    grid_sum<3>(v, red, ctr, [&](double *t) {
        sc->cost_trial = 0.5 * t[0];
        sc->model = 0.5 * t[1];
        sc->n_cheir_trial = (unsigned long long)t[2];
    });
}

}  // namespace ba

using namespace ba;

namespace {

bool finite_n(const double *x, int64_t cnt) {
    for (int64_t k = 0; k < cnt; ++k)
        if (!std::isfinite(x[k])) return false;
    return true;
}

// Temporary device buffers of one formation, freed on every exit.
struct Scratch {
    std::vector<void *> ptrs;
    cudaError_t alloc(void **d, size_t bytes) {
        cudaError_t e = cudaMalloc(d, bytes < 16 ? 16 : bytes);
        if (e == cudaSuccess) ptrs.push_back(*d);
        return e;
    }
    cudaError_t put(void **d, const void *src, size_t bytes) {
        cudaError_t e = alloc(d, bytes);
        return e != cudaSuccess ? e : cudaMemcpy(*d, src, bytes, cudaMemcpyHostToDevice);
    }
    ~Scratch() {
        for (void *p : ptrs) cudaFree(p);
    }
};

// The block pattern and the slot-pair lists of k_vbi_blocks.  Every
// observation a (internal order: by point, then camera) has ns slots, slot s
// in block blk(a, s).  The pattern holds every diagonal block and each
// (beta <= gamma) that two slots of one point fall in; the pairs of a block
// are, point by point in track order, the ordered slot pairs (x in beta,
// y in gamma) - all of them when beta == gamma - stored as their
// observations.
struct VbiLayout {
    std::vector<int32_t> row_ptr, col, pptr;
    std::vector<int2> plist;
};

template <class Blk>
ba_status vbi_layout(int32_t nblk, int64_t P, const std::vector<int32_t> &trk_ptr, int ns, Blk blk, VbiLayout &L) {
    std::vector<uint64_t> keys;
    keys.reserve((size_t)nblk + trk_ptr[P] * 4);
    for (int32_t b = 0; b < nblk; ++b) keys.push_back((uint64_t)b * nblk + b);
    std::vector<int32_t> sb;
    for (int64_t k = 0; k < P; ++k) {
        sb.clear();
        for (int32_t a = trk_ptr[k]; a < trk_ptr[k + 1]; ++a)
            for (int s = 0; s < ns; ++s) sb.push_back(blk(a, s));
        for (size_t x = 0; x < sb.size(); ++x)
            for (size_t y = 0; y < sb.size(); ++y)
                if (sb[x] < sb[y]) keys.push_back((uint64_t)sb[x] * nblk + sb[y]);
    }
    std::sort(keys.begin(), keys.end());
    keys.erase(std::unique(keys.begin(), keys.end()), keys.end());
    if ((int64_t)keys.size() >= (int64_t)INT32_MAX) return set_error(BA_ERR_INVALID_ARG, "too many RCS blocks");
    L.row_ptr.assign(nblk + 1, 0);
    L.col.resize(keys.size());
    for (size_t q = 0; q < keys.size(); ++q) {
        L.row_ptr[keys[q] / nblk + 1]++;
        L.col[q] = (int32_t)(keys[q] % nblk);
    }
    for (int32_t b = 0; b < nblk; ++b) L.row_ptr[b + 1] += L.row_ptr[b];
    const int64_t nnzb = (int64_t)keys.size();
    auto block_of = [&](int32_t beta, int32_t gamma) {
        const int32_t *c0 = L.col.data() + L.row_ptr[beta], *c1 = L.col.data() + L.row_ptr[beta + 1];
        return (int64_t)(std::lower_bound(c0, c1, gamma) - L.col.data());
    };
    std::vector<int64_t> cnt(nnzb + 1, 0);
    std::vector<std::pair<int32_t, int32_t>> sl;  // (block, observation) of the point's slots
    auto each_pair = [&](auto &&fn) {
        for (int64_t k = 0; k < P; ++k) {
            sl.clear();
            for (int32_t a = trk_ptr[k]; a < trk_ptr[k + 1]; ++a)
                for (int s = 0; s < ns; ++s) sl.emplace_back(blk(a, s), a);
            for (size_t x = 0; x < sl.size(); ++x)
                for (size_t y = 0; y < sl.size(); ++y)
                    if (sl[x].first <= sl[y].first) fn(block_of(sl[x].first, sl[y].first), sl[x].second, sl[y].second);
        }
    };
    each_pair([&](int64_t b, int32_t, int32_t) { cnt[b + 1]++; });
    for (int64_t b = 0; b < nnzb; ++b) cnt[b + 1] += cnt[b];
    if (cnt[nnzb] >= (int64_t)INT32_MAX) return set_error(BA_ERR_INVALID_ARG, "more than 2^31 slot pairs");
    L.pptr.assign(cnt.begin(), cnt.end());
    L.plist.resize(cnt[nnzb]);
    std::vector<int64_t> fill(cnt.begin(), cnt.end() - 1);
    each_pair([&](int64_t b, int32_t x, int32_t y) { L.plist[fill[b]++] = make_int2(x, y); });
    return BA_OK;
}

// The points in the order of their track lengths (stable).
std::vector<int32_t> order_by_length(const std::vector<int32_t> &trk_ptr, int64_t P) {
    int32_t most = 0;
    for (int64_t k = 0; k < P; ++k) most = std::max(most, trk_ptr[k + 1] - trk_ptr[k]);
    std::vector<int64_t> at((size_t)most + 2, 0);
    for (int64_t k = 0; k < P; ++k) at[trk_ptr[k + 1] - trk_ptr[k] + 1]++;
    for (int32_t l = 0; l <= most; ++l) at[l + 1] += at[l];
    std::vector<int32_t> ord(P);
    for (int64_t k = 0; k < P; ++k) ord[at[trk_ptr[k + 1] - trk_ptr[k]]++] = (int32_t)k;
    return ord;
}

// Device inputs of the formation, owned by the caller of vbi_form.
struct VbiDev {
    int *ocam = nullptr, *opt = nullptr, *trk = nullptr, *pptr = nullptr, *jc0 = nullptr, *err = nullptr;
    int *ord = nullptr;  // points by track length
    int2 *plist = nullptr;
    double *uv = nullptr, *Mq = nullptr, *camc = nullptr;  // Mq: 9 values per point (k_vbi_factor)
    void *J = nullptr, *PE = nullptr;  // rows in the storage precision: VJW and VPW values per observation
};

// e and J at (cams, intr, pts): the cameras' [R, t] into d.camc, then the rows
// and, with sc, their cost.
template <typename T>
cudaError_t vbi_linearize_T(ba_vbsmc *h, const VbiDev &d, int64_t m, int n, const double *cams, const double *intr,
                            const double *pts, VbiScalars *sc, double *red, unsigned *ctr) {
    k_vbi_camcache<<<(n + 31) / 32, 32, 0, h->st>>>(n, cams, d.camc);
    const int g = (int)std::min<int64_t>((m + VLT - 1) / VLT, 152 * 16);
    k_vbi_linearize<T><<<g, VLT, 0, h->st>>>(m, d.ocam, d.opt, d.uv, d.camc, intr, pts, (T *)d.J, sc, red, ctr);
    return cudaGetLastError();
}
cudaError_t vbi_linearize(ba_vbsmc *h, const VbiDev &d, int64_t m, int n, const double *cams, const double *intr,
                          const double *pts, VbiScalars *sc = nullptr, double *red = nullptr,
                          unsigned *ctr = nullptr) {
    return h->fp32 ? vbi_linearize_T<float>(h, d, m, n, cams, intr, pts, sc, red, ctr)
                   : vbi_linearize_T<double>(h, d, m, n, cams, intr, pts, sc, red, ctr);
}

// From the stored rows: M and q per point, the factor rows, then the damped
// RCS into h's values and b (queued on h's stream; M^-1 is left to vb_finish).
template <typename T>
void vbi_factor_T(ba_vbsmc *h, const VbiDev &d, int64_t P, int64_t m, double lambda) {
    const int gp = (int)std::min<int64_t>((P + 127) / 128, 152 * 16), gm = (int)std::min<int64_t>((m + 255) / 256, 152 * 16);
    k_vbi_factor<T><<<gp, 128, 0, h->st>>>(P, d.ord, d.trk, (const T *)d.J, lambda, d.Mq, d.err);
    k_vbi_rows<T><<<gm, 256, 0, h->st>>>(m, d.opt, (const T *)d.J, d.Mq, (T *)d.PE);
}
cudaError_t vbi_form(ba_vbsmc *h, const VbiDev &d, int64_t P, int64_t m, double lambda) {
    cudaError_t e = cudaMemsetAsync(d.err, 0, sizeof(int), h->st);
    if (e != cudaSuccess) return e;
    if (h->fp32) {
        vbi_factor_T<float>(h, d, P, m, lambda);
        const int64_t g = (h->n + h->nnzb + VB32_WARPS - 1) / VB32_WARPS;
        k_vbi_blocks32<<<(unsigned)g, 32 * VB32_WARPS, 0, h->st>>>(
            h->n, h->row_ptr, h->nnzb, h->brow, h->col, h->cdim, d.jc0, h->off, h->boff, d.pptr, d.plist, (const float *)d.J,
            (const float *)d.PE, lambda, (float *)h->val, (float *)h->b);
    } else {
        vbi_factor_T<double>(h, d, P, m, lambda);
        const int64_t g = (h->nnzb + VB64_WARPS - 1) / VB64_WARPS;
        k_vbi_blocks64<<<(unsigned)g, 32 * VB64_WARPS, 0, h->st>>>(
            h->nnzb, h->brow, h->col, h->cdim, d.jc0, h->off, h->boff, d.pptr, d.plist, (const double *)d.J,
            (const double *)d.PE, lambda, (double *)h->val, (double *)h->b);
    }
    return cudaGetLastError();
}

// Eq. 5 and the trial state of an LM step from the solution dxc: the points
// and the cameras (with their [R, t]); then, after ev, the trial cost.
struct VbiTrial {
    const double *cams, *intr, *pts;
    double *cams_t, *intr_t, *pts_t, *camc_t, *dxp;
    VbiScalars *sc;
    double *red;
    unsigned *ctr;
};
template <typename T>
cudaError_t vbi_trial_T(ba_vbsmc *h, const VbiDev &d, int64_t P, int64_t m, int n, const VbiTrial &t, cudaEvent_t ev) {
    const T *dxc = (const T *)h->vec[0];
    const int gp = (int)std::min<int64_t>((P + 127) / 128, 152 * 16), gm = (int)std::min<int64_t>((m + 255) / 256, 152 * 16);
    const int go = (int)std::min<int64_t>((m + 255) / 256, 152 * 4);
    k_vbi_jdx<T><<<gm, 256, 0, h->st>>>(m, d.ocam, (const T *)d.J, h->cdim, h->off, dxc, (T *)d.PE);
    k_vbi_dxp<T><<<gp, 128, 0, h->st>>>(P, d.ord, d.trk, (const T *)d.PE, d.Mq, t.pts, t.dxp, t.pts_t);
    k_vbi_update_cams<T><<<(n + 31) / 32, 32, 0, h->st>>>(n, t.cams, t.intr, h->cdim, h->off, dxc, t.cams_t, t.intr_t,
                                                          t.camc_t);
    const cudaError_t e = cudaEventRecord(ev, h->st);
    if (e != cudaSuccess) return e;
    k_vbi_trial<T><<<go, 256, 0, h->st>>>(m, d.ocam, d.opt, d.uv, (const T *)d.J, h->cdim, h->off, dxc, t.dxp, t.camc_t,
                                          t.intr_t, t.pts_t, t.sc, t.red, t.ctr);
    return cudaGetLastError();
}

// One-shot formation of a variable-size RCS (the two creation entry points).
ba_status vbi_create(const ba_options &o, int32_t nblk, const std::vector<int32_t> &cdim,
                     const std::vector<int32_t> *jc0, const HostSetup &hs, const VbiLayout &L, int64_t n_pts,
                     int64_t n_obs, const std::vector<double> &uv, const double *cams, int32_t n_cams,
                     const std::vector<double> &intr, const std::vector<double> &ptsi, double lambda, ba_vbsmc **out) {
    ba_vbsmc *h = nullptr;
    ba_status s = vb_build(o, nblk, cdim.data(), (int64_t)L.col.size(), L.row_ptr.data(), L.col.data(), &h);
    if (s) return s;
    Scratch sc;
    VbiDev d;
    double *d_cams = nullptr, *d_intr = nullptr, *d_pts = nullptr;
    cudaError_t e = cudaSuccess;
    auto step = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
    };
    step(sc.put((void **)&d.ocam, hs.obs_cam.data(), n_obs * sizeof(int32_t)));
    step(sc.put((void **)&d.opt, hs.obs_pt.data(), n_obs * sizeof(int32_t)));
    step(sc.put((void **)&d.trk, hs.trk_ptr.data(), (n_pts + 1) * sizeof(int32_t)));
    step(sc.put((void **)&d.ord, order_by_length(hs.trk_ptr, n_pts).data(), n_pts * sizeof(int32_t)));
    step(sc.put((void **)&d.pptr, L.pptr.data(), L.pptr.size() * sizeof(int32_t)));
    step(sc.put((void **)&d.plist, L.plist.data(), L.plist.size() * sizeof(int2)));
    if (jc0) step(sc.put((void **)&d.jc0, jc0->data(), jc0->size() * sizeof(int32_t)));
    step(sc.put((void **)&d.uv, uv.data(), uv.size() * sizeof(double)));
    step(sc.put((void **)&d_cams, cams, (size_t)n_cams * 6 * sizeof(double)));
    step(sc.put((void **)&d_intr, intr.data(), intr.size() * sizeof(double)));
    step(sc.put((void **)&d_pts, ptsi.data(), ptsi.size() * sizeof(double)));
    step(sc.alloc((void **)&d.J, (size_t)n_obs * VJW * h->esz));
    step(sc.alloc((void **)&d.PE, (size_t)n_obs * VPW * h->esz));
    step(sc.alloc((void **)&d.camc, (size_t)n_cams * 12 * sizeof(double)));
    step(sc.alloc((void **)&d.Mq, (size_t)n_pts * 9 * sizeof(double)));
    step(sc.alloc((void **)&d.err, sizeof(int)));
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        ba_vbsmc_destroy(h);
        return set_error(BA_ERR_OOM, "cudaMalloc failed");
    }
    if (e == cudaSuccess) e = vbi_linearize(h, d, n_obs, n_cams, d_cams, d_intr, d_pts);
    if (e == cudaSuccess) e = vbi_form(h, d, n_pts, n_obs, lambda);
    int flag = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&flag, d.err, sizeof(int), cudaMemcpyDeviceToHost, h->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->st);
    if (e != cudaSuccess) {
        ba_vbsmc_destroy(h);
        return set_error(BA_ERR_CUDA, (std::string("forming the RCS with interiors: ") + cudaGetErrorString(e)).c_str());
    }
    if (flag == BA_ERR_NOT_SPD) {
        ba_vbsmc_destroy(h);
        return set_error(BA_ERR_NOT_SPD, "a point's V is not positive definite");
    }
    if ((s = vb_finish(h))) {
        ba_vbsmc_destroy(h);
        return s;
    }
    *out = h;
    return BA_OK;
}

// Observation inputs in the internal order (by point, then camera).
void internal_inputs(const HostSetup &hs, int64_t n_pts, int64_t n_obs, const double *obs_uv, const double *pts,
                     std::vector<double> &uv, std::vector<double> &ptsi) {
    uv.resize(2 * n_obs);
    ptsi.resize(3 * n_pts);
    for (int64_t a = 0; a < n_obs; ++a) {
        uv[2 * a] = obs_uv[2 * hs.obs_perm[a]];
        uv[2 * a + 1] = obs_uv[2 * hs.obs_perm[a] + 1];
    }
    for (int64_t k = 0; k < n_pts; ++k)
        for (int c = 0; c < 3; ++c) ptsi[3 * k + c] = pts[3 * hs.pt_perm[k] + c];
}

ba_status check_scene(int32_t n_cams, const double *cams, int64_t n_pts, const double *pts, int64_t n_obs,
                      const int32_t *obs_cam, const int64_t *obs_pt, const double *obs_uv, double lambda) {
    if (!cams || !pts || !obs_cam || !obs_pt || !obs_uv) return set_error(BA_ERR_INVALID_ARG, "null input array");
    if (n_cams <= 0 || n_pts <= 0 || n_obs <= 0) return set_error(BA_ERR_INVALID_ARG, "sizes must be positive");
    if (!(lambda >= 0.0) || !std::isfinite(lambda)) return set_error(BA_ERR_INVALID_ARG, "lambda must be finite and >= 0");
    if (!finite_n(cams, (int64_t)n_cams * 6) || !finite_n(pts, n_pts * 3) || !finite_n(obs_uv, n_obs * 2))
        return set_error(BA_ERR_NONFINITE, "non-finite camera, point or observation value");
    return BA_OK;
}

}  // namespace

struct ba_vbi_problem {
    ba_options opt{};
    int32_t n = 0;
    int64_t P = 0, m = 0;
    HostSetup hs;
    std::vector<int32_t> cdim;
    ba_vbsmc *h = nullptr;  // the RCS storage, its block-Jacobi M^-1 and PCG
    VbiDev d;
    double *cams = nullptr, *intr = nullptr, *pts = nullptr, *cams_t = nullptr, *intr_t = nullptr, *pts_t = nullptr;
    double *dxp = nullptr, *red = nullptr, *camc_t = nullptr;
    unsigned *ctr = nullptr;
    VbiScalars *sc = nullptr, *sc_host = nullptr;
    std::vector<void *> allocs;
    cudaEvent_t ev[6] = {};
    double lambda = 1e-4, nu = 2.0, F = 0.0;
    bool linearized = false, stepped = false, dead = false;
    int64_t dev_bytes = 0;
};

namespace {

ba_status vbi_fail(ba_vbi_problem *p, cudaError_t e, const char *what) {
    if (e == cudaSuccess) return BA_OK;
    p->dead = true;
    return set_error(BA_ERR_CUDA, (std::string(what) + ": " + cudaGetErrorString(e)).c_str());
}

ba_status vbi_alloc(ba_vbi_problem *p, void **dptr, size_t bytes) {
    bytes = bytes < 16 ? 16 : bytes;
    if (p->opt.device_mem_cap && (size_t)p->dev_bytes + p->h->dev_bytes + bytes > p->opt.device_mem_cap)
        return set_error(BA_ERR_OOM, "device_mem_cap reached");
    cudaError_t e = cudaMalloc(dptr, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return set_error(BA_ERR_OOM, "cudaMalloc failed");
    }
    if (e != cudaSuccess) return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    p->allocs.push_back(*dptr);
    p->dev_bytes += (int64_t)bytes;
    return BA_OK;
}

ba_status vbi_put(ba_vbi_problem *p, void **dptr, const void *src, size_t bytes) {
    ba_status s = vbi_alloc(p, dptr, bytes);
    if (s) return s;
    return vbi_fail(p, cudaMemcpy(*dptr, src, bytes, cudaMemcpyHostToDevice), "upload");
}

void vbi_free(ba_vbi_problem *p) {
    if (!p) return;
    if (p->h) {
        cudaStreamSynchronize(p->h->st);
        ba_vbsmc_destroy(p->h);
    }
    for (auto &e : p->ev)
        if (e) cudaEventDestroy(e);
    for (void *q : p->allocs) cudaFree(q);
    if (p->sc_host) cudaFreeHost(p->sc_host);
    delete p;
}

}  // namespace

extern "C" {

ba_status ba_vbsmc_create_interiors(const ba_options *opt, int32_t n_cams, const double *cams, const double *intr,
                                    const int32_t *cdim, int64_t n_pts, const double *pts, int64_t n_obs,
                                    const int32_t *obs_cam, const int64_t *obs_pt, const double *obs_uv, double lambda,
                                    ba_vbsmc **out) {
    if (!out) return set_error(BA_ERR_INVALID_ARG, "null output pointer");
    *out = nullptr;
    ba_options o;
    if (opt) o = *opt; else ba_options_default(&o);
    if (o.precision != BA_FP64 && o.precision != BA_FP32) return set_error(BA_ERR_INVALID_ARG, "bad precision");
    ba_status s = check_scene(n_cams, cams, n_pts, pts, n_obs, obs_cam, obs_pt, obs_uv, lambda);
    if (s) return s;
    if (!intr || !cdim) return set_error(BA_ERR_INVALID_ARG, "null input array");
    for (int32_t i = 0; i < n_cams; ++i)
        if (cdim[i] != 6 && cdim[i] != VB_CI) return set_error(BA_ERR_INVALID_ARG, "cdim must be 6 or 11");
    if (!finite_n(intr, (int64_t)n_cams * 5)) return set_error(BA_ERR_NONFINITE, "non-finite interior value");
    HostSetup hs;
    std::string err;
    s = symbolic_setup(n_cams, n_pts, n_obs, obs_cam, obs_pt, nullptr, OBS_MAX_DEFAULT, true, hs, err);
    if (s) return set_error(s, err.c_str());
    VbiLayout L;
    if ((s = vbi_layout(n_cams, n_pts, hs.trk_ptr, 1, [&](int32_t a, int) { return hs.obs_cam[a]; }, L))) return s;
    std::vector<double> uv, ptsi;
    internal_inputs(hs, n_pts, n_obs, obs_uv, pts, uv, ptsi);
    std::vector<int32_t> cd(cdim, cdim + n_cams);
    std::vector<double> in(intr, intr + 5 * (size_t)n_cams);
    return vbi_create(o, n_cams, cd, nullptr, hs, L, n_pts, n_obs, uv, cams, n_cams, in, ptsi, lambda, out);
}

ba_status ba_vbsmc_create_shared(const ba_options *opt, int32_t n_images, const double *cams, int32_t n_phys,
                                 const double *intr_phys, const int32_t *phys, int64_t n_pts, const double *pts,
                                 int64_t n_obs, const int32_t *obs_cam, const int64_t *obs_pt, const double *obs_uv,
                                 double lambda, ba_vbsmc **out) {
    if (!out) return set_error(BA_ERR_INVALID_ARG, "null output pointer");
    *out = nullptr;
    ba_options o;
    if (opt) o = *opt; else ba_options_default(&o);
    if (o.precision != BA_FP64 && o.precision != BA_FP32) return set_error(BA_ERR_INVALID_ARG, "bad precision");
    ba_status s = check_scene(n_images, cams, n_pts, pts, n_obs, obs_cam, obs_pt, obs_uv, lambda);
    if (s) return s;
    if (!intr_phys || !phys) return set_error(BA_ERR_INVALID_ARG, "null input array");
    if (n_phys <= 0 || (int64_t)n_images + n_phys >= (1 << 30))
        return set_error(BA_ERR_INVALID_ARG, "need 0 < n_phys and n_images + n_phys < 2^30");
    for (int32_t i = 0; i < n_images; ++i)
        if (phys[i] < 0 || phys[i] >= n_phys) return set_error(BA_ERR_INVALID_ARG, "phys index out of range");
    if (!finite_n(intr_phys, (int64_t)n_phys * 5)) return set_error(BA_ERR_NONFINITE, "non-finite interior value");
    HostSetup hs;
    std::string err;
    s = symbolic_setup(n_images, n_pts, n_obs, obs_cam, obs_pt, nullptr, OBS_MAX_DEFAULT, true, hs, err);
    if (s) return set_error(s, err.c_str());
    const int32_t nblk = n_images + n_phys;
    VbiLayout L;
    auto blk = [&](int32_t a, int sl) { return sl == 0 ? hs.obs_cam[a] : n_images + phys[hs.obs_cam[a]]; };
    if ((s = vbi_layout(nblk, n_pts, hs.trk_ptr, 2, blk, L))) return s;
    std::vector<double> uv, ptsi;
    internal_inputs(hs, n_pts, n_obs, obs_uv, pts, uv, ptsi);
    std::vector<int32_t> cd(nblk, 6), jc0(nblk, 0);
    for (int32_t q = n_images; q < nblk; ++q) {
        cd[q] = 5;
        jc0[q] = 6;
    }
    std::vector<double> in(5 * (size_t)n_images);  // each image's interiors: its physical camera's
    for (int32_t i = 0; i < n_images; ++i)
        for (int c = 0; c < 5; ++c) in[5 * i + c] = intr_phys[5 * phys[i] + c];
    return vbi_create(o, nblk, cd, &jc0, hs, L, n_pts, n_obs, uv, cams, n_images, in, ptsi, lambda, out);
}

ba_status ba_vbi_problem_create(const ba_options *opt, int32_t n_cams, const double *cams, const double *intr,
                                const int32_t *cdim, int64_t n_pts, const double *pts, int64_t n_obs,
                                const int32_t *obs_cam, const int64_t *obs_pt, const double *obs_uv,
                                ba_vbi_problem **out) {
    if (!out) return set_error(BA_ERR_INVALID_ARG, "null output pointer");
    *out = nullptr;
    ba_options o;
    if (opt) o = *opt; else ba_options_default(&o);
    if (o.precision != BA_FP64 && o.precision != BA_FP32) return set_error(BA_ERR_INVALID_ARG, "bad precision");
    if (!(o.lambda0 > 0) || !std::isfinite(o.lambda0)) return set_error(BA_ERR_INVALID_ARG, "lambda0 must be > 0");
    if (!(o.pcg_rel_tol > 0) || o.pcg_max_iters < 0) return set_error(BA_ERR_INVALID_ARG, "bad PCG options");
    ba_status s = check_scene(n_cams, cams, n_pts, pts, n_obs, obs_cam, obs_pt, obs_uv, 0.0);
    if (s) return s;
    if (!intr || !cdim) return set_error(BA_ERR_INVALID_ARG, "null input array");
    for (int32_t i = 0; i < n_cams; ++i)
        if (cdim[i] != 6 && cdim[i] != VB_CI) return set_error(BA_ERR_INVALID_ARG, "cdim must be 6 or 11");
    if (!finite_n(intr, (int64_t)n_cams * 5)) return set_error(BA_ERR_NONFINITE, "non-finite interior value");
    ba_vbi_problem *p = new ba_vbi_problem();
    p->opt = o;
    p->n = n_cams;
    p->P = n_pts;
    p->m = n_obs;
    p->lambda = o.lambda0;
    p->cdim.assign(cdim, cdim + n_cams);
    std::string err;
    s = symbolic_setup(n_cams, n_pts, n_obs, obs_cam, obs_pt, nullptr, OBS_MAX_DEFAULT, true, p->hs, err);
    if (s) {
        vbi_free(p);
        return set_error(s, err.c_str());
    }
    VbiLayout L;
    const HostSetup &hs = p->hs;
    if ((s = vbi_layout(n_cams, n_pts, hs.trk_ptr, 1, [&](int32_t a, int) { return hs.obs_cam[a]; }, L))) {
        vbi_free(p);
        return s;
    }
    if ((s = vb_build(o, n_cams, cdim, (int64_t)L.col.size(), L.row_ptr.data(), L.col.data(), &p->h))) {
        p->h = nullptr;
        vbi_free(p);
        return s;
    }
    std::vector<double> uv, ptsi;
    internal_inputs(hs, n_pts, n_obs, obs_uv, pts, uv, ptsi);
    const size_t C6 = (size_t)n_cams * 6 * 8, C5 = (size_t)n_cams * 5 * 8, P3 = (size_t)n_pts * 3 * 8;
    if (!s) s = vbi_put(p, (void **)&p->d.ocam, hs.obs_cam.data(), n_obs * sizeof(int32_t));
    if (!s) s = vbi_put(p, (void **)&p->d.opt, hs.obs_pt.data(), n_obs * sizeof(int32_t));
    if (!s) s = vbi_put(p, (void **)&p->d.trk, hs.trk_ptr.data(), (n_pts + 1) * sizeof(int32_t));
    if (!s) s = vbi_put(p, (void **)&p->d.ord, order_by_length(hs.trk_ptr, n_pts).data(), n_pts * sizeof(int32_t));
    if (!s) s = vbi_put(p, (void **)&p->d.pptr, L.pptr.data(), L.pptr.size() * sizeof(int32_t));
    if (!s) s = vbi_put(p, (void **)&p->d.plist, L.plist.data(), L.plist.size() * sizeof(int2));
    if (!s) s = vbi_put(p, (void **)&p->d.uv, uv.data(), uv.size() * sizeof(double));
    if (!s) s = vbi_alloc(p, (void **)&p->d.J, (size_t)n_obs * VJW * p->h->esz);
    if (!s) s = vbi_alloc(p, (void **)&p->d.PE, (size_t)n_obs * VPW * p->h->esz);
    if (!s) s = vbi_alloc(p, (void **)&p->d.camc, (size_t)n_cams * 12 * sizeof(double));
    if (!s) s = vbi_alloc(p, (void **)&p->camc_t, (size_t)n_cams * 12 * sizeof(double));
    if (!s) s = vbi_alloc(p, (void **)&p->d.Mq, (size_t)n_pts * 9 * sizeof(double));
    if (!s) s = vbi_alloc(p, (void **)&p->d.err, sizeof(int));
    if (!s) s = vbi_put(p, (void **)&p->cams, cams, C6);
    if (!s) s = vbi_put(p, (void **)&p->intr, intr, C5);
    if (!s) s = vbi_put(p, (void **)&p->pts, ptsi.data(), P3);
    if (!s) s = vbi_alloc(p, (void **)&p->cams_t, C6);
    if (!s) s = vbi_alloc(p, (void **)&p->intr_t, C5);
    if (!s) s = vbi_alloc(p, (void **)&p->pts_t, P3);
    if (!s) s = vbi_alloc(p, (void **)&p->dxp, P3);
    if (!s) s = vbi_alloc(p, (void **)&p->red, (size_t)RED_SLOTS * sizeof(double));
    if (!s) s = vbi_alloc(p, (void **)&p->ctr, 64);
    if (!s) s = vbi_alloc(p, (void **)&p->sc, sizeof(VbiScalars));
    if (!s) s = vbi_fail(p, cudaMemset(p->ctr, 0, 64), "memset");
    if (!s) s = vbi_fail(p, cudaMallocHost((void **)&p->sc_host, sizeof(VbiScalars)), "cudaMallocHost");
    for (auto &e : p->ev)
        if (!s) s = vbi_fail(p, cudaEventCreate(&e), "event");
    if (s) {
        vbi_free(p);
        return s;
    }
    *out = p;
    return BA_OK;
}

void ba_vbi_problem_destroy(ba_vbi_problem *p) { vbi_free(p); }

ba_status ba_vbi_lm_step(ba_vbi_problem *p, ba_step_info *info) {
    if (!p) return set_error(BA_ERR_INVALID_ARG, "null problem");
    if (p->dead) return set_error(BA_ERR_STATE, "the problem is unusable after an earlier error");
    ba_vbsmc *h = p->h;
    cudaStream_t st = h->st;
    ba_status s;
    const bool relin = !p->linearized;
    if ((s = vbi_fail(p, cudaEventRecord(p->ev[0], st), "event"))) return s;
    if (relin) {
        if ((s = vbi_fail(p, vbi_linearize(h, p->d, p->m, p->n, p->cams, p->intr, p->pts, p->sc, p->red, p->ctr),
                          "k_vbi_linearize")))
            return s;
    }
    if ((s = vbi_fail(p, cudaEventRecord(p->ev[1], st), "event"))) return s;
    // Eq. 3-4 with c_i unknowns per camera, then the block-Jacobi M^-1
    if ((s = vbi_fail(p, vbi_form(h, p->d, p->P, p->m, p->lambda), "forming the RCS"))) return s;
    int flag = 0;
    if ((s = vbi_fail(p, cudaMemcpyAsync(&flag, p->d.err, sizeof(int), cudaMemcpyDeviceToHost, st), "copy")))
        return s;
    if ((s = vb_finish(h))) {  // synchronises
        if (s != BA_ERR_NOT_SPD) p->dead = true;
        return s;
    }
    if (flag == BA_ERR_NOT_SPD) return set_error(BA_ERR_NOT_SPD, "a point's V is not positive definite");
    if (relin) {
        if ((s = vbi_fail(p, cudaMemcpy(p->sc_host, p->sc, sizeof(VbiScalars), cudaMemcpyDeviceToHost), "copy")))
            return s;
        p->F = p->sc_host->cost;
        p->linearized = true;
    }
    if ((s = vbi_fail(p, cudaEventRecord(p->ev[2], st), "event"))) return s;
    // Sec. 3.2: block-Jacobi PCG on S dx_c = b
    int iters = 0;
    double rel = 0.0;
    s = ba_vbsmc_solve(h, p->opt.pcg_rel_tol, p->opt.pcg_max_iters, nullptr, &iters, &rel, nullptr);
    if (s != BA_OK && s != BA_ERR_NO_CONVERGENCE) {
        if (s != BA_ERR_NOT_SPD) p->dead = true;
        return s;
    }
    if ((s = vbi_fail(p, cudaEventRecord(p->ev[3], st), "event"))) return s;
    // Eq. 5, the trial state, its cost and the model decrease
    const VbiTrial t{p->cams, p->intr, p->pts, p->cams_t, p->intr_t, p->pts_t, p->camc_t, p->dxp, p->sc, p->red,
                     p->ctr + 1};
    const cudaError_t te = h->fp32 ? vbi_trial_T<float>(h, p->d, p->P, p->m, p->n, t, p->ev[4])
                                   : vbi_trial_T<double>(h, p->d, p->P, p->m, p->n, t, p->ev[4]);
    if ((s = vbi_fail(p, te, "trial kernels"))) return s;
    if ((s = vbi_fail(p, cudaEventRecord(p->ev[5], st), "event"))) return s;
    if ((s = vbi_fail(p, cudaMemcpyAsync(p->sc_host, p->sc, sizeof(VbiScalars), cudaMemcpyDeviceToHost, st), "copy")))
        return s;
    if ((s = vbi_fail(p, cudaStreamSynchronize(st), "sync"))) return s;
    // gain ratio and Nielsen's damping rule, as the 6-unknown LM step
    const double F0 = p->F, F1 = p->sc_host->cost_trial, pred = p->sc_host->model;
    const double rho = pred > 0 ? (F0 - F1) / pred : -INFINITY;
    const bool ok = pred > 0 && rho > 1e-3 && std::isfinite(F1);
    ba_step_info loc{};
    loc.cost_before = F0;
    loc.cost_trial = F1;
    loc.predicted = pred;
    loc.rho = rho;
    loc.lambda = p->lambda;
    loc.accepted = ok ? 1 : 0;
    loc.pcg_iters = iters;
    loc.rcs_rel_resid = rel;
    loc.n_cheirality = (int64_t)p->sc_host->n_cheir_trial;
    float ms[5] = {0, 0, 0, 0, 0};
    for (int k = 0; k < 5; ++k) cudaEventElapsedTime(&ms[k], p->ev[k], p->ev[k + 1]);
    loc.ms[0] = ms[0];                  // linearize and cost
    loc.ms[1] = ms[1];                  // RCS formation and M^-1
    loc.ms[2] = ms[2];                  // PCG
    loc.ms[3] = ms[3];                  // Eq. 5 and the trial cameras
    loc.ms[4] = ms[4];                  // trial cost and model decrease
    loc.ms[5] = ms[0] + ms[1] + ms[2] + ms[3] + ms[4];
    if (ok) {
        std::swap(p->cams, p->cams_t);
        std::swap(p->intr, p->intr_t);
        std::swap(p->pts, p->pts_t);
        std::swap(p->d.camc, p->camc_t);
        p->F = F1;
        p->linearized = false;
        p->lambda *= std::max(1.0 / 3.0, 1.0 - std::pow(2.0 * rho - 1.0, 3));
        p->nu = 2.0;
    } else {
        p->lambda *= p->nu;
        p->nu *= 2.0;
    }
    loc.cost_after = ok ? F1 : F0;
    p->stepped = true;
    if (info) *info = loc;
    return BA_OK;
}

ba_status ba_vbi_get_state(const ba_vbi_problem *p, double *cams, double *intr, double *pts) {
    if (!p) return set_error(BA_ERR_INVALID_ARG, "null problem");
    if (p->dead) return set_error(BA_ERR_STATE, "the problem is unusable after an earlier error");
    ba_vbi_problem *q = const_cast<ba_vbi_problem *>(p);
    ba_status s;
    if ((s = vbi_fail(q, cudaStreamSynchronize(p->h->st), "sync"))) return s;
    if (cams && (s = vbi_fail(q, cudaMemcpy(cams, p->cams, (size_t)p->n * 48, cudaMemcpyDeviceToHost), "copy")))
        return s;
    if (intr && (s = vbi_fail(q, cudaMemcpy(intr, p->intr, (size_t)p->n * 40, cudaMemcpyDeviceToHost), "copy")))
        return s;
    // (the points keep the caller's order: pattern-only setup)
    if (pts && (s = vbi_fail(q, cudaMemcpy(pts, p->pts, (size_t)p->P * 24, cudaMemcpyDeviceToHost), "copy")))
        return s;
    return BA_OK;
}

ba_status ba_vbi_set_state(ba_vbi_problem *p, const double *cams, const double *intr, const double *pts,
                           double lambda, double nu) {
    if (!p) return set_error(BA_ERR_INVALID_ARG, "null problem");
    if (p->dead) return set_error(BA_ERR_STATE, "the problem is unusable after an earlier error");
    if (!cams || !intr || !pts) return set_error(BA_ERR_INVALID_ARG, "null input array");
    if (!(lambda > 0) || !std::isfinite(lambda) || !(nu > 0) || !std::isfinite(nu))
        return set_error(BA_ERR_INVALID_ARG, "lambda and nu must be finite and > 0");
    if (!finite_n(cams, (int64_t)p->n * 6) || !finite_n(intr, (int64_t)p->n * 5))
        return set_error(BA_ERR_NONFINITE, "non-finite state value");
    // the points go to the trial points' array and are checked there; the
    // arrays change places only when every value is finite (checked and copied
    // by way of a host vector, this call and ba_vbi_get_state took 0.6 ms more
    // at 99,000 points)
    cudaStream_t st = p->h->st;
    ba_status s;
    unsigned bad = 0, *flag = p->ctr + 15;
    if ((s = vbi_fail(p, cudaMemcpyAsync(p->pts_t, pts, (size_t)p->P * 24, cudaMemcpyHostToDevice, st), "copy"))) return s;
    if ((s = vbi_fail(p, cudaMemsetAsync(flag, 0, sizeof(unsigned), st), "memset"))) return s;
    if ((s = vbi_fail(p, run_count_nonfinite(st, p->pts_t, p->P * 3, flag), "k_count_nonfinite"))) return s;
    if ((s = vbi_fail(p, cudaMemcpyAsync(&bad, flag, sizeof(unsigned), cudaMemcpyDeviceToHost, st), "copy"))) return s;
    if ((s = vbi_fail(p, cudaStreamSynchronize(st), "sync"))) return s;
    if (bad) return set_error(BA_ERR_NONFINITE, "non-finite state value");
    std::swap(p->pts, p->pts_t);
    if ((s = vbi_fail(p, cudaMemcpyAsync(p->cams, cams, (size_t)p->n * 48, cudaMemcpyHostToDevice, st), "copy"))) return s;
    if ((s = vbi_fail(p, cudaMemcpyAsync(p->intr, intr, (size_t)p->n * 40, cudaMemcpyHostToDevice, st), "copy"))) return s;
    if ((s = vbi_fail(p, cudaStreamSynchronize(st), "sync"))) return s;
    p->lambda = lambda;
    p->nu = nu;
    p->linearized = false;
    p->stepped = false;
    return BA_OK;
}

ba_status ba_vbi_get_lm_state(const ba_vbi_problem *p, double *lambda, double *nu, double *cost) {
    if (!p) return set_error(BA_ERR_INVALID_ARG, "null problem");
    if (p->dead) return set_error(BA_ERR_STATE, "the problem is unusable after an earlier error");
    if (lambda) *lambda = p->lambda;
    if (nu) *nu = p->nu;
    if (cost) {
        if (!p->linearized) {  // the cost of the current state
            ba_vbi_problem *q = const_cast<ba_vbi_problem *>(p);
            ba_status s;
            if ((s = vbi_fail(q, vbi_linearize(p->h, p->d, p->m, p->n, p->cams, p->intr, p->pts, p->sc, p->red,
                                               p->ctr), "k_vbi_linearize")))
                return s;
            if ((s = vbi_fail(q, cudaMemcpyAsync(p->sc_host, p->sc, sizeof(VbiScalars), cudaMemcpyDeviceToHost,
                                                 p->h->st), "copy")))
                return s;
            if ((s = vbi_fail(q, cudaStreamSynchronize(p->h->st), "sync"))) return s;
            q->F = p->sc_host->cost;
            q->linearized = true;
        }
        *cost = p->F;
    }
    return BA_OK;
}

ba_status ba_vbi_get_step(const ba_vbi_problem *p, double *dxc, double *dxp) {
    if (!p) return set_error(BA_ERR_INVALID_ARG, "null problem");
    if (p->dead) return set_error(BA_ERR_STATE, "the problem is unusable after an earlier error");
    if (!p->stepped) return set_error(BA_ERR_STATE, "no step taken since creation or the last ba_vbi_set_state");
    ba_vbi_problem *q = const_cast<ba_vbi_problem *>(p);
    ba_status s;
    if ((s = vbi_fail(q, cudaStreamSynchronize(p->h->st), "sync"))) return s;
    if (dxc) {
        std::vector<char> raw(p->h->N * p->h->esz);
        if ((s = vbi_fail(q, cudaMemcpy(raw.data(), p->h->vec[0], raw.size(), cudaMemcpyDeviceToHost), "copy")))
            return s;
        for (int64_t k = 0; k < p->h->N; ++k)
            dxc[k] = p->h->fp32 ? (double)reinterpret_cast<const float *>(raw.data())[k]
                                : reinterpret_cast<const double *>(raw.data())[k];
    }
    if (dxp && (s = vbi_fail(q, cudaMemcpy(dxp, p->dxp, (size_t)p->P * 24, cudaMemcpyDeviceToHost), "copy"))) return s;
    return BA_OK;
}

const ba_vbsmc *ba_vbi_system(const ba_vbi_problem *p) { return p ? p->h : nullptr; }

ba_status ba_vbi_info(const ba_vbi_problem *p, int64_t *n_unknowns, int64_t *n_blocks, int64_t *device_bytes) {
    if (!p) return set_error(BA_ERR_INVALID_ARG, "null problem");
    if (n_unknowns) *n_unknowns = p->h->N;
    if (n_blocks) *n_blocks = p->h->nnzb;
    if (device_bytes) *device_bytes = p->dev_bytes + (int64_t)p->h->dev_bytes;
    return BA_OK;
}

}  // extern "C"
