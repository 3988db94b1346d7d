// Allocation-free block-Jacobi PCG on a caller-owned BSMC system (FP32).
//
// Some callers cannot call cudaMalloc: code that runs while a framework owns
// the device memory pool (a caching allocator, a fixed arena), real-time
// loops that must not take the allocator's lock or its implicit device
// synchronisation, and hosts with a hard device-memory budget.  For them
// ba_pcg_solve_static solves S x = b with the caller's device buffers for the
// inputs and the output, and keeps its own scratch (the PCG vectors z, d, q,
// the block-Jacobi inverses and the reduction slots) in one file-scope
// __device__ array of fixed size.  The array is created when the library is
// loaded on a device and lives until the process exits, on every GPU that
// loads the library.
//
// Every call shares the one array: calls that overlap on the GPU (two streams,
// or two host threads) race on it.  Each call clears the reduction counters
// and the product vector before use; the array otherwise keeps whatever the
// last call left.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "device_util.cuh"

namespace ba {

namespace {

constexpr int kStaticMaxCams = 8192;
constexpr size_t kScalOff = 0;      // StaticScalars
constexpr size_t kRedOff = 512;     // per-CTA partial sums (4096 doubles)
constexpr size_t kVecBytes = (size_t)6 * kStaticMaxCams * sizeof(float);
constexpr size_t kBarOff = kRedOff + 2048 * sizeof(double);  // arrival counters, behind the partials
constexpr size_t kVecOff = kRedOff + 4096 * sizeof(double);  // z, d0, d1, q0, q1
constexpr size_t kMinvOff = kVecOff + 5 * kVecBytes;
constexpr size_t kStaticBytes = kMinvOff + (size_t)36 * kStaticMaxCams * sizeof(float);
static_assert(AR_SUB * 32 * sizeof(unsigned) <= 2048 * sizeof(double), "counters fit behind the partials");
static_assert(kVecOff % 256 == 0 && kVecBytes % 256 == 0 && kMinvOff % 256 == 0, "scratch layout");

struct StaticScalars {
    double rr, rr0;
    int iters, err;
};
static_assert(sizeof(StaticScalars) <= 256, "scalar slot");

static __device__ __align__(256) unsigned char g_pcg_scratch[kStaticBytes];

constexpr size_t kStaticSmem = 216 * 1024;  // dynamic shared memory of the solve at most

constexpr int kMaxDevices = 64;
std::mutex g_mu;
unsigned char *g_ptr[kMaxDevices] = {};

// Block-Jacobi: M_i^-1 = inverse of the first (diagonal) block of row i.
// Row i is checked first: its blocks lie in [0, nnzb), the first is the
// diagonal block and the other columns ascend above i (the upper-triangle
// layout).  A malformed row - for instance one of a matrix stored with both
// triangles, which the two-sided product would count twice - sets
// BA_ERR_INVALID_ARG; a diagonal block that is not SPD sets BA_ERR_NOT_SPD.
// Either error stops the solve before its first iteration.
// Eight lanes per camera (chol6_lanes, FP64).
__global__ void __launch_bounds__(32) k_static_minv(int n, int64_t nnzb, const int *__restrict__ row_ptr,
                                                    const int *__restrict__ col, const float *__restrict__ val,
                                                    float *__restrict__ Minv, StaticScalars *sc) {
    const int i = (blockIdx.x * 32 + threadIdx.x) >> 3, r = threadIdx.x & 7;
    const int rs = i < n ? row_ptr[i] : 0, re = i < n ? row_ptr[i + 1] : 0;
    bool ok = i < n && rs >= 0 && re > rs && (int64_t)re <= nnzb && (i + 1 < n || (int64_t)re == nnzb);
    ok = ok && col[rs] == i;
    for (int k = rs + 1 + r; ok && k < re; k += 8) ok = col[k] > col[k - 1] && col[k] < n;
    ok = (__ballot_sync(0xffffffffu, ok) >> (threadIdx.x & 24) & 0xffu) == 0xffu;  // all eight lanes
    double a[6], x[6], out[6];
    const float *d = val + (int64_t)(ok ? rs : 0) * BW;
#pragma unroll
    for (int c = 0; c < 6; ++c) a[c] = ok && r < 6 ? (double)d[6 * r + c] : 0.0;
    const bool spd = chol6_lanes<double>(a, x);
    inv6_row<double>(x, out);
    if (i >= n || r >= 6) return;
    if (r == 0) {
        if (!ok) atomicExch(&sc->err, (int)BA_ERR_INVALID_ARG);
        else if (!spd) atomicCAS(&sc->err, 0, (int)BA_ERR_NOT_SPD);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) Minv[36 * (int64_t)i + 6 * r + q] = ok && spd ? (float)out[q] : 0.f;
}

// The whole solve in one cooperative launch.  CTA c owns block rows c R ..
// c R + R - 1: thread t keeps x, r, z, d and its row of M^-1 of the CTA's t-th
// vector entry in registers, and the rows' blocks (with their columns) are
// copied to shared memory once, as far as they fit (`cap` blocks; the others
// are read from the caller's arrays each time).  Per iteration a warp per row
// applies each stored block as S_ij d_j to its row and as S_ij^T d_i to q_j
// (vector reductions in L2; q alternates between two buffers, the one of the
// next iteration cleared by its owners), d^T S d is summed per block as (2 for
// j > i, 1 for j = i) d_i^T S_ij d_j, so two grid exchanges per iteration are
// enough.  Every grid wait is bounded (BA_ERR_TIMEOUT).  What bounds it: the
// exchanges (about 3 us each) and the round trip of the neighbours' gather.
// Against two launches per iteration with the vectors in memory and a host
// read-back every eight: 28 -> 11 us per iteration at 1,250 cameras.
constexpr int ST_THREADS = 512;  // at least 6 rows of the largest n on any SM count >= 97
__global__ void __launch_bounds__(ST_THREADS, 1)
    k_static_pcg(int n, int rows, const int *__restrict__ row_ptr, const int *__restrict__ col,
                 const float *__restrict__ val, const float *__restrict__ b, const float *__restrict__ Minv, float *x,
                 float *z, float *d0, float *d1, float *q0, float *q1, StaticScalars *sc, double *red, unsigned *bar,
                 double tol2, int max_iters, int cap, long long limit_cycles) {
    extern __shared__ __align__(16) float s_blk[];  // cap blocks, then their columns
    __shared__ float s_d[ST_THREADS], s_own[ST_THREADS], s_r[ST_THREADS];
    __shared__ double s_ab;
    int *s_col = reinterpret_cast<int *>(s_blk + (size_t)cap * BW);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, comp6 = fold6_comp(lane);
    const int row0 = blockIdx.x * rows, R = min(rows, n - row0);
    const bool own = (int)threadIdx.x < 6 * R;
    const int e = 6 * row0 + threadIdx.x, lrow = threadIdx.x / 6, comp = threadIdx.x - 6 * lrow;
    const int nown = (6 * R + 31) >> 5;
    float M[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, xv = 0.f, rv = 0.f, zv = 0.f, dv = 0.f;
    if (own) {
#pragma unroll
        for (int c = 0; c < 6; ++c) M[c] = Minv[6 * (size_t)e + c];
        rv = b[e];
        s_r[threadIdx.x] = rv;
        d0[e] = 0.f;
        q0[e] = 0.f;
        q1[e] = 0.f;
    }
    __syncthreads();
    auto precond = [&]() {
        const float *r6 = s_r + 6 * lrow;
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < 6; ++c) s = fmaf(M[c], r6[c], s);
        return s;
    };
    unsigned gen = 0;
    double v2[2] = {0.0, 0.0};
    if (own) {
        zv = precond();
        z[e] = zv;
        const double rd = widen(rv);
        v2[0] = rd * widen(zv);
        v2[1] = rd * rd;
    }
    if (!grid_allreduce_w0<2>(v2, red, gen++, bar, &sc->err, limit_cycles, nown, [](const double(&)[2], bool) {}))
        return;
    double rz = v2[0];
    const double rr0 = v2[1];
    auto leave = [&](int it, double rr, int err) {
        if (own) x[e] = xv;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            sc->rr0 = rr0;
            sc->rr = rr;
            sc->iters = it;
            if (err) sc->err = err;
        }
    };
    // a malformed row or an indefinite diagonal block ends the solve here
    if (rr0 == 0.0 || max_iters <= 0 || *(volatile int *)&sc->err != 0) {
        leave(0, rr0, 0);
        return;
    }
    const int k0 = __ldg(row_ptr + row0), nblk = __ldg(row_ptr + row0 + R) - k0, ns = min(nblk, cap);
    for (int q = threadIdx.x; q < ns * BW; q += blockDim.x) s_blk[q] = __ldg(val + (int64_t)k0 * BW + q);
    for (int q = threadIdx.x; q < ns; q += blockDim.x) s_col[q] = __ldg(col + k0 + q);
    double beta = 0.0;
    for (int it = 0;;) {
        const float *dold = (it & 1) ? d1 : d0;
        float *dnew = (it & 1) ? d0 : d1, *q = (it & 1) ? q1 : q0, *qn = (it & 1) ? q0 : q1;
        const float bt = (float)beta;
        if (own) {
            dv = fmaf(bt, dv, zv);
            s_d[threadIdx.x] = dv;
            dnew[e] = dv;
        }
        __syncthreads();  // also: the shared blocks before the first iteration
        double v1[1] = {0.0};
        for (int lr = w; lr < R; lr += ST_THREADS / 32) {
            const int i = row0 + lr, kb = __ldg(row_ptr + i) - k0, ke = __ldg(row_ptr + i + 1) - k0;
            float di[6], acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int c = 0; c < 6; ++c) di[c] = s_d[6 * lr + c];
            for (int k = kb + lane; k < ke; k += 32) {
                float S[36], dj[6];
                int j;
                if (k < ns) {
                    j = s_col[k];
                    const float4 *p = reinterpret_cast<const float4 *>(s_blk + k * BW);
#pragma unroll
                    for (int t = 0; t < 9; ++t) {
                        const float4 u = p[t];
                        S[4 * t] = u.x; S[4 * t + 1] = u.y; S[4 * t + 2] = u.z; S[4 * t + 3] = u.w;
                    }
                } else {
                    j = __ldg(col + k0 + k);
#pragma unroll
                    for (int t = 0; t < 36; ++t) S[t] = __ldg(val + (int64_t)(k0 + k) * BW + t);
                }
                if (j == i) {
#pragma unroll
                    for (int c = 0; c < 6; ++c) dj[c] = di[c];
                } else {
                    float o[6];
                    load6(z + 6 * j, dj);
                    load6(dold + 6 * j, o);
#pragma unroll
                    for (int c = 0; c < 6; ++c) dj[c] = fmaf(bt, o[c], dj[c]);
                }
                double qf = 0.0;
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    float t = 0.f;
#pragma unroll
                    for (int c = 0; c < 6; ++c) t = fmaf(S[6 * r + c], dj[c], t);
                    acc[r] += t;
                    qf = fma(widen(di[r]), widen(t), qf);
                }
                if (j != i) {
                    float u[6];
#pragma unroll
                    for (int c = 0; c < 6; ++c) {
                        u[c] = 0.f;
#pragma unroll
                        for (int r = 0; r < 6; ++r) u[c] = fmaf(S[6 * r + c], di[r], u[c]);
                    }
                    red_add6_f(q + 6 * (int64_t)j, u);
                    qf += qf;
                }
                v1[0] += qf;
            }
            const float t = warp_fold6(acc, lane);
            if (fold6_owner(lane)) s_own[6 * lr + comp6] = t;
        }
        __syncthreads();
        if (!grid_allreduce_w0<1>(v1, red, gen++, bar, &sc->err, limit_cycles, min(R, ST_THREADS / 32),
                                  [&](const double(&t)[1], bool) { s_ab = rz / t[0]; }))
            return;
        if (!(v1[0] > 0.0)) {
            leave(it, v2[1], (int)BA_ERR_NOT_SPD);
            return;
        }
        const float alpha = (float)s_ab;
        if (own) {
            const float qe = s_own[threadIdx.x] + __ldcg(q + e);
            qn[e] = 0.f;
            xv = fmaf(alpha, dv, xv);
            rv = fmaf(-alpha, qe, rv);
            s_r[threadIdx.x] = rv;
        }
        __syncthreads();
        v2[0] = v2[1] = 0.0;
        if (own) {
            zv = precond();
            z[e] = zv;
            const double rd = widen(rv);
            v2[0] = rd * widen(zv);
            v2[1] = rd * rd;
        }
        if (!grid_allreduce_w0<2>(v2, red, gen++, bar, &sc->err, limit_cycles, nown,
                                  [&](const double(&t)[2], bool) { s_ab = t[0] / rz; }))
            return;
        ++it;
        if (v2[1] <= tol2 * rr0 || it >= max_iters) {
            leave(it, v2[1], 0);
            return;
        }
        beta = s_ab;
        rz = v2[0];
    }
}

// Device address of the scratch array on the current device; the first call
// on a device looks it up (cudaGetSymbolAddress) with that device current.
cudaError_t scratch_on_current_device(unsigned char **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_pcg_scratch);
        if (e != cudaSuccess) return e;
        g_ptr[dev] = (unsigned char *)p;
    }
    *out = g_ptr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace ba

using namespace ba;

extern "C" ba_status ba_pcg_solve_static(int32_t n, int64_t nnzb, const int32_t *row_ptr, const int32_t *col,
                                         const float *val, const float *b, float *x, double rel_tol,
                                         int32_t max_iters, void *cuda_stream, int32_t *iters_out,
                                         double *rel_resid_out) {
    if (n <= 0 || nnzb < n) return set_error(BA_ERR_INVALID_ARG, "ba_pcg_solve_static: need n > 0 and nnzb >= n");
    if (n > kStaticMaxCams)
        return set_error(BA_ERR_INVALID_ARG, "ba_pcg_solve_static: n exceeds the static scratch limit of 8192 cameras");
    if (!row_ptr || !col || !val || !b || !x) return set_error(BA_ERR_INVALID_ARG, "ba_pcg_solve_static: null pointer");
    if (!(rel_tol > 0) || max_iters < 0) return set_error(BA_ERR_INVALID_ARG, "ba_pcg_solve_static: bad tolerance");
    const int iters_cap = max_iters > 0 ? max_iters : (6 * n > 1000 ? 6 * n : 1000);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    unsigned char *base = nullptr;
    cudaError_t e = scratch_on_current_device(&base);
    if (e != cudaSuccess) return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    StaticScalars *sc = (StaticScalars *)(base + kScalOff);
    double *red = (double *)(base + kRedOff);
    unsigned *bar = (unsigned *)(base + kBarOff);
    float *vec[5];
    for (int k = 0; k < 5; ++k) vec[k] = (float *)(base + kVecOff + k * kVecBytes);
    float *Minv = (float *)(base + kMinvOff);

    // counters and the error flag start at zero on every call
    if ((e = cudaMemsetAsync(bar, 0, AR_SUB * 32 * sizeof(unsigned), st)) != cudaSuccess)
        return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    if ((e = cudaMemsetAsync(sc, 0, sizeof(StaticScalars), st)) != cudaSuccess)
        return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    k_static_minv<<<(n + 3) / 4, 32, 0, st>>>(n, nnzb, row_ptr, col, val, Minv, sc);
    if ((e = cudaGetLastError()) != cudaSuccess) return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    // shared memory for the blocks: what a CTA's share of them needs, with
    // half as much again for uneven rows, at most what a CTA can have
    int per_sm = 0, n_sm = 0;
    if ((e = cudaFuncSetAttribute(k_static_pcg, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStaticSmem)) !=
        cudaSuccess)
        return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    if ((e = occupancy((const void *)k_static_pcg, ST_THREADS, kStaticSmem, &per_sm, &n_sm)) != cudaSuccess)
        return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    int rows = (n + n_sm - 1) / n_sm;
    const int grid = (n + rows - 1) / rows;
    if (per_sm < 1 || 6 * rows > ST_THREADS)
        return set_error(BA_ERR_CUDA, "ba_pcg_solve_static: the device has too few SMs for the cooperative launch");
    const int64_t share = (nnzb + grid - 1) / grid;
    int cap = (int)std::min<int64_t>(share + share / 2 + 32, (int64_t)(kStaticSmem / (BW * 4 + 4)));
    size_t smem = (size_t)cap * (BW * 4 + 4);
    int nn = n, mi = iters_cap;
    double tol2 = rel_tol * rel_tol;
    long long limit = 4000000000LL;  // ~2 s of SM clock per grid wait
    const float *Mi = Minv;
    void *args[] = {&nn, &rows, &row_ptr, &col, &val, &b, &Mi, &x, &vec[0], &vec[1], &vec[2], &vec[3], &vec[4], &sc,
                    &red, &bar, &tol2, &mi, &cap, &limit};
    if ((e = cudaLaunchCooperativeKernel((const void *)k_static_pcg, dim3(grid), dim3(ST_THREADS), args, smem, st)) !=
        cudaSuccess)
        return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    StaticScalars hs{};
    if ((e = cudaMemcpyAsync(&hs, sc, sizeof(hs), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
        return set_error(BA_ERR_CUDA, cudaGetErrorString(e));
    if (hs.err == BA_ERR_TIMEOUT) return set_error(BA_ERR_TIMEOUT, "ba_pcg_solve_static: a grid wait gave up");
    if (iters_out) *iters_out = hs.iters;
    const double rel = hs.rr0 > 0 ? sqrt(hs.rr / hs.rr0) : 0.0;
    if (rel_resid_out) *rel_resid_out = rel;
    if (hs.err == BA_ERR_INVALID_ARG)
        return set_error(BA_ERR_INVALID_ARG,
                         "ba_pcg_solve_static: malformed BSMC pattern (row starts, diagonal block first, ascending "
                         "upper-triangle columns)");
    if (hs.err == BA_ERR_NOT_SPD) return set_error(BA_ERR_NOT_SPD, "ba_pcg_solve_static: matrix is not positive definite");
    if (!(hs.rr <= tol2 * hs.rr0)) return set_error(BA_ERR_NO_CONVERGENCE, "ba_pcg_solve_static: iteration cap reached");
    return BA_OK;
}
