// Least squares on the device: the normal-equation operator u = A^T (A x) and CGLS
// (conjugate gradients on A^T A x = A^T b).  The paper measures SpMV-SpVTM pairs
// because first-order methods for wide or tall problems are built from them
// (Sec. V); here the SpVTM consumes the SpMV's result.  Every vector operation runs
// in the kernels below; the scalars of the iteration stay in device memory, and the
// host reads them only every few iterations to test convergence.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "device_common.cuh"
#include "plan_impl.h"

namespace gbk {
namespace {

#define CG_TRY(expr)                                                              \
    do {                                                                          \
        cudaError_t _e = (expr);                                                  \
        if (_e != cudaSuccess) return set_error(SPMV_ERR_CUDA, cudaGetErrorString(_e)); \
    } while (0)

size_t cg_align(size_t v, size_t a) { return (v + a - 1) / a * a; }
bool cg_aligned16(const void *ptr) { return (reinterpret_cast<uintptr_t>(ptr) & 15u) == 0; }

constexpr int DOT_THREADS = 256;
constexpr int DOT_BLOCKS = 608;  // at most; fixed: the summation order must not depend on the device
// Blocks of a dot product of that length: at least 8 elements a thread.
int dot_blocks(int64_t len) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(DOT_BLOCKS, (len + 8 * DOT_THREADS - 1) / (8 * DOT_THREADS)));
}

struct CgScalars {
    double gamma, gamma0, delta, alpha, beta;
};

template <typename T> __device__ __forceinline__ void two_sum(T &s, T &c, T v) {
    const T t = s + v;
    const T bp = t - s;
    c += (s - (t - bp)) + (v - bp);
    s = t;
}

// a . b and the scalar update of the iteration.  Block g takes elements g DOT_THREADS + t, then every
// G DOT_THREADS-th, in order; compensated sums; the block reduces its threads in a fixed tree
// order; the block that finishes last adds the block sums in order (thread t: t, t + 32, ..; then
// a butterfly).  what = 0: gamma0 = gamma = sum (start); 1: delta = sum, alpha = gamma / delta;
// 2: beta = sum / gamma, gamma = sum.  (As two kernels, the first over 608 blocks whatever the
// length, 11 + 4 us for 400,000 FP64 elements and 6 + 4 for 4,000, and a launch more.)
template <typename T>
__global__ void __launch_bounds__(DOT_THREADS) dot_kernel(const T *a, const T *b, int64_t len, double *part, int what,
                                                          CgScalars *sc, int *done) {
    __shared__ T sh_s[DOT_THREADS], sh_c[DOT_THREADS];
    __shared__ bool last;
    grid_release();
    grid_wait();
    T s = T(0), c = T(0);
    const int64_t stride = (int64_t)gridDim.x * DOT_THREADS;
    for (int64_t i = (int64_t)blockIdx.x * DOT_THREADS + threadIdx.x; i < len; i += 4 * stride) {
        T u[4], v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const bool in = i + e * stride < len;
            u[e] = in ? a[i + e * stride] : T(0);
            v[e] = in ? b[i + e * stride] : T(0);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (i + e * stride < len) two_sum(s, c, u[e] * v[e]);
    }
    sh_s[threadIdx.x] = s;
    sh_c[threadIdx.x] = c;
    __syncthreads();
    for (int w = DOT_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            T ss = sh_s[threadIdx.x], cc = sh_c[threadIdx.x];
            two_sum(ss, cc, sh_s[threadIdx.x + w]);
            cc += sh_c[threadIdx.x + w];
            sh_s[threadIdx.x] = ss;
            sh_c[threadIdx.x] = cc;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[blockIdx.x] = (double)sh_s[0] + (double)sh_c[0];
        __threadfence();
        last = atomicAdd(done, 1) == (int)gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    double t = 0.0;
    for (int q = threadIdx.x; q < (int)gridDim.x; q += 32) t += __ldcg(part + q);
    for (int d = 16; d > 0; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
    if (threadIdx.x == 0) {
        *done = 0;  // for the next dot product
        if (what == 0) {
            sc->gamma = sc->gamma0 = t;
        } else if (what == 1) {
            sc->delta = t;
            sc->alpha = t > 0.0 ? sc->gamma / t : 0.0;
        } else {
            sc->beta = sc->gamma > 0.0 ? t / sc->gamma : 0.0;
            sc->gamma = t;
        }
    }
}

// x += alpha p (n entries), r -= alpha q (m entries)
template <typename T>
__global__ void xr_update_kernel(T *x, const T *p, int64_t n, T *r, const T *q, int64_t m, const CgScalars *sc) {
    grid_release();
    grid_wait();
    const T alpha = (T)sc->alpha;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t len = n > m ? n : m;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += stride) {
        // (the four loads first: the pointers may alias as far as the compiler knows)
        const bool in_x = i < n, in_r = i < m;
        const T xi = in_x ? x[i] : T(0), pi = in_x ? p[i] : T(0), ri = in_r ? r[i] : T(0), qi = in_r ? q[i] : T(0);
        if (in_x) x[i] = xi + alpha * pi;
        if (in_r) r[i] = ri - alpha * qi;
    }
}

// p = s + beta p (beta = 0 copies)
template <typename T>
__global__ void p_update_kernel(T *p, const T *s, int64_t n, const CgScalars *sc, int first) {
    grid_release();
    grid_wait();
    const T beta = first ? T(0) : (T)sc->beta;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        p[i] = first ? s[i] : s[i] + beta * p[i];
}

// r = b - r
template <typename T>
__global__ void residual_kernel(const T *__restrict__ b, T *__restrict__ r, int64_t m) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) r[i] = b[i] - r[i];
}

template <typename T> struct Cgls {
    spmv_plan_s *p;
    cudaStream_t s;
    int grid;
    T *r = nullptr, *sv = nullptr, *pv = nullptr, *q = nullptr;
    double *part = nullptr;
    CgScalars *sc = nullptr;

    // blocks of an element-wise kernel of that length: all at once, up to the grid
    int blocks_for(int64_t len) const { return (int)std::max<int64_t>(1, std::min<int64_t>(grid, (len + 255) / 256)); }

    cudaError_t dot(const T *a, const T *b, int64_t len, int what) {
        return launch_overlapped(dot_kernel<T>, dim3(dot_blocks(len)), dim3(DOT_THREADS), 0, s, a, b, len, part, what, sc,
                                 reinterpret_cast<int *>(sc + 1));
    }

    spmv_status run(const T *bvec, T *x, int max_iters, double tol, int32_t *iters_done, double *rel) {
        const int64_t m = p->m, n = p->n;
        const T *cin = x;
        void *cout = r;
        spmv_status st = run_op(p, SPMV_OP_AX, 1, reinterpret_cast<const void *const *>(&cin), &cout, s);
        if (st != SPMV_OK) return st;
        residual_kernel<T><<<grid, 256, 0, s>>>(bvec, r, m);
        const T *rin = r;
        void *sout = sv;
        if ((st = run_op(p, SPMV_OP_VTA, 1, reinterpret_cast<const void *const *>(&rin), &sout, s)) != SPMV_OK)
            return st;
        CG_TRY(dot(sv, sv, n, 0));
        CG_TRY(launch_overlapped(p_update_kernel<T>, dim3(blocks_for(n)), dim3(256), 0, s, pv, sv, n, sc, 1));
        CgScalars h{};
        int it = 0;
        while (it < max_iters) {
            const T *pin = pv;
            void *qout = q;
            if ((st = run_op(p, SPMV_OP_AX, 1, reinterpret_cast<const void *const *>(&pin), &qout, s)) != SPMV_OK)
                return st;
            CG_TRY(dot(q, q, m, 1));
            CG_TRY(launch_overlapped(xr_update_kernel<T>, dim3(blocks_for(std::max(n, m))), dim3(256), 0, s, x, pv, n, r, q, m, sc));
            if ((st = run_op(p, SPMV_OP_VTA, 1, reinterpret_cast<const void *const *>(&rin), &sout, s)) != SPMV_OK)
                return st;
            CG_TRY(dot(sv, sv, n, 2));
            CG_TRY(launch_overlapped(p_update_kernel<T>, dim3(blocks_for(n)), dim3(256), 0, s, pv, sv, n, sc, 0));
            ++it;
            if (it % 8 == 0 || it == max_iters) {  // convergence test on the host
                CG_TRY(cudaMemcpyAsync(&h, sc, sizeof(h), cudaMemcpyDeviceToHost, s));
                CG_TRY(cudaStreamSynchronize(s));
                if (!(h.gamma0 > 0.0) || std::sqrt(h.gamma / h.gamma0) <= tol) break;
            }
        }
        CG_TRY(cudaMemcpyAsync(&h, sc, sizeof(h), cudaMemcpyDeviceToHost, s));
        CG_TRY(cudaStreamSynchronize(s));
        if (iters_done) *iters_done = it;
        if (rel) *rel = h.gamma0 > 0.0 ? std::sqrt(h.gamma / h.gamma0) : 0.0;
        return SPMV_OK;
    }
};

template <typename T>
spmv_status cgls_typed(spmv_plan_s *p, const void *b, void *x, int max_iters, double tol, cudaStream_t s,
                       int32_t *iters_done, double *rel) {
    Cgls<T> c{p, s, 0};
    int sms = 0;
    CG_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device));
    c.grid = std::max(1, sms * 4);
    const size_t m = (size_t)std::max<int64_t>(p->m, 1), n = (size_t)std::max<int64_t>(p->n, 1);
    void *block = nullptr;
    const size_t off_s = cg_align(m * sizeof(T), 256), off_p = off_s + cg_align(n * sizeof(T), 256);
    const size_t off_q = off_p + cg_align(n * sizeof(T), 256), off_part = off_q + cg_align(m * sizeof(T), 256);
    const size_t off_sc = off_part + cg_align(DOT_BLOCKS * sizeof(double), 256);
    const size_t total = off_sc + sizeof(CgScalars) + sizeof(int);  // (the dot products' block counter behind the scalars)
    CG_TRY(dev_alloc(&block, total));
    char *mem = static_cast<char *>(block);
    c.r = reinterpret_cast<T *>(mem);
    c.sv = reinterpret_cast<T *>(mem + off_s);
    c.pv = reinterpret_cast<T *>(mem + off_p);
    c.q = reinterpret_cast<T *>(mem + off_q);
    c.part = reinterpret_cast<double *>(mem + off_part);
    c.sc = reinterpret_cast<CgScalars *>(mem + off_sc);
    cudaError_t e = cudaMemsetAsync(c.sc, 0, sizeof(CgScalars) + sizeof(int), s);
    spmv_status st = e == cudaSuccess ? c.run(static_cast<const T *>(b), static_cast<T *>(x), max_iters, tol, iters_done,
                                               rel)
                                      : set_error(SPMV_ERR_CUDA, cudaGetErrorString(e));
    cudaStreamSynchronize(s);
    dev_free(block, p->device);
    return st;
}

}  // namespace
}  // namespace gbk

using namespace gbk;

extern "C" {

spmv_status spmv_normal(spmv_plan_t p, const void *x, void *u, void *y, void *stream) {
    if (!p) return set_error(SPMV_ERR_INVALID_ARG, "null plan");
    if (!x || !u) return set_error(SPMV_ERR_INVALID_ARG, "null vector");
    if (!cg_aligned16(x) || !cg_aligned16(u) || !cg_aligned16(y))
        return set_error(SPMV_ERR_INVALID_ARG, "vectors must be 16-byte aligned device memory");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    void *yb = y;
    if (!yb) {
        std::lock_guard<std::mutex> lk(p->host_mu);
        if (!p->ynorm) CG_TRY(dev_malloc(&p->ynorm, (size_t)std::max<int64_t>(p->m, 1) * p->sx + 16));
        yb = p->ynorm;
    }
    const void *xin = x;
    spmv_status st = run_op(p, SPMV_OP_AX, 1, &xin, &yb, s);
    if (st != SPMV_OK) return st;
    const void *yin = yb;
    return run_op(p, SPMV_OP_VTA, 1, &yin, &u, s);
}

spmv_status spmv_cgls(spmv_plan_t p, const void *b, void *x, int32_t max_iters, double tol, void *stream,
                      int32_t *iters_done, double *rel_grad) {
    if (!p) return set_error(SPMV_ERR_INVALID_ARG, "null plan");
    if (!b || !x) return set_error(SPMV_ERR_INVALID_ARG, "null vector");
    if (!cg_aligned16(b) || !cg_aligned16(x))
        return set_error(SPMV_ERR_INVALID_ARG, "vectors must be 16-byte aligned device memory");
    if (max_iters < 0 || !(tol >= 0.0)) return set_error(SPMV_ERR_INVALID_ARG, "max_iters >= 0 and tol >= 0 required");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (p->vec_t == SPMV_F64) return cgls_typed<double>(p, b, x, max_iters, tol, s, iters_done, rel_grad);
    return cgls_typed<float>(p, b, x, max_iters, tol, s, iters_done, rel_grad);
}

}  // extern "C"
