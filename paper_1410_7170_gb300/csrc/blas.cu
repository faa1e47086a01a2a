// BLAS-1 kernels on flat arrays: deterministic reductions (norms, complex dots,
// multi-dots for Gram-Schmidt), axpy variants and precision conversion. All are
// HBM-streaming; reductions accumulate in FP64 in a fixed order.
#include <algorithm>

#include "internal.h"
#include "reduce.cuh"

namespace ovl {

namespace {

struct Nothing {};
struct StoreFin1 {
    double *res;
    __device__ Nothing before() const { return {}; }
    __device__ void operator()(const double *s, Nothing) const { res[0] = s[0]; }
};
struct StoreFin2 {
    double *res;
    __device__ Nothing before() const { return {}; }
    __device__ void operator()(const double *s, Nothing) const { res[0] = s[0]; res[1] = s[1]; }
};

// Per-thread partial sums are kept in the vector's own precision T (a grid-stride
// thread sees only a few elements), and so are the warp sums; warps, blocks and the grid
// are summed in FP64.
template <typename T>
__global__ void k_norm2(const T *__restrict__ x, long n, RedScratch rs, double *res) {
    T a = 0;
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x)
        a += x[k] * x[k];
    T v[1] = {a};
    grid_reduce<1>(v, rs, StoreFin1{res});
}

// <x, y> = sum conj(x) y over complex numbers stored as (re, im) pairs
template <typename T>
__global__ void k_cdot(const T *__restrict__ x, const T *__restrict__ y, long nc, RedScratch rs, double *res) {
    T a = 0, b = 0;
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < nc; k += (long)gridDim.x * blockDim.x) {
        const T xr = x[2 * k], xi = x[2 * k + 1];
        const T yr = y[2 * k], yi = y[2 * k + 1];
        a += xr * yr + xi * yi;
        b += xr * yi - xi * yr;
    }
    T v[2] = {a, b};
    grid_reduce<2>(v, rs, StoreFin2{res});
}

__global__ void k_axpby(double a, const double *__restrict__ x, double b, double *__restrict__ y, long n) {
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x)
        y[k] = a * x[k] + b * y[k];
}
__global__ void k_axpby_f(float a, const float *__restrict__ x, float b, float *__restrict__ y, long n) {
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x)
        y[k] = a * x[k] + b * y[k];
}
__global__ void k_caxpy(double ar, double ai, const double *__restrict__ x, double *__restrict__ y, long nc) {
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < nc; k += (long)gridDim.x * blockDim.x) {
        const double xr = x[2 * k], xi = x[2 * k + 1];
        y[2 * k] += ar * xr - ai * xi;
        y[2 * k + 1] += ar * xi + ai * xr;
    }
}

// Multi-dot: blockIdx.y = vector index; partials[k][blockIdx.x] (complex).
template <typename T>
__global__ void k_multidot_part(const T *__restrict__ base, long stride, int m, const T *__restrict__ w, long nc,
                                double *partials) {
    const T *v = base + (long)blockIdx.y * stride;
    T a = 0, b = 0;
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < nc; k += (long)gridDim.x * blockDim.x) {
        const T vr = v[2 * k], vi = v[2 * k + 1];
        const T wr = w[2 * k], wi = w[2 * k + 1];
        a += vr * wr + vi * wi;
        b += vr * wi - vi * wr;
    }
    const T t[2] = {a, b};
    double s[2];
    block_sum<2>(t, s);
    if (threadIdx.x == 0) {
        partials[((long)blockIdx.y * gridDim.x + blockIdx.x) * 2] = s[0];
        partials[((long)blockIdx.y * gridDim.x + blockIdx.x) * 2 + 1] = s[1];
    }
}
__global__ void k_multidot_sum(const double *partials, int nb, double *out) {
    double s[2] = {0.0, 0.0};
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        s[0] += partials[((long)blockIdx.x * nb + b) * 2];
        s[1] += partials[((long)blockIdx.x * nb + b) * 2 + 1];
    }
    block_sum<2>(s);
    if (threadIdx.x == 0) {
        out[2 * blockIdx.x] = s[0];
        out[2 * blockIdx.x + 1] = s[1];
    }
}

template <typename T>
__global__ void k_multiaxpy(const T *__restrict__ base, long stride, int m, const double *__restrict__ c,
                            T *__restrict__ w, long nc) {
    __shared__ T cs[2 * 128];   // coefficients in the vectors' precision
    for (int k = threadIdx.x; k < 2 * m; k += blockDim.x) cs[k] = (T)c[k];
    __syncthreads();
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < nc; k += (long)gridDim.x * blockDim.x) {
        T ar = w[2 * k], ai = w[2 * k + 1];
        for (int j = 0; j < m; j++) {
            const T *v = base + (long)j * stride;
            const T vr = v[2 * k], vi = v[2 * k + 1];
            ar += cs[2 * j] * vr - cs[2 * j + 1] * vi;
            ai += cs[2 * j] * vi + cs[2 * j + 1] * vr;
        }
        w[2 * k] = ar;
        w[2 * k + 1] = ai;
    }
}

// ---- Gram-Schmidt without the host (gs_dots, gs_subtract, gs_combine)
// 16-byte words: one complex double or two complex floats.
template <typename T> struct GsWord;
template <> struct GsWord<double> {
    using W = double2;
    // a thread's sum over its words, group by group (dot adds to what open returns), and what the block
    // adds up
    using Part = double;
    struct Sum {
        double s = 0.0;
        __device__ double open() const { return s; }
        __device__ void close(double x) { s = x; }
        __device__ Part value() const { return s; }
    };
    __device__ static void dot(W v, W w, double &a, double &b) {
        a += v.x * w.x + v.y * w.y;
        b += v.x * w.y - v.y * w.x;
    }
    __device__ static void axpy(double cr, double ci, W v, W &w) {
        w.x += cr * v.x - ci * v.y;
        w.y += cr * v.y + ci * v.x;
    }
    __device__ static W scaled(double s, W w) { return make_double2(s * w.x, s * w.y); }
    __device__ static W zero() { return make_double2(0.0, 0.0); }
};
template <> struct GsWord<float> {
    using W = float4;
    using Part = fsum;
    struct Sum {
        fsum s;
        __device__ float open() const { return 0.f; }
        __device__ void close(float x) { s.add(x); }
        __device__ Part value() const { return s; }
    };
    __device__ static void dot(W v, W w, float &a, float &b) {
        a += v.x * w.x + v.y * w.y + v.z * w.z + v.w * w.w;
        b += v.x * w.y - v.y * w.x + v.z * w.w - v.w * w.z;
    }
    __device__ static void axpy(float cr, float ci, W v, W &w) {
        w.x += cr * v.x - ci * v.y;
        w.y += cr * v.y + ci * v.x;
        w.z += cr * v.z - ci * v.w;
        w.w += cr * v.w + ci * v.z;
    }
    __device__ static W scaled(float s, W w) { return make_float4(s * w.x, s * w.y, s * w.z, s * w.w); }
    __device__ static W zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
};
constexpr int kGsMax = 128;   // basis vectors

// Grid (blocks, m + 1, right-hand sides); vector m is w itself. The last block of a right-hand side
// sums the partials in block order and writes its record.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_gs_dots(const T *__restrict__ base, long stride, int m,
                                                    const T *__restrict__ w, long n, RowList rows, double *out,
                                                    long ostride, bool one_pass, const double *prev, double *partials,
                                                    unsigned *counters) {
    using G = GsWord<T>;
    using W = typename G::W;
    const int z = blockIdx.z, i = blockIdx.y;
    if (prev && prev[z * ostride + 2 * m + 4] != 0.0) return;   // uniform over the right-hand side
    const long off = (long)rows.row[z] * n, nw = n * (long)sizeof(T) / (long)sizeof(W);
    const W *x = reinterpret_cast<const W *>(w + off);
    const W *v = i < m ? reinterpret_cast<const W *>(base + (long)i * stride + off) : x;
    // Four words of each vector in flight per thread: the grid is small (gs_grid). In FP32 a plain sum
    // never runs over more than four words (16 products); the groups are added with their errors (fsum),
    // and so are the threads. The kernel has 2 blocks per SM over all vectors, so that with one FP32 sum
    // per thread the relative error of ||w||^2 at 32^4 was 1e-8 at 32 vectors and 4e-8 at 75 (chains of
    // 5800 products and more): 1e-10 now, at the same time (DRAM and latency bound).
    typename G::Sum sa, sb;
    const long step = (long)gridDim.x * blockDim.x;
    long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; k + 3 * step < nw; k += 4 * step) {
        W p[4], q[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            p[u] = v[k + u * step];
            q[u] = x[k + u * step];
        }
        T a = sa.open(), b = sb.open();
#pragma unroll
        for (int u = 0; u < 4; u++) G::dot(p[u], q[u], a, b);
        sa.close(a);
        sb.close(b);
    }
    for (; k < nw; k += step) {
        T a = sa.open(), b = sb.open();
        G::dot(v[k], x[k], a, b);
        sa.close(a);
        sb.close(b);
    }
    const typename G::Part t[2] = {sa.value(), sb.value()};
    double s[2];
    block_sum<2>(t, s);
    __shared__ int is_last;
    __shared__ double h[2 * kGsMax + 2];
    const int gx = gridDim.x;
    double *part = partials + (long)z * gridDim.y * gx * 2;
    if (threadIdx.x == 0) {
        part[((long)i * gx + blockIdx.x) * 2] = s[0];
        part[((long)i * gx + blockIdx.x) * 2 + 1] = s[1];
        is_last = arrive(counters + z) == (unsigned)(gridDim.y * gx - 1);
    }
    __syncthreads();
    if (!is_last) return;
    double *o = out + z * ostride;
    const int lane = threadIdx.x & 31;
    for (int q = threadIdx.x >> 5; q <= m; q += kBlock / 32) {
        double d[2] = {0.0, 0.0};
        for (int k = lane; k < gx; k += 32) {
            d[0] += __ldcg(part + ((long)q * gx + k) * 2);
            d[1] += __ldcg(part + ((long)q * gx + k) * 2 + 1);
        }
        warp_sum<2>(d);
        if (lane == 0) {
            o[2 * q] = h[2 * q] = d[0];
            o[2 * q + 1] = h[2 * q + 1] = q < m ? d[1] : 0.0;
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        double q[1] = {0.0};
        for (int k = lane; k < 2 * m; k += 32) q[0] += h[k] * h[k];
        warp_sum<1>(q);
        if (lane == 0) {
            const double ww = h[2 * m], left = ww - q[0];
            const double hn = left <= 0.0 ? 0.0 : sqrt(left);   // NaN stays NaN
            o[2 * m + 2] = hn;
            o[2 * m + 3] = hn > 0.0 ? 1.0 / hn : 0.0;
            o[2 * m + 4] = one_pass && left > 0.1 * ww ? 1.0 : 0.0;
            counters[z] = 0u;
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_gs_subtract(const T *__restrict__ base, long stride, int m,
                                                        const double *__restrict__ h, long ostride,
                                                        const double *__restrict__ prev, T *w, T *next, long n,
                                                        RowList rows) {
    using G = GsWord<T>;
    using W = typename G::W;
    __shared__ T cs[2 * kGsMax];
    const int z = blockIdx.y;
    const double *hz = h + z * ostride;
    const bool one = hz[2 * m + 4] != 0.0;
    if (prev && prev[z * ostride + 2 * m + 4] != 0.0) return;
    for (int k = threadIdx.x; k < 2 * m; k += blockDim.x) cs[k] = (T)(-hz[k]);
    __syncthreads();
    const bool fin = prev || one;   // the last subtraction: normalise into next
    const T sc = fin ? (T)hz[2 * m + 3] : T(1);
    const long off = (long)rows.row[z] * n, nw = n * (long)sizeof(T) / (long)sizeof(W);
    const W *v = reinterpret_cast<const W *>(base + off), *x = reinterpret_cast<const W *>(w + off);
    W *o = reinterpret_cast<W *>((fin ? next : w) + off);
    const long sw = stride * (long)sizeof(T) / (long)sizeof(W);
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < nw; k += (long)gridDim.x * blockDim.x) {
        W a = x[k];
#pragma unroll 4
        for (int j = 0; j < m; j++) G::axpy(cs[2 * j], cs[2 * j + 1], v[j * sw + k], a);
        o[k] = fin ? G::scaled(sc, a) : a;
    }
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_gs_combine(const T *__restrict__ base, long stride, int m,
                                                       const double *__restrict__ c, T *x, bool add, long n,
                                                       RowList rows, RowColumns cols) {
    using G = GsWord<T>;
    using W = typename G::W;
    __shared__ T cs[2 * kGsMax];
    const int z = blockIdx.y, mz = cols.n[z];
    for (int k = threadIdx.x; k < 2 * mz; k += blockDim.x) cs[k] = (T)c[2 * m * z + k];
    __syncthreads();
    const long off = (long)rows.row[z] * n, nw = n * (long)sizeof(T) / (long)sizeof(W);
    const W *v = reinterpret_cast<const W *>(base + off);
    W *o = reinterpret_cast<W *>(x + off);
    const long sw = stride * (long)sizeof(T) / (long)sizeof(W);
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < nw; k += (long)gridDim.x * blockDim.x) {
        W a = add ? o[k] : G::zero();
#pragma unroll 4
        for (int j = 0; j < mz; j++) G::axpy(cs[2 * j], cs[2 * j + 1], v[j * sw + k], a);
        o[k] = a;
    }
}

__global__ void k_d2f(const double *__restrict__ x, float *__restrict__ y, long n) {
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x)
        y[k] = (float)x[k];
}
__global__ void k_f2d(const float *__restrict__ x, double *__restrict__ y, long n) {
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x)
        y[k] = (double)x[k];
}

inline int stream_grid(long n) {
    long b = (n + kBlock - 1) / kBlock;
    const long cap = 152L * 16;   // enough resident blocks to fill 152 SMs several times
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

cudaError_t dev_norm2(const double *x, long n, double *res, RedScratch rs, cudaStream_t st) {
    k_norm2<double><<<red_grid(n), kBlock, 0, st>>>(x, n, rs, res);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t dev_norm2_f(const float *x, long n, double *res, RedScratch rs, cudaStream_t st) {
    k_norm2<float><<<red_grid(n), kBlock, 0, st>>>(x, n, rs, res);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t dev_cdot(const double *x, const double *y, long n, double *res, RedScratch rs, cudaStream_t st) {
    k_cdot<double><<<red_grid(n / 2), kBlock, 0, st>>>(x, y, n / 2, rs, res);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t dev_cdot_f(const float *x, const float *y, long n, double *res, RedScratch rs, cudaStream_t st) {
    k_cdot<float><<<red_grid(n / 2), kBlock, 0, st>>>(x, y, n / 2, rs, res);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t dev_axpby(double a, const double *x, double b, double *y, long n, cudaStream_t st) {
    k_axpby<<<stream_grid(n), kBlock, 0, st>>>(a, x, b, y, n);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t dev_axpby_f(float a, const float *x, float b, float *y, long n, cudaStream_t st) {
    k_axpby_f<<<stream_grid(n), kBlock, 0, st>>>(a, x, b, y, n);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t dev_caxpy(double ar, double ai, const double *x, double *y, long n, cudaStream_t st) {
    k_caxpy<<<stream_grid(n / 2), kBlock, 0, st>>>(ar, ai, x, y, n / 2);
    count_launches(1);
    return cudaGetLastError();
}

constexpr int kMdBlocks = 256;   // partial blocks per vector of a multi-dot

cudaError_t dev_multidot(const double *base, long stride, int m, const double *w, long n, double *out,
                         double *partials, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    int gx = (int)((n / 2 + kBlock - 1) / kBlock);
    if (gx > kMdBlocks) gx = kMdBlocks;
    if (gx < 1) gx = 1;
    k_multidot_part<double><<<dim3(gx, m), kBlock, 0, st>>>(base, stride, m, w, n / 2, partials);
    k_multidot_sum<<<m, kBlock, 0, st>>>(partials, gx, out);
    count_launches(2);
    return cudaGetLastError();
}
cudaError_t dev_multidot_f(const float *base, long stride, int m, const float *w, long n, double *out,
                           double *partials, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    int gx = (int)((n / 2 + kBlock - 1) / kBlock);
    if (gx > kMdBlocks) gx = kMdBlocks;
    if (gx < 1) gx = 1;
    k_multidot_part<float><<<dim3(gx, m), kBlock, 0, st>>>(base, stride, m, w, n / 2, partials);
    k_multidot_sum<<<m, kBlock, 0, st>>>(partials, gx, out);
    count_launches(2);
    return cudaGetLastError();
}
cudaError_t dev_multiaxpy(const double *base, long stride, int m, const double *c, double *w, long n,
                          cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    k_multiaxpy<double><<<stream_grid(n / 2), kBlock, 0, st>>>(base, stride, m, c, w, n / 2);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t dev_multiaxpy_f(const float *base, long stride, int m, const double *c, float *w, long n,
                            cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    k_multiaxpy<float><<<stream_grid(n / 2), kBlock, 0, st>>>(base, stride, m, c, w, n / 2);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t dev_d2f(const double *x, float *y, long n, cudaStream_t st) {
    k_d2f<<<stream_grid(n), kBlock, 0, st>>>(x, y, n);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t dev_f2d(const float *x, double *y, long n, cudaStream_t st) {
    k_f2d<<<stream_grid(n), kBlock, 0, st>>>(x, y, n);
    count_launches(1);
    return cudaGetLastError();
}

// Blocks per vector: about per_sm per SM over all vectors and right-hand sides, none without words.
// The dot products take few (each block ends with a fence and an atomic: at 16^4 17 us with 1216
// blocks), and no more than the partial sums have room for.
constexpr long kGsPartials = 128 * 256;   // complex partial sums
static int gs_grid(long words, long vectors, int per_sm) {
    const long b = (words + kBlock - 1) / kBlock, cap = std::max(4L, (long)per_sm * device_sm_count() / vectors);
    return (int)std::max(1L, std::min({b, cap, kGsPartials / vectors}));
}
template <typename T>
cudaError_t gs_dots(const T *base, long stride, int m, const T *w, long n, const RowList &rows, double *out,
                    long ostride, bool one_pass, const double *prev, double *partials, unsigned *counters,
                    cudaStream_t st) {
    const int gx = gs_grid(n * (long)sizeof(T) / 16, (long)(m + 1) * rows.n, 2);
    k_gs_dots<T><<<dim3(gx, m + 1, rows.n), kBlock, 0, st>>>(base, stride, m, w, n, rows, out, ostride, one_pass, prev,
                                                             partials, counters);
    count_launches(1);
    return cudaGetLastError();
}
template <typename T>
cudaError_t gs_subtract(const T *base, long stride, int m, const double *h, long ostride, const double *prev, T *w,
                        T *next, long n, const RowList &rows, cudaStream_t st) {
    k_gs_subtract<T><<<dim3(gs_grid(n * (long)sizeof(T) / 16, rows.n, 8), rows.n), kBlock, 0, st>>>(base, stride, m, h, ostride,
                                                                                              prev, w, next, n, rows);
    count_launches(1);
    return cudaGetLastError();
}
template <typename T>
cudaError_t gs_combine(const T *base, long stride, int m, const double *c, T *x, bool add, long n, const RowList &rows,
                       const RowColumns &cols, cudaStream_t st) {
    k_gs_combine<T><<<dim3(gs_grid(n * (long)sizeof(T) / 16, rows.n, 8), rows.n), kBlock, 0, st>>>(base, stride, m, c, x, add,
                                                                                             n, rows, cols);
    count_launches(1);
    return cudaGetLastError();
}
#define OVL_GS(T)                                                                                                     \
    template cudaError_t gs_dots<T>(const T *, long, int, const T *, long, const RowList &, double *, long, bool,      \
                                    const double *, double *, unsigned *, cudaStream_t);                              \
    template cudaError_t gs_subtract<T>(const T *, long, int, const double *, long, const double *, T *, T *, long,    \
                                        const RowList &, cudaStream_t);                                               \
    template cudaError_t gs_combine<T>(const T *, long, int, const double *, T *, bool, long, const RowList &,         \
                                       const RowColumns &, cudaStream_t);
OVL_GS(float)
OVL_GS(double)
#undef OVL_GS

}  // namespace ovl
