// Layout conversion and the Wilson-Dirac stencil kernels (Eq. Wilson-Dirac).
#include "convert.h"
#include "hops.cuh"
#include "internal.h"
#include "reduce.cuh"
#include "wilson_site.cuh"

#include <algorithm>
#include <atomic>

namespace ovl {

static std::atomic<long> g_launches{0};
static thread_local bool g_counting = true;
void count_launches(long n) {
    if (g_counting) g_launches.fetch_add(n, std::memory_order_relaxed);
}
long launches_total() { return g_launches.load(std::memory_order_relaxed); }
void set_launch_counting(bool on) { g_counting = on; }

int device_sm_count() {
    static int cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return 152;
    }
    if (!cache[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 152;
        }
        cache[dev] = n;
    }
    return cache[dev];
}

// ------------------------------------------------------------------ gauge upload
// One thread per (site, mu): SU(3) check, then -1/2 U in both precisions (FP32: rows 0 and 1).
__global__ void k_pack_gauge(Geom g, const double2 *__restrict__ lex, double2 *u64, float4 *u32, int *bad,
                             double tol) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)g.V * 4) return;
    const int s = (int)(t >> 2), mu = (int)(t & 3);
    cpx<double> u[3][3];
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
            double2 v = lex[(size_t)t * 9 + a * 3 + b];
            u[a][b] = cpx<double>{v.x, v.y};
        }
    // unitarity: max |(U U^H - I)_ab|; det U = 1
    double err = 0.0;
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
            cpx<double> d = cmul_conj(u[b][0], u[a][0]) + cmul_conj(u[b][1], u[a][1]) + cmul_conj(u[b][2], u[a][2]);
            if (a == b) d.re -= 1.0;
            err = fmax(err, sqrt(norm2(d)));
        }
    cpx<double> det = u[0][0] * (u[1][1] * u[2][2] - u[1][2] * u[2][1]) -
                      u[0][1] * (u[1][0] * u[2][2] - u[1][2] * u[2][0]) +
                      u[0][2] * (u[1][0] * u[2][1] - u[1][1] * u[2][0]);
    det.re -= 1.0;
    err = fmax(err, sqrt(norm2(det)));
    if (!(err <= tol)) atomicExch(bad, 1);   // also catches NaN
    int x[4];
    int r = s;
    x[3] = r % g.L[3]; r /= g.L[3];
    x[2] = r % g.L[2]; r /= g.L[2];
    x[1] = r % g.L[1]; x[0] = r / g.L[1];
    const int p = (x[0] + x[1] + x[2] + x[3]) & 1, i = s >> 1;
    // stored as kLinkScale U (the hopping term's -1/2 folded in)
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) u[a][b] = kLinkScale * u[a][b];
    double2 *d64 = u64 + ((size_t)(p * 4 + mu) * kLink64Words) * g.Vh + i;
#pragma unroll
    for (int c = 0; c < 9; c++) d64[(size_t)c * g.Vh] = make_double2(u[c / 3][c % 3].re, u[c / 3][c % 3].im);
    float4 *d32 = u32 + ((size_t)(p * 4 + mu) * 3) * g.Vh + i;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const cpx<double> e0 = u[(2 * c) / 3][(2 * c) % 3], e1 = u[(2 * c + 1) / 3][(2 * c + 1) % 3];
        d32[(size_t)c * g.Vh] = make_float4((float)e0.re, (float)e0.im, (float)e1.re, (float)e1.im);
    }
}

cudaError_t pack_gauge(const Geom &g, const double *lex, double2 *u64, float4 *u32, int *bad, double tol,
                       cudaStream_t st) {
    k_pack_gauge<<<plain_grid((long)g.V * 4), kBlock, 0, st>>>(g, (const double2 *)lex, u64, u32, bad, tol);
    count_launches(1);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ spinor layout
// Boundary vectors (lexicographic [s][12] complex doubles) <-> even-odd spinors of the
// library's formats, one pass over memory each way.
//
// Bound: HBM. A site of the boundary layout is 192 contiguous bytes, a site of the internal
// layouts 6 or 12 words Vh words apart, so a thread per site would have one of the two sides
// scattered. A block of 256 threads instead moves 64 consecutive sites through shared memory:
// both sides are read and written in whole 512-byte rows. Sites 2i and 2i + 1 share the
// checkerboard index i, so they are kept 32 rows apart in shared memory and a row is 13 words
// long: the eight 16-byte reads of a quarter warp (consecutive i, one component) then fall on
// different banks. The format conversion (by integer instructions, convert.h) and the test for NaN
// and Inf ride along. Measured at 64 x 32^3, FP32 format (603 MB each way): 308 us in and 397 us out
// as separate kernels with one thread per site (pack 120, test 102, d2f 85; f2d 87, unpack 310),
// 181 and 121 us in one pass with conversions on the FP64 unit, 104 and 114 us (5.8 and 5.3 TB/s)
// with integer ones.
constexpr int kIoTile = 64, kIoRow = 13;

// Word j of a site's internal format from / to its 12 complex numbers.
template <typename ST> struct IoWord;
template <> struct IoWord<double2> {
    static constexpr int N = 12;
    __device__ static double2 get(const double2 *v, int j) { return v[j]; }
    __device__ static void put(double2 *v, int j, double2 w) { v[j] = w; }
};
template <> struct IoWord<float4> {
    static constexpr int N = 6;
    __device__ static float4 get(const double2 *v, int j) {
        const double2 a = v[2 * j], b = v[2 * j + 1];
        return make_float4(d2f(a.x), d2f(a.y), d2f(b.x), d2f(b.y));
    }
    __device__ static void put(double2 *v, int j, float4 w) {
        v[2 * j] = make_double2(f2d(w.x), f2d(w.y));
        v[2 * j + 1] = make_double2(f2d(w.z), f2d(w.w));
    }
};
template <> struct IoWord<ffw> {
    static constexpr int N = 12;
    // word j: real (j even) or imaginary part of one colour of two spins; its two complex numbers
    __device__ static int first(int j) { return j < 6 ? j >> 1 : 3 + (j >> 1); }
    __device__ static ffw get(const double2 *v, int j) {
        const double *x = reinterpret_cast<const double *>(v + first(j)) + (j & 1);
        ffw w;
        d2ff(x[0], w.h0, w.l0);
        d2ff(x[6], w.h1, w.l1);
        return w;
    }
    __device__ static void put(double2 *v, int j, ffw w) {
        double *x = reinterpret_cast<double *>(v + first(j)) + (j & 1);
        x[0] = ff2d(w.h0, w.l0);
        x[6] = ff2d(w.h1, w.l1);
    }
};

__device__ __forceinline__ int io_row(int s) { return ((s >> 1) + (kIoTile / 2) * (s & 1)) * kIoRow; }
// parity of x0 + x1 + x2 at checkerboard index i: site (p, i) is lexicographic site
// 2 i + ((p + this) & 1)
__device__ __forceinline__ int io_row_parity(const Geom &g, int i) {
    int x3h, x2, x1;
    const int r = div_mod(i, g.Lh3, g.inv[2], x3h), q = div_mod(r, g.L[2], g.inv[1], x2);
    return (div_mod(q, g.L[1], g.inv[0], x1) + x1 + x2) & 1;
}

// bad: flags set when a component is NaN or Inf (device memory, and the host's copy), or NULL
template <typename ST>
__global__ void __launch_bounds__(kBlock) k_spinor_in(Geom g, ST *__restrict__ dst, long stride,
                                                      const double2 *__restrict__ lex, InputFlags bad) {
    __shared__ double2 sm[kIoTile * kIoRow];
    constexpr int N = IoWord<ST>::N;
    const int s0 = blockIdx.x * kIoTile, ns = min(kIoTile, g.V - s0);
    lex += ((size_t)blockIdx.y * g.V + s0) * 12;
    dst += (size_t)blockIdx.y * stride;
    bool fine = true;
#pragma unroll
    for (int q = 0; q < kIoTile * 12 / kBlock; q++) {
        const int e = threadIdx.x + q * kBlock;
        if (e < ns * 12) {
            const double2 v = __ldcs(lex + e);
            fine = fine && finite_bits(v.x) && finite_bits(v.y);
            sm[io_row(e / 12) + e % 12] = v;
        }
    }
    if (!fine && bad.device) {
        *(volatile int *)bad.device = 1;
        *(volatile int *)bad.host = 1;
    }
    __syncthreads();
    const int i = threadIdx.x & 31;   // the same for every word of this thread
    if (2 * i >= ns) return;
    const int gi = s0 / 2 + i, b = io_row_parity(g, gi);
#pragma unroll
    for (int k = threadIdx.x >> 5; k < 2 * N; k += kBlock / 32) {
        const int p = k >= N, j = k - p * N;
        dst[(size_t)k * g.Vh + gi] = IoWord<ST>::get(sm + io_row(2 * i + ((p + b) & 1)), j);
    }
}

// Nothing is written if *skip is set (an input of the same call was not finite).
template <typename ST>
__global__ void __launch_bounds__(kBlock) k_spinor_out(Geom g, double2 *__restrict__ lex, const ST *__restrict__ src,
                                                       long stride, const int *skip) {
    __shared__ double2 sm[kIoTile * kIoRow];
    constexpr int N = IoWord<ST>::N;
    if (skip && *(const volatile int *)skip) return;
    const int s0 = blockIdx.x * kIoTile, ns = min(kIoTile, g.V - s0);
    lex += ((size_t)blockIdx.y * g.V + s0) * 12;
    src += (size_t)blockIdx.y * stride;
    const int i = threadIdx.x & 31;
    if (2 * i < ns) {
        const int gi = s0 / 2 + i, b = io_row_parity(g, gi);
        constexpr int W = kBlock / 32, Q = (2 * N + W - 1) / W;   // words per thread
        ST w[Q];
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int k = (threadIdx.x >> 5) + q * W;
            if (k < 2 * N) w[q] = src[(size_t)k * g.Vh + gi];
        }
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int k = (threadIdx.x >> 5) + q * W, p = k >= N, j = k - p * N;
            if (k < 2 * N) IoWord<ST>::put(sm + io_row(2 * i + ((p + b) & 1)), j, w[q]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kIoTile * 12 / kBlock; q++) {
        const int e = threadIdx.x + q * kBlock;
        if (e < ns * 12) __stcs(lex + e, sm[io_row(e / 12) + e % 12]);
    }
}

template <typename ST>
cudaError_t spinor_in(const Geom &g, ST *dst, long stride, const double *lex, int n, InputFlags bad, cudaStream_t st) {
    k_spinor_in<ST><<<dim3((g.V + kIoTile - 1) / kIoTile, n), kBlock, 0, st>>>(g, dst, stride, (const double2 *)lex,
                                                                              bad);
    count_launches(1);
    return cudaGetLastError();
}
template <typename ST>
cudaError_t spinor_out(const Geom &g, double *lex, const ST *src, long stride, int n, const int *skip,
                       cudaStream_t st) {
    k_spinor_out<ST><<<dim3((g.V + kIoTile - 1) / kIoTile, n), kBlock, 0, st>>>(g, (double2 *)lex, src, stride, skip);
    count_launches(1);
    return cudaGetLastError();
}
template cudaError_t spinor_in<double2>(const Geom &, double2 *, long, const double *, int, InputFlags, cudaStream_t);
template cudaError_t spinor_in<float4>(const Geom &, float4 *, long, const double *, int, InputFlags, cudaStream_t);
template cudaError_t spinor_in<ffw>(const Geom &, ffw *, long, const double *, int, InputFlags, cudaStream_t);
template cudaError_t spinor_out<double2>(const Geom &, double *, const double2 *, long, int, const int *, cudaStream_t);
template cudaError_t spinor_out<float4>(const Geom &, double *, const float4 *, long, int, const int *, cudaStream_t);
template cudaError_t spinor_out<ffw>(const Geom &, double *, const ffw *, long, int, const int *, cudaStream_t);

// FP64 <-> FP32 even-odd spinors (double2 [p][12][Vh] <-> float4 [p][6][Vh]), one per grid row
__global__ void k_spinor_d2f(Geom g, const double2 *__restrict__ a, float4 *__restrict__ b) {
    a += (size_t)blockIdx.y * 12 * g.V;
    b += (size_t)blockIdx.y * 6 * g.V;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.V) return;
    const int p = t >= g.Vh, i = t - p * g.Vh;
    const double2 *x = a + (size_t)p * 12 * g.Vh + i;
    float4 *y = b + (size_t)p * 6 * g.Vh + i;
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const double2 u = x[(size_t)(2 * c) * g.Vh], v = x[(size_t)(2 * c + 1) * g.Vh];
        y[(size_t)c * g.Vh] = make_float4(d2f(u.x), d2f(u.y), d2f(v.x), d2f(v.y));
    }
}
__global__ void k_spinor_f2d(Geom g, const float4 *__restrict__ a, double2 *__restrict__ b) {
    a += (size_t)blockIdx.y * 6 * g.V;
    b += (size_t)blockIdx.y * 12 * g.V;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.V) return;
    const int p = t >= g.Vh, i = t - p * g.Vh;
    const float4 *x = a + (size_t)p * 6 * g.Vh + i;
    double2 *y = b + (size_t)p * 12 * g.Vh + i;
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const float4 w = x[(size_t)c * g.Vh];
        y[(size_t)(2 * c) * g.Vh] = make_double2(f2d(w.x), f2d(w.y));
        y[(size_t)(2 * c + 1) * g.Vh] = make_double2(f2d(w.z), f2d(w.w));
    }
}
cudaError_t spinor_d2f(const Geom &g, const double2 *a, float4 *b, cudaStream_t st, int n) {
    k_spinor_d2f<<<dim3(plain_grid(g.V), n), kBlock, 0, st>>>(g, a, b);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t spinor_f2d(const Geom &g, const float4 *a, double2 *b, cudaStream_t st, int n) {
    k_spinor_f2d<<<dim3(plain_grid(g.V), n), kBlock, 0, st>>>(g, a, b);
    count_launches(1);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ stencil
// out = a [g5] D_W(m0) in + b z, one thread per site, in FP32 and on some lattices in FP64 (wilson_f64).
// Bound in FP32: the latency of the neighbour gathers, which go to L2 three times in four, at 16 warps
// per SM (128 registers); at 64 x 32^3 with memory 60% and the L1 data pipe 48% busy (167 us: 0.71 of the
// copy bandwidth). One wave of blocks that stride over the lattice keeps the blocks of an SM and their
// neighbours on other SMs close together in time: 32^4 107 -> 90 us, 24^4 40 -> 35, 64 x 32^3 182 -> 170,
// 16^4 10.2 -> 9.2, against a block per 256 sites; with the order of site_of_thread 81, 31.3, 168 and 8.3.
template <typename R, typename ST>
__global__ void __launch_bounds__(kBlock, MinBlocks<R>::value)
    k_wilson(Geom g, const ST *__restrict__ U, const ST *__restrict__ in, ST *__restrict__ out, R m4, int g5, R a,
             const ST *z, R b, int spb) {
    if (threadIdx.x >= spb) return;
    for (int t = blockIdx.x * spb + threadIdx.x; t < g.V; t += gridDim.x * spb) {
        int p, i;
        site_of_thread(t, p, i);
        cpx<R> hop[12], own[12], res[12];
        wilson_hop<R>(g, U, in, p, i, hop);
        load_spinor<R>(in, g.Vh, p, i, own);
        wilson_combine<R>(m4, own, hop, res);
        if (g5) apply_g5(res);
        if (z) {
            cpx<R> zz[12];
            load_spinor<R>(z, g.Vh, p, i, zz);
#pragma unroll
            for (int c = 0; c < 12; c++) res[c] = a * res[c] + b * zz[c];
        } else {
#pragma unroll
            for (int c = 0; c < 12; c++) res[c] = a * res[c];
        }
        store_spinor<R>(out, g.Vh, p, i, res);
    }
}

// D_W(m0) in FP32 straight into n boundary vectors (complex doubles). The 256 sites of a block's turn
// are consecutive in both orders, so their results go through shared memory (26 words of 4 bytes
// per site: the 8-byte stores of half a warp fall on different banks) and leave in whole rows,
// instead of going to memory in the internal format and back through a kernel of their own
// (k_spinor_out): per site 96 B written and 96 B read less. 64 x 32^3: 170 + 114 us -> 226 us.
constexpr int kLexRow = 26;
__global__ void __launch_bounds__(kBlock, MinBlocks<float>::value)
    k_wilson_lex(Geom g, const float4 *__restrict__ U, const float4 *__restrict__ in, double2 *__restrict__ lex,
                 long stride, float m4, const int *skip) {
    extern __shared__ float lex_rows[];   // [kBlock][kLexRow]
    if (skip && *(const volatile int *)skip) return;
    in += blockIdx.y * stride;
    lex += blockIdx.y * stride * 2;
    for (int base = blockIdx.x * kBlock; base < g.V; base += gridDim.x * kBlock) {
        const int t = base + threadIdx.x;
        if (t < g.V) {
            int p, i;
            site_of_thread(t, p, i);
            cpx<float> hop[12], own[12], res[12];
            wilson_hop<float>(g, U, in, p, i, hop);
            load_spinor<float>(in, g.Vh, p, i, own);
            wilson_combine<float>(m4, own, hop, res);
            const int s = 2 * i + ((p + io_row_parity(g, i)) & 1) - base;
            float2 *row = reinterpret_cast<float2 *>(lex_rows + s * kLexRow);
#pragma unroll
            for (int c = 0; c < 12; c++) row[c] = make_float2(res[c].re, res[c].im);
        }
        __syncthreads();
        const int n = min(kBlock, g.V - base) * 12;
        for (int e = threadIdx.x; e < n; e += kBlock) {
            const float2 w = *reinterpret_cast<const float2 *>(lex_rows + (e / 12) * kLexRow + 2 * (e % 12));
            __stcs(lex + (size_t)base * 12 + e, make_double2(f2d(w.x), f2d(w.y)));
        }
        __syncthreads();   // the next turn overwrites the rows
    }
}
cudaError_t wilson_f32_lex(const Geom &g, const float4 *U, const float4 *in, double *lex, float m0, int n,
                           const int *skip, cudaStream_t st) {
    constexpr int smem = kBlock * kLexRow * sizeof(float);   // 26 KB
    const int slots = std::max(1, g.nsm * MinBlocks<float>::value / n), need = (g.V + kBlock - 1) / kBlock;
    k_wilson_lex<<<dim3(std::min(slots, need), n), kBlock, smem, st>>>(g, U, in, (double2 *)lex, 6L * g.V, m0 + 4.f, skip);
    count_launches(1);
    return cudaGetLastError();
}

// out = a [g5] D_W(m0) in + b z in FP64 or float-float, one warp per hop (hops.cuh); blockIdx.y =
// right-hand side, vectors `stride` words apart.
template <typename R>
__global__ void __launch_bounds__(kHopBlock, HopBlocks<R>::value)
    k_wilson_hops(Geom g, const typename HopTiles<R>::Link *__restrict__ U,
                  const typename HopTiles<R>::Store *__restrict__ in, typename HopTiles<R>::Store *__restrict__ out,
                  long stride, R m4, int g5, R a, const typename HopTiles<R>::Store *z, R b) {
    using H = HopTiles<R>;
    in += blockIdx.y * stride;
    out += blockIdx.y * stride;
    if (z) z += blockIdx.y * stride;
    const auto fm = H::factor(m4), fa = H::factor(a), fb = H::factor(b);
    const auto own = [&](int p, int i, int it, int e) { return H::load(in, g.Vh, p, i, it, e); };
    hop_tiles<R>(g, blockIdx.x, gridDim.x, U, in, own, [&](int p, int i, int it, int e, typename H::Elem hop, int,
                                                            typename H::Elem o) {
        typename H::Elem r = H::fma(fm, o, hop);
        r = H::mul(fa, H::neg_if(r, g5 && H::upper(it)));
        if (z) r = H::fma(fb, H::load(z, g.Vh, p, i, it, e), r);
        H::store(out, g.Vh, p, i, it, e, r);
    });
}
template <typename R, typename LT, typename ST>
static cudaError_t wilson_hops(const Geom &g, const LT *U, const ST *in, ST *out, long stride, int n, double m0, int g5,
                               double a, const ST *z, double b, cudaStream_t st) {
    k_wilson_hops<R><<<dim3(hop_grid<R>(g, n, false), n), kHopBlock, 0, st>>>(g, U, in, out, stride, R(m0 + 4.0), g5,
                                                                               R(a), z, R(b));
    count_launches(1);
    return cudaGetLastError();
}
// D_W(m0) in FP64 straight into n boundary vectors. The FP64 units bound the stencil at all sizes, so
// that 8-byte stores 192 bytes apart cost nothing beside them; a kernel for the way out and its
// launch cost 5 us of a call (35 at 4^4).
__global__ void __launch_bounds__(kHopBlock, HopBlocks<double>::value)
    k_wilson_hops_lex(Geom g, const double2 *__restrict__ U, const double2 *__restrict__ in, double *__restrict__ lex,
                      long stride, double m4, const int *skip) {
    using H = HopTiles<double>;
    if (skip && *(const volatile int *)skip) return;
    in += blockIdx.y * stride;
    lex += blockIdx.y * stride * 2;
    const auto own = [&](int p, int i, int it, int e) { return H::load(in, g.Vh, p, i, it, e); };
    hop_tiles<double>(g, blockIdx.x, gridDim.x, U, in, own, [&](int p, int i, int it, int e, double hop, int s, double o) {
        H::store_lex(lex, s, it, e, H::fma(m4, o, hop));
    });
}
cudaError_t wilson_f64_lex(const Geom &g, const double2 *U, const double2 *in, double *lex, double m0, int n,
                           const int *skip, cudaStream_t st) {
    k_wilson_hops_lex<<<dim3(hop_grid<double>(g, n, false), n), kHopBlock, 0, st>>>(g, U, in, lex, 12L * g.V, m0 + 4.0,
                                                                                    skip);
    count_launches(1);
    return cudaGetLastError();
}
// The same in float-float. The tile's 32 sites are consecutive in both orders; a lane holds one real of
// two spins, so the results go through shared memory (26 doubles per site) and leave in whole rows:
// per site 192 B written and 192 B read less. The whole call at 24^4 209 -> 198 us.
constexpr int kFfLexRow = 26;
__global__ void __launch_bounds__(kHopBlock, HopBlocks<ff>::value)
    k_wilson_ff_lex(Geom g, const ffl *__restrict__ U, const ffw *__restrict__ in, double2 *__restrict__ lex, ff m4,
                    const int *skip) {
    using H = HopTiles<ff>;
    __shared__ __align__(16) double rows[H::tile * kFfLexRow];
    if (skip && *(const volatile int *)skip) return;
    const auto fm = H::factor(m4);
    const int s0 = blockIdx.x * H::tile;
    const auto own = [&](int p, int i, int it, int e) { return H::load(in, g.Vh, p, i, it, e); };
    hop_tiles<ff>(g, blockIdx.x, gridDim.x, U, in, own, [&](int p, int i, int it, int, ff2 hop, int s, ff2 o) {
        const float4 w = ff2_word(H::fma(fm, o, hop));
        double *row = rows + (s - s0) * kFfLexRow + 2 * IoWord<ffw>::first(it) + (it & 1);
        row[0] = ff2d(w.x, w.z);
        row[6] = ff2d(w.y, w.w);
    });
    __syncthreads();
    const int n = min(H::tile, g.V - s0) * 12;
    for (int e = threadIdx.x; e < n; e += kHopBlock)
        __stcs(lex + (size_t)s0 * 12 + e,
               *reinterpret_cast<const double2 *>(rows + (e / 12) * kFfLexRow + 2 * (e % 12)));
}
cudaError_t wilson_ff_lex(const Geom &g, const ffl *U, const ffw *in, double *lex, double m0, const int *skip,
                          cudaStream_t st) {
    k_wilson_ff_lex<<<hop_grid<ff>(g, 1, false), kHopBlock, 0, st>>>(g, U, in, (double2 *)lex, ff(m0 + 4.0), skip);
    count_launches(1);
    return cudaGetLastError();
}
// FP64: one warp per hop, 1.60 ns a site at all sizes (2^19 sites and more); one thread per site takes 1.55 ns
// over the part of its threads that have a site, and is taken where that is at least 97.5% of
// them (whole waves of 304 blocks of 256): 28^4 0.987 -> 0.967 ms, 40 x 32^3 2.10 -> 2.05, 64 x 32^3
// 3.35 -> 3.25, but 32^4 (96%) 1.680 against 1.687 and 30^4 (95%) 1.299 against 1.326.
cudaError_t wilson_f64(const Geom &g, const double2 *U, const double2 *in, double2 *out, double m0, int g5,
                       double a, const double2 *z, double b, cudaStream_t st) {
    const LaunchShape ls = balanced_shape(g.V, g.nsm, MinBlocks<double>::value, 1 << 30);
    if (g.V >= 1 << 19 && g.V >= 0.975 * ls.grid * ls.block) {
        k_wilson<double><<<ls.grid, ls.block, 0, st>>>(g, U, in, out, m0 + 4.0, g5, a, z, b, ls.spb);
        count_launches(1);
        return cudaGetLastError();
    }
    return wilson_hops<double>(g, U, in, out, 0, 1, m0, g5, a, z, b, st);
}
cudaError_t wilson_batch_f64(const Geom &g, const double2 *U, const double2 *in, double2 *out, long stride, int nrhs,
                             double m0, int g5, double a, const double2 *z, double b, cudaStream_t st) {
    return wilson_hops<double>(g, U, in, out, stride, nrhs, m0, g5, a, z, b, st);
}
cudaError_t wilson_batch_ff(const Geom &g, const ffl *U, const ffw *in, ffw *out, long stride, int nrhs, double m0,
                            int g5, double a, const ffw *z, double b, cudaStream_t st) {
    return wilson_hops<ff>(g, U, in, out, stride, nrhs, m0, g5, a, z, b, st);
}
cudaError_t wilson_ff(const Geom &g, const ffl *U, const ffw *in, ffw *out, double m0, int g5, double a,
                      const ffw *z, double b, cudaStream_t st) {
    return wilson_hops<ff>(g, U, in, out, 0, 1, m0, g5, a, z, b, st);
}
cudaError_t wilson_f32(const Geom &g, const float4 *U, const float4 *in, float4 *out, float m0, int g5,
                       float a, const float4 *z, float b, cudaStream_t st) {
    if (g.tps32 == 4) return wilson_hops<float>(g, U, in, out, 0, 1, m0, g5, a, z, b, st);
    const LaunchShape ls = balanced_shape(g.V, g.nsm, MinBlocks<float>::value, g.nsm * MinBlocks<float>::value);
    k_wilson<float><<<ls.grid, ls.block, 0, st>>>(g, U, in, out, m0 + 4.0f, g5, a, z, b, ls.spb);
    count_launches(1);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ 16-bit stencil
// out = D_W(m0) in with 16-bit links and 16-bit spinors (FP16 with a per-site scale, or
// BF16), arithmetic in FP32: per site 4 x 24 B of links and the input and output spinors
// (52 B each in FP16, 48 B in BF16) are the algorithmic traffic, about half of the FP32
// stencil's 384 B.
template <typename LT, typename SIn, typename SOut>
__global__ void __launch_bounds__(kBlock, 2) k_wilson16(Geom g, const LT *__restrict__ U, SIn in, SOut out, float m4,
                                                      int spb) {
    const int t = blockIdx.x * spb + threadIdx.x;
    if (threadIdx.x >= spb || t >= g.V) return;
    int p, i;
    site_of_thread(t, p, i);
    cpx<float> hop[12], own[12], res[12];
    wilson_hop<float>(g, U, in, p, i, hop);
    load_spinor<float>(in, g.Vh, p, i, own);
    wilson_combine<float>(m4, own, hop, res);
    store_spinor<float>(out, g.Vh, p, i, res);
}

// FP32 links (rows 0 and 1, float4 [p][mu][3][Vh]) -> 16-bit links (uint2 [p][mu][3][Vh]):
// every float4 word becomes one 8-byte word.
template <typename L16>
__global__ void k_link_to16(const float4 *__restrict__ u32, L16 *u16, long n) {
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
        const float4 v = u32[k];
        reinterpret_cast<uint2 *>(u16)[k] = make_uint2(pack16(u16, v.x, v.y), pack16(u16, v.z, v.w));
    }
}
// FP32 even-odd spinor <-> FP16 (per-site scale) or BF16 even-odd spinor
template <typename S16>
__global__ void k_spinor_f2h(Geom g, const float4 *__restrict__ a, S16 b) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.V) return;
    const int p = t >= g.Vh, i = t - p * g.Vh;
    cpx<float> v[12];
    load_spinor<float>(a, g.Vh, p, i, v);
    store_spinor<float>(b, g.Vh, p, i, v);
}
template <typename S16C>
__global__ void k_spinor_h2f(Geom g, S16C a, float4 *__restrict__ b) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.V) return;
    const int p = t >= g.Vh, i = t - p * g.Vh;
    cpx<float> v[12];
    load_spinor<float>(a, g.Vh, p, i, v);
    store_spinor<float>(b, g.Vh, p, i, v);
}

cudaError_t links_to16(const Geom &g, const float4 *u32, void *u16, bool bf16, cudaStream_t st) {
    const long n = (long)g.V * 4 * 3;
    const int grid = (int)std::min<long>((n + kBlock - 1) / kBlock, 16L * g.nsm);
    if (bf16) k_link_to16<LinkB><<<grid, kBlock, 0, st>>>(u32, (LinkB *)u16, n);
    else k_link_to16<LinkH><<<grid, kBlock, 0, st>>>(u32, (LinkH *)u16, n);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t spinor_f2h(const Geom &g, const float4 *a, uint4 *v, float *norm, bool bf16, cudaStream_t st) {
    if (bf16) k_spinor_f2h<Bf16Spinor><<<plain_grid(g.V), kBlock, 0, st>>>(g, a, Bf16Spinor{v});
    else k_spinor_f2h<HalfSpinor><<<plain_grid(g.V), kBlock, 0, st>>>(g, a, HalfSpinor{v, norm});
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t spinor_h2f(const Geom &g, const uint4 *v, const float *norm, float4 *b, bool bf16, cudaStream_t st) {
    if (bf16) k_spinor_h2f<Bf16SpinorC><<<plain_grid(g.V), kBlock, 0, st>>>(g, Bf16SpinorC{v}, b);
    else k_spinor_h2f<HalfSpinorC><<<plain_grid(g.V), kBlock, 0, st>>>(g, HalfSpinorC{v, norm}, b);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t wilson_16(const Geom &g, const void *u16, const uint4 *in, const float *in_norm, uint4 *out, float *out_norm,
                      float m0, bool bf16, cudaStream_t st) {
    const LaunchShape ls = balanced_shape(g.V, g.nsm, 2, 1 << 30);
    if (bf16)
        k_wilson16<LinkB, Bf16SpinorC, Bf16Spinor><<<ls.grid, ls.block, 0, st>>>(
            g, (const LinkB *)u16, Bf16SpinorC{in}, Bf16Spinor{out}, m0 + 4.f, ls.spb);
    else
        k_wilson16<LinkH, HalfSpinorC, HalfSpinor><<<ls.grid, ls.block, 0, st>>>(
            g, (const LinkH *)u16, HalfSpinorC{in, in_norm}, HalfSpinor{out, out_norm}, m0 + 4.f, ls.spb);
    count_launches(1);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ float-float conversion
// hi = fl32(x), lo = fl32(x - hi) per real; back, hi + lo in FP64.
__global__ void k_links_d2ff(const double2 *__restrict__ x, ffl *__restrict__ y, long n) {
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
        const double2 v = x[k];
        ffl w;
        d2ff(v.x, w.rh, w.rl);
        d2ff(v.y, w.ih, w.il);
        y[k] = w;
    }
}
// Thread k: checkerboard index, colour and spin pair of one parity of one spinor (6 Vh of them
// per parity): two complex numbers of two spins <-> the words of their real and imaginary parts.
__global__ void k_spinor_d2ff(const double2 *__restrict__ x, ffw *__restrict__ y, int Vh, long n) {
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
        const long i = k % Vh, r = k / Vh;         // r = 6 * (parity and spinor) + 3 * pair + colour
        const long m = r / 6, w = r % 6, c = w % 3 + 6 * (w / 3);
        const double2 a = x[(12 * m + c) * Vh + i], b = x[(12 * m + c + 3) * Vh + i];
        ffw re, im;
        d2ff(a.x, re.h0, re.l0);
        d2ff(b.x, re.h1, re.l1);
        d2ff(a.y, im.h0, im.l0);
        d2ff(b.y, im.h1, im.l1);
        y[(12 * m + 2 * w) * Vh + i] = re;
        y[(12 * m + 2 * w + 1) * Vh + i] = im;
    }
}
__global__ void k_spinor_ff2d(const ffw *__restrict__ x, double2 *__restrict__ y, int Vh, long n) {
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
        const long i = k % Vh, r = k / Vh;
        const long m = r / 6, w = r % 6, c = w % 3 + 6 * (w / 3);
        const ffw a = x[(12 * m + 2 * w) * Vh + i], b = x[(12 * m + 2 * w + 1) * Vh + i];
        y[(12 * m + c) * Vh + i] = make_double2(ff2d(a.h0, a.l0), ff2d(b.h0, b.l0));
        y[(12 * m + c + 3) * Vh + i] = make_double2(ff2d(a.h1, a.l1), ff2d(b.h1, b.l1));
    }
}
static int conv_grid(long n) {
    long b = (n + kBlock - 1) / kBlock;
    const long cap = 16L * device_sm_count();
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}
cudaError_t links_d2ff(const double2 *x, ffl *y, long n, cudaStream_t st) {
    k_links_d2ff<<<conv_grid(n), kBlock, 0, st>>>(x, y, n);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t spinor_d2ff(const Geom &g, const double2 *x, ffw *y, cudaStream_t st, int n) {
    const long k = 6L * g.V * n;
    k_spinor_d2ff<<<conv_grid(k), kBlock, 0, st>>>(x, y, g.Vh, k);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t spinor_ff2d(const Geom &g, const ffw *x, double2 *y, cudaStream_t st, int n) {
    const long k = 6L * g.V * n;
    k_spinor_ff2d<<<conv_grid(k), kBlock, 0, st>>>(x, y, g.Vh, k);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace ovl
