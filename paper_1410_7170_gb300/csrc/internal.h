// Internal interfaces between the library's translation units (not part of the ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <complex>
#include <string>

#include "common.cuh"
#include "ff.cuh"

namespace ovl {

constexpr int kMaxPoles = 64;
constexpr int kBlock = 256;             // threads per block of site-parallel kernels
constexpr int kMaxRedBlocks = 4096;     // cap on blocks of a reducing kernel (grid-stride beyond)
constexpr int kMaxRedValues = 4;        // doubles reduced by one kernel

// Scratch of the deterministic two-level reductions: per-block partial sums, and
// a counter the last finishing block uses to find that it is last.
struct RedScratch {
    double *partials;      // [kMaxRedValues][kMaxRedBlocks]
    unsigned *counter;     // one word, zero between launches
    // of grid row y, where each has one reduced value and a counter of its own
    __device__ RedScratch row(int y) const { return RedScratch{partials + (size_t)y * kMaxRedBlocks, counter + y}; }
};

// Minimum resident blocks per SM requested from the compiler for the one-thread-per-site stencils:
// at 128 registers two 256-thread blocks fit on an SM (one wave of 256 blocks at 16^4 on 152 SMs).
template <typename R> struct MinBlocks { static constexpr int value = 1; };
template <> struct MinBlocks<double> { static constexpr int value = 2; };
template <> struct MinBlocks<float> { static constexpr int value = 2; };

// SMs of the current device (queried once per device and cached).
int device_sm_count();

// Blocks of a grid-striding reduction over n_threads elements: enough to fill every SM a
// few times, few enough that the per-block partials and the arrival counter stay cheap.
inline int red_grid(long n_threads) {
    long b = (n_threads + kBlock - 1) / kBlock;
    const long cap = 4L * device_sm_count();
    if (b > cap) b = cap;
    if (b > kMaxRedBlocks) b = kMaxRedBlocks;
    if (b < 1) b = 1;
    return (int)b;
}
// Launch shape for a site-parallel kernel over n sites: the block count is a multiple of
// nsm * per_sm (every SM holds the same number of blocks in every wave), each block owns
// spb consecutive sites (thread t < spb of block b handles site b * spb + t, striding by
// grid * spb), and the block size is spb rounded up to whole warps.
struct LaunchShape {
    int grid, block, spb;
};
inline LaunchShape balanced_shape(long n, int nsm, int per_sm, int max_blocks) {
    if (nsm <= 0) nsm = 1;
    const long slots = (long)nsm * per_sm;
    long waves = (n + slots * kBlock - 1) / (slots * kBlock);
    if (waves < 1) waves = 1;
    long nblk = slots * waves;
    if (nblk > max_blocks) nblk = (max_blocks / slots) * slots;
    if (nblk < 1) nblk = 1;
    long spb = (n + nblk - 1) / nblk;
    spb = (spb + 7) / 8 * 8;         // quarter warps on whole lines (site_of_thread)
    if (spb > kBlock) spb = kBlock;   // more sites than threads: the kernel strides
    const int T = (int)((spb + 31) / 32 * 32);
    return LaunchShape{(int)nblk, T, (int)spb};
}

inline int plain_grid(long n_threads) {
    long b = (n_threads + kBlock - 1) / kBlock;
    return (int)(b < 1 ? 1 : b);
}

// ---------------------------------------------------------------- layouts / gauge
// lex: V*4*9 complex doubles [s][mu][a][b]. Writes the FP64 and FP32 12-real copies;
// sets *bad to 1 if some link misses unitarity or det = 1 by more than tol.
cudaError_t pack_gauge(const Geom &g, const double *lex, double2 *u64, float4 *u32, int *bad, double tol,
                       cudaStream_t st);
// n boundary vectors [V][12] complex doubles, back to back <-> even-odd spinors `stride` storage
// words apart, ST = double2, float4 or ffw. Reading sets both flags of `bad` (if given) when a
// component is NaN or Inf; writing does nothing if *skip (device memory, nullable) is set.
struct InputFlags {
    int *device, *host;   // host: pinned memory, written from the device
};
template <typename ST>
cudaError_t spinor_in(const Geom &g, ST *dst, long stride, const double *lex, int n, InputFlags bad, cudaStream_t st);
template <typename ST>
cudaError_t spinor_out(const Geom &g, double *lex, const ST *src, long stride, int n, const int *skip, cudaStream_t st);

// even-odd FP64 <-> FP32 conversion of n spinors back to back
cudaError_t spinor_d2f(const Geom &g, const double2 *a, float4 *b, cudaStream_t st, int n = 1);
cudaError_t spinor_f2d(const Geom &g, const float4 *a, double2 *b, cudaStream_t st, int n = 1);

// ---------------------------------------------------------------- stencils
// out = a * [gamma5] D_W(m0) in + b * z   (z may be NULL; then b is ignored)
cudaError_t wilson_f64(const Geom &g, const double2 *U, const double2 *in, double2 *out, double m0, int g5,
                       double a, const double2 *z, double b, cudaStream_t st);
cudaError_t wilson_f32(const Geom &g, const float4 *U, const float4 *in, float4 *out, float m0, int g5,
                       float a, const float4 *z, float b, cudaStream_t st);
// D_W(m0) of n even-odd spinors back to back into n boundary vectors; nothing is written if *skip
// (device memory, nullable) is set
cudaError_t wilson_f64_lex(const Geom &g, const double2 *U, const double2 *in, double *lex, double m0, int n,
                           const int *skip, cudaStream_t st);
cudaError_t wilson_f32_lex(const Geom &g, const float4 *U, const float4 *in, double *lex, float m0, int n,
                           const int *skip, cudaStream_t st);
cudaError_t wilson_ff_lex(const Geom &g, const ffl *U, const ffw *in, double *lex, double m0, const int *skip,
                          cudaStream_t st);
// float-float stencil; fields in the layouts of ff.cuh
cudaError_t wilson_ff(const Geom &g, const ffl *U, const ffw *in, ffw *out, double m0, int g5, double a,
                      const ffw *z, double b, cudaStream_t st);
// 16-bit stencil: out = D_W(m0) in with 16-bit links (from links_to16) and 16-bit spinors,
// FP16 with a per-site scale (norm arrays of V floats) or BF16 (norms unused), FP32 arithmetic
cudaError_t links_to16(const Geom &g, const float4 *u32, void *u16, bool bf16, cudaStream_t st);
cudaError_t spinor_f2h(const Geom &g, const float4 *a, uint4 *v, float *norm, bool bf16, cudaStream_t st);
cudaError_t spinor_h2f(const Geom &g, const uint4 *v, const float *norm, float4 *b, bool bf16, cudaStream_t st);
cudaError_t wilson_16(const Geom &g, const void *u16, const uint4 *in, const float *in_norm, uint4 *out, float *out_norm,
                      float m0, bool bf16, cudaStream_t st);
// FP64 -> float-float links (n complex words), and FP64 <-> float-float conversion of n even-odd
// spinors back to back
cudaError_t links_d2ff(const double2 *x, ffl *y, long n, cudaStream_t st);
cudaError_t spinor_d2ff(const Geom &g, const double2 *x, ffw *y, cudaStream_t st, int n = 1);
cudaError_t spinor_ff2d(const Geom &g, const ffw *x, double2 *y, cudaStream_t st, int n = 1);

// ---------------------------------------------------------------- BLAS-1 (flat arrays of n doubles)
// Reductions return through device memory `res` (written by the last block).
cudaError_t dev_norm2(const double *x, long n, double *res, RedScratch rs, cudaStream_t st);
// res[0] = Re <x,y>, res[1] = Im <x,y> (complex interleaved, n doubles = n/2 complex)
cudaError_t dev_cdot(const double *x, const double *y, long n, double *res, RedScratch rs, cudaStream_t st);
// y = a x + b y (real a, b)
cudaError_t dev_axpby(double a, const double *x, double b, double *y, long n, cudaStream_t st);
// y += (ar + i ai) x  (complex, interleaved)
cudaError_t dev_caxpy(double ar, double ai, const double *x, double *y, long n, cudaStream_t st);
// Arnoldi helpers: out[2k..2k+1] = <v_k, w> for k < m (v_k = base + k*stride), deterministic
cudaError_t dev_multidot(const double *base, long stride, int m, const double *w, long n, double *out,
                         double *partials, cudaStream_t st);
// w += sum_k c_k v_k, c complex interleaved in device memory (m <= 128)
cudaError_t dev_multiaxpy(const double *base, long stride, int m, const double *c, double *w, long n,
                          cudaStream_t st);
// float <-> double conversion of flat arrays (same element order)
cudaError_t dev_d2f(const double *x, float *y, long n, cudaStream_t st);
cudaError_t dev_f2d(const float *x, double *y, long n, cudaStream_t st);
// y = a*x + b*y on floats
cudaError_t dev_axpby_f(float a, const float *x, float b, float *y, long n, cudaStream_t st);
cudaError_t dev_norm2_f(const float *x, long n, double *res, RedScratch rs, cudaStream_t st);
cudaError_t dev_cdot_f(const float *x, const float *y, long n, double *res, RedScratch rs, cudaStream_t st);
// multi-dot / multi-axpy with float vectors (accumulation in double)
cudaError_t dev_multidot_f(const float *base, long stride, int m, const float *w, long n, double *out,
                           double *partials, cudaStream_t st);

// Gram-Schmidt steps of the FGMRES solvers, several right-hand sides at once, without the host.
// Vector y of a basis entry is n reals after vector 0. T = float or double.
struct RowList {
    int n, row[12];   // the right-hand sides that take part (grid rows)
};
// Record of row k at out + k * ostride: [0, 2m) = <v_i, w> (complex), [2m] = ||w||^2, [2m+1] = 0,
// then hn = sqrt(max(0, ||w||^2 - sum |<v_i, w>|^2)), 1 / hn (0 for hn = 0), and 1 if one pass is
// enough (one_pass allowed and hn^2 > 0.1 ||w||^2), else 0. Needs 2m + 5 doubles.
// prev: the record of the first pass, or NULL; where it says that one pass is enough nothing is done.
constexpr int gs_record(int m) { return 2 * m + 6; }
template <typename T>
cudaError_t gs_dots(const T *base, long stride, int m, const T *w, long n, const RowList &rows, double *out,
                    long ostride, bool one_pass, const double *prev, double *partials, unsigned *counters,
                    cudaStream_t st);
// Subtracts sum_i h_i v_i, h from the record of this pass. First pass (prev NULL): the result goes to
// next, scaled by 1 / hn, where one pass is enough, and back to w otherwise; second pass: to next,
// scaled, except where one pass was enough.
template <typename T>
cudaError_t gs_subtract(const T *base, long stride, int m, const double *h, long ostride, const double *prev, T *w,
                        T *next, long n, const RowList &rows, cudaStream_t st);
// x (+)= sum_i c_i v_i, i < cols.n[k] <= m for row k, its complex coefficients at c + 2 * m * k (device);
// add = false: assigned. Entries past a row's own columns are not read: its solver may never have
// written them, and a zero coefficient would turn a NaN there into a NaN in x.
struct RowColumns {
    int n[12];
};
template <typename T>
cudaError_t gs_combine(const T *base, long stride, int m, const double *c, T *x, bool add, long n, const RowList &rows,
                       const RowColumns &cols, cudaStream_t st);
cudaError_t dev_multiaxpy_f(const float *base, long stride, int m, const double *c, float *w, long n,
                            cudaStream_t st);
// x[k] = seeded pseudo-random values in [-1, 1) (a counter hash of k and the seed)
cudaError_t fill_random_f32(float *x, long n, unsigned seed, cudaStream_t st);

// ---------------------------------------------------------------- multishift CG
constexpr int kMaxRing = 4;   // iterations whose shift updates are done together, at most
constexpr int kBatchRing = 2;   // the same in batches, where the rings' vectors count as often as there are right-hand sides

// Device-side state of one multishift solve (Q^2 + sigma_l) x_l = b, l < n, with the
// Zolotarev accumulation y = b + sum_l w_l x_l. sigma[0] is the base (smallest) shift.
struct MsState {
    int n;                     // shifts
    int iter;                  // iterations done
    int done;                  // 1: all shifts converged (kernels then do nothing)
    int status;                // 0 ok, 1 breakdown / non-finite scalar
    double bb;                 // ||b||^2
    double rr;                 // ||r_k||^2 (base residual)
    double pp;                 // ||p_0||^2 by the recurrence ||p_k||^2 = ||r_k||^2 + b_{k-1}^2 ||p_{k-1}||^2
    double alpha, alpha_prev, beta_prev;
    float alpha_f[2], sigma0_f[2];   // alpha and sigma[0] as float-float (hi, lo)
    double tol;                // target relative accuracy of the rational function
    double sigma[kMaxPoles];   // shifts
    double w[kMaxPoles];       // weights of x_l in y
    double crit[kMaxPoles];    // drop shift l when crit_l * |zeta_l| * ||r|| <= tol * ||b||
    double zeta[kMaxPoles], zeta_prev[kMaxPoles];
    double ratio[kMaxPoles], critz2[kMaxPoles];     // zeta_{k+1} / zeta_k, (crit zeta_{k+1})^2
    double scale, inv_rr, inv_bb;                   // scale, 1 / (scale ||r||^2), 1 / (scale ||b||^2)
    int active[kMaxPoles];
    // iterations whose shift updates are pending, oldest first: the coefficients of the rescaled
    // directions (y += wa p~_l, p~_l = r + bl p~_l) and the shifts that take part (bit l)
    int npend;
    unsigned on[kMaxRing][kMaxPoles / 32];
    double wa[kMaxRing][kMaxPoles], bl[kMaxRing][kMaxPoles];
    float wa_f[kMaxRing][kMaxPoles][2], bl_f[kMaxRing][kMaxPoles][2], beta_f[2];   // the same and beta_prev as
                                                                                   // float-float (hi, lo)
    int *hist;                 // optional: hist[k] = shifts updated in iteration k (instrumentation)
    int hist_cap;
};

// Workspace vectors of nrhs multishift solves in storage type ST. Residuals and base directions are
// rings of `ring` vectors per right-hand side (a power of two, at most kMaxRing): r_k and p_0(k) are
// entry k % ring. t = Q p_0 and y (the accumulated argument of the rational function) are one vector
// per right-hand side, the directions p_l, l >= 1, start at p + y * prow.
template <typename ST>
struct MsBatch {
    ST *r, *p0, *t, *y, *p;
    long stride;   // words per vector
    long prow;
    int ring;
    __host__ __device__ ST *r_at(int y_, int k) const { return r + ((long)y_ * ring + (k & (ring - 1))) * stride; }
    __host__ __device__ ST *p0_at(int y_, int k) const { return p0 + ((long)y_ * ring + (k & (ring - 1))) * stride; }
};
// Vectors per right-hand side with npole directions.
constexpr int ms_vectors(int npole, int ring) { return 2 * ring + 2 + npole - 1; }

// Event records around the kernels of an iteration (instrumentation; ev = NULL: none). only >= 0:
// just from record `only` on. flags: cudaEventRecordExternal inside graphs.
struct MsEvents {
    cudaEvent_t *ev = nullptr;
    unsigned flags = 0;
    int only = 0;
    cudaError_t record(int k, cudaStream_t st) const {
        return ev && k >= only ? cudaEventRecordWithFlags(ev[k], st, flags) : cudaSuccess;
    }
};

// Half-precision variant of the FP32 multishift vectors: p_0 (the base direction, which
// drives the Krylov process), r, t and y stay FP32; the shifted directions p_l, l >= 1,
// are stored as FP16 scaled by a per-site FP32 norm (see HalfSpinor).
struct MsVectorsH {
    float4 *r, *t, *y, *p0;
    uint4 *ph;          // p_l for l >= 1 at ph + (l - 1) * words_h
    float *pn;          // their per-site norms at pn + (l - 1) * V
    long words;         // float4 words per FP32 vector (6 V)
    long words_h;       // uint4 words per FP16 vector (3 V)
};

// Right-hand sides of a launch, and of the batch that they belong to: a batch that does not fit the
// memory is done in parts, with the launch shapes of the whole (they decide the order of the
// reductions), so that its results don't depend on the memory that was free.
struct MsRows {
    int n, of;
    MsRows(int n_) : n(n_), of(n_) {}
    MsRows(int n_, int of_) : n(n_), of(of_) {}
};
// One multishift iteration of nrhs right-hand sides (state st[y]; grid row y) = three launches: Q p,
// residual update, and p_0 or, where flush is set, the pending shift updates with it. A caller sets
// flush at least in every ring-th iteration, and in the last one before it reads y or the state.
// rs.partials: nrhs * kMaxRedBlocks doubles; counters: nrhs words, zero between launches.
cudaError_t ms_init(const Geom &g, MsRows nrhs, MsState *s, MsBatch<double2> v, const double2 *b, RedScratch rs,
                    unsigned *counters, cudaStream_t st);
cudaError_t ms_init(const Geom &g, MsRows nrhs, MsState *s, MsBatch<float4> v, const float4 *b, RedScratch rs,
                    unsigned *counters, cudaStream_t st);
cudaError_t ms_init(const Geom &g, MsRows nrhs, MsState *s, MsBatch<ffw> v, const ffw *b, RedScratch rs,
                    unsigned *counters, cudaStream_t st);
cudaError_t ms_iter(const Geom &g, const double2 *U, double m0, MsRows nrhs, MsState *s, MsBatch<double2> v, RedScratch rs,
                    unsigned *counters, bool flush, cudaStream_t st, const MsEvents &ev);
cudaError_t ms_iter(const Geom &g, const float4 *U, double m0, MsRows nrhs, MsState *s, MsBatch<float4> v, RedScratch rs,
                    unsigned *counters, bool flush, cudaStream_t st, const MsEvents &ev);
cudaError_t ms_iter(const Geom &g, const ffl *U, double m0, MsRows nrhs, MsState *s, MsBatch<ffw> v, RedScratch rs,
                    unsigned *counters, bool flush, cudaStream_t st, const MsEvents &ev);
// one right-hand side with 16-bit shifted directions, updated in every iteration
cudaError_t ms_init_half(const Geom &g, int n, MsState *s, MsVectorsH v, const float4 *b, RedScratch rs, bool bf16,
                         cudaStream_t st);
cudaError_t ms_iter_half(const Geom &g, const float4 *U, double m0, MsState *s, MsVectorsH v, RedScratch rs, bool bf16,
                         cudaStream_t st, const MsEvents &ev);

// ---------------------------------------------------------------- several right-hand sides
constexpr int kMaxBatch = 12;   // right-hand sides per batch (threads 32 x nrhs per block)

// out_y = a [gamma5] D_W(m0) in_y + b z_y for y < nrhs; vectors `stride` storage words apart.
cudaError_t wilson_batch_f64(const Geom &g, const double2 *U, const double2 *in, double2 *out, long stride, int nrhs,
                             double m0, int g5, double a, const double2 *z, double b, cudaStream_t st);
cudaError_t wilson_batch_ff(const Geom &g, const ffl *U, const ffw *in, ffw *out, long stride, int nrhs, double m0,
                            int g5, double a, const ffw *z, double b, cudaStream_t st);
cudaError_t wilson_batch_f32(const Geom &g, const float4 *U, const float4 *in, float4 *out, long stride, int nrhs,
                             float m0, int g5, float a, const float4 *z, float b, cudaStream_t st);

// Process-wide count of kernel launches issued by the library (instrumentation).
void count_launches(long n);
long launches_total();
void set_launch_counting(bool on);

// Message returned by ovl_last_error(NULL) on the calling thread.
void set_thread_error(const std::string &msg);

// ---------------------------------------------------------------- host Zolotarev
int zolotarev_host(double k, int n, double *d0, double *a, double *c, double *delta);

// Eigenvalues (ascending) and eigenvectors (columns of Z, row-major) of a small complex
// Hermitian matrix A (row-major, overwritten), by Householder tridiagonalisation and implicit QR; 0 on convergence.
int hermitian_eig(int n, std::complex<double> *A, double *w, std::complex<double> *Z);

}  // namespace ovl
