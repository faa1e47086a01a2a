// Multishift conjugate gradients for the Zolotarev partial fractions of sign(Q).
//
// The n shifted systems (Q^2 + sigma_l) x_l = b share one Krylov space. The base
// system (smallest shift sigma_0) runs plain CG; shift l keeps its own direction
// p_l and scalars from the shifted-CG recurrences (Jegerlehner, hep-lat/9612014;
// Frommer, "BiCGStab(l) for families of shifted linear systems", 2003):
//
//   zeta_{k+1} = zeta_k zeta_{k-1} a_{k-1} /
//                ( a_k b_{k-1} (zeta_{k-1} - zeta_k) + zeta_{k-1} a_{k-1} (1 + (sigma_l - sigma_0) a_k) )
//   a^l_k = a_k zeta_{k+1}/zeta_k,   b^l_k = b_k (zeta_{k+1}/zeta_k)^2
//   x_l += a^l_k p_l,   p_l = zeta_{k+1} r_{k+1} + b^l_k p_l,   r^l = zeta r.
//
// x_l is never stored: the rational function needs only y = b + sum_l w_l x_l, so
// each iteration adds w_l a^l_k p_l to y. Shift l is dropped once its residual
// bound crit_l |zeta_l| ||r|| falls below tol ||b||.
//
// The directions are stored rescaled, p~_l = p_l / zeta_l (p~_0 = p_0, zeta_0 = 1; p~_l
// stays of the size of r). The updates then take one fused multiply-add per real each,
// against three instructions for the unscaled form (the FP64 shift update is bound by
// the FP64 pipes):
//   y += (w_l a_k zeta_{k+1}) p~_l,   p~_l = r_{k+1} + (b_k zeta_{k+1}/zeta_k) p~_l.
//
// One iteration = three kernels, all scalars stay on the device:
//   ms_q:  t = Q p_0 (stencil with gamma5),                          reduce ||t||^2 -> alpha
//   ms_r:  r_{k+1} = r_k - alpha (gamma5 D_W t + sigma_0 p_0),        reduce ||r_{k+1}||^2 -> beta, shift scalars
//   ms_p0: p_0 = r_{k+1} + beta p_0                                   (the next ms_q reads it)
// and, in every `ring`-th iteration in place of ms_p0,
//   ms_shifts: for the pending iterations k in turn
//              y += sum_l w~_l p~_l ; p~_l = r_{k+1} + b~_l p~_l      (pure streaming)
// The last `ring` residuals and base directions are kept, and so are the coefficients of those
// iterations (MsState::wa, bl, on): the shifted directions only feed y, so they can be brought up
// to date several iterations at a time, reading and writing each p~_l and y once instead of every
// time. Reals per site and iteration with n shifts: 72 + 48 n with an update in every iteration,
// 120 + 12 n with ring = 4, 120 + 24 n with ring = 2 (batches, where the extra vectors count).
// Measured per iteration (us), updates in every iteration -> ring 4: FP32 32^4 469 (fused into the
// residual kernel) -> 350, FP32 16^4 41 (fused) -> 35, float-float 16^4 116 -> 107 (the updates
// themselves 35 -> 22, bound by their float-float arithmetic), FP64 8^4 43 -> 41.
// (p_0, Q^2 p_0) = ||Q p_0||^2 because Q is Hermitian (Eq. gamma_5_symmetry).
// After convergence (state->done) every kernel returns at once, so a fixed number
// of iterations can be queued or captured in a CUDA graph without host round trips.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "hops.cuh"
#include "internal.h"
#include "reduce.cuh"
#include "wilson_site.cuh"

namespace ovl {

namespace {

// Scalars that the streaming and stencil kernels of the FP32 arithmetics read are stored as
// float-float beside their FP64 value: converting them in every thread kept the FP64 units busy for
// 4 us of every ms_p0 and for a third of every float-float stencil.
__device__ __forceinline__ void store_ff(float *to, double x) {
    const ff f(x);
    to[0] = f.hi;
    to[1] = f.lo;
}

// alpha = (r, r) / (p, (Q^2 + sigma_0) p) with (p, Q^2 p) = ||Q p||^2, reduced by ms_q. ||p||^2 of one
// right-hand side comes from the scalar recurrence ||p_k||^2 = ||r_k||^2 + beta^2 ||p_{k-1}||^2, which
// holds because r_k is orthogonal to p_{k-1} in CG; this spares ms_q the sum. Batches (OWN) sum it, into the
// same number, ||Q p||^2 + sigma_0 ||p||^2: in FP32 the recurrence drifts to 5e-7 in 40 iterations (16^4),
// the sum is good to 1e-9. Float-float batches use the recurrence, as one right-hand side does.
template <bool OWN>
struct AlphaFin {
    MsState *s;
    struct In {
        double sigma0, pp, rr;
    };
    __device__ In before() const { return {s->sigma[0], s->pp, s->rr}; }
    __device__ void operator()(const double *v, const In &in) const {
        const double pAp = OWN ? v[0] : v[0] + in.sigma0 * in.pp;
        const double a = in.rr / pAp;
        if (!(pAp > 0.0) || !isfinite(a)) {
            s->status = 1;
            s->done = 1;
            return;
        }
        s->alpha = a;
        store_ff(s->alpha_f, a);
    }
};
// sum + sigma_0 b for a thread's sums of ||Q p||^2 and ||p||^2; in FP32 with both words of sigma_0, whose
// rounding all threads would share
__device__ __forceinline__ void add_shifted(const MsState &s, double b, double &sum) { sum = fma_r(s.sigma[0], b, sum); }
__device__ __forceinline__ void add_shifted(const MsState &s, const fsum &b, fsum &sum) {
    sum.add(__fmul_rn(s.sigma0_f[0], b.s));
    sum.add(fma_r(s.sigma0_f[1], b.s, __fmul_rn(s.sigma0_f[0], b.e)));
}

// Shift scalars of an iteration, in two parts, one lane per shift (lane j: shifts j, j + 32). A
// dependent FP64 instruction takes 64 clocks or more on GB300 (half a lane per clock and scheduler),
// so all divisions and roots at the end of the residual kernel cost about 3 us. ShiftScalars does what
// does not need ||r_{k+1}||^2, in a block of its own during that kernel: zeta_{k+1}, the coefficients
// of y, zeta_{k+1} / zeta_k, the squared drop criterion and the reciprocals of ||r_k||^2 and ||b||^2
// (scaled, so that they exist for any ||b||^2 > 0). ShiftFin does the rest at the end of the kernel.
struct ShiftScalars {
    MsState *s;
    __device__ void operator()(int lane) const {
        const double a = s->alpha, ap = s->alpha_prev, bp = s->beta_prev;
        const int slot = s->npend;
        for (int l = lane; l < s->n; l += 32) {
            if (!s->active[l]) continue;
            const double z = s->zeta[l], zp = s->zeta_prev[l];
            double zn = 1.0;
            if (l > 0) {
                const double den = a * bp * (zp - z) + zp * ap * (1.0 + (s->sigma[l] - s->sigma[0]) * a);
                zn = (den != 0.0) ? z * zp * ap / den : 0.0;
            }
            // directions stored as p~_l = p_l / zeta_l (see the header): y += w_l a zeta_new p~_l,
            // p~_l = r + b ratio p~_l
            const double wa = s->w[l] * (a * zn);
            s->wa[slot][l] = wa;
            store_ff(s->wa_f[slot][l], wa);
            s->ratio[l] = (z != 0.0) ? zn / z : 0.0;
            const double c = s->crit[l] * zn;
            s->critz2[l] = c * c;
            s->zeta_prev[l] = z;
            s->zeta[l] = zn;
        }
        if (lane == 0) {
            const double scale = s->bb < 1e-150 ? 0x1p500 : 1.0;
            s->scale = scale;
            s->inv_rr = 1.0 / (s->rr * scale);
            s->inv_bb = 1.0 / (s->bb * scale);
        }
    }
};
struct ShiftFin {
    MsState *s;
    static constexpr int kSets = kMaxPoles / 32;
    struct In {
        double scale, inv_rr, inv_bb, tol, pp, alpha, ratio[kSets], critz2[kSets];
        int n, slot, iter, hist_cap, active[kSets];
        int *hist;
    };
    __device__ In before(int lane) const {
        In in{s->scale, s->inv_rr, s->inv_bb, s->tol, s->pp, s->alpha, {}, {}, s->n, s->npend, s->iter, s->hist_cap, {},
              s->hist};
#pragma unroll
        for (int j = 0; j < kSets; j++) {
            in.ratio[j] = s->ratio[32 * j + lane];
            in.critz2[j] = s->critz2[32 * j + lane];
            in.active[j] = s->active[32 * j + lane];
        }
        return in;
    }
    __device__ void operator()(const double *v, int lane, const In &in) const {
        const double rr_new = v[0], rs = rr_new * in.scale;
        const double beta = rs * in.inv_rr;
        if (!isfinite(beta)) {
            if (lane == 0) {
                s->status = 1;
                s->done = 1;
            }
            return;
        }
        const double rel = rs * in.inv_bb, tol2 = in.tol * in.tol;
        int any = 0, nupd = 0;
#pragma unroll
        for (int j = 0; j < kSets; j++) {
            const int l = 32 * j + lane;
            const bool on = l < in.n && in.active[j];
            const unsigned m = __ballot_sync(0xffffffffu, on);
            if (lane == 0) s->on[in.slot][j] = m;
            nupd += __popc(m);
            if (!on) continue;
            const double bl = beta * in.ratio[j];
            s->bl[in.slot][l] = bl;
            store_ff(s->bl_f[in.slot][l], bl);
            // residual bound after this iteration's update: this was the shift's last one, except
            // for the base shift, whose direction drives the Krylov space
            if (in.critz2[j] * rel > tol2) any = 1;
            else if (l > 0) s->active[l] = 0;
        }
        any = __any_sync(0xffffffffu, any);
        if (lane == 0) {
            if (in.hist && in.iter < in.hist_cap) in.hist[in.iter] = nupd;
            s->alpha_prev = in.alpha;
            s->beta_prev = beta;
            store_ff(s->beta_f, beta);
            s->pp = rr_new + beta * beta * in.pp;
            s->rr = rr_new;
            s->iter = in.iter + 1;
            s->npend = in.slot + 1;
            if (!any) s->done = 2;   // ms_shifts brings y up to date, then the solve is done
        }
    }
};

// A thread's sum over its sites
template <typename R> struct SiteSum;
template <> struct SiteSum<float> { using type = fsum; };
template <> struct SiteSum<double> { using type = double; };
__device__ __forceinline__ void sum_add(fsum &s, float x) { s.add(x); }
__device__ __forceinline__ void sum_add(double &s, double x) { s += x; }

// One thread per site (FP32; FP64 on large lattices), right-hand side blockIdx.y:
// t = gamma5 D_W(m) p_0 ; ||t||^2 (OWN: + sigma_0 ||p_0||^2) -> alpha.
template <typename R, bool OWN, typename ST>
__global__ void __launch_bounds__(kBlock, MinBlocks<R>::value)
    k_ms_q_site(Geom g, const ST *__restrict__ U, R m4, MsState *st, MsBatch<ST> v, RedScratch rs, int spb) {
    MsState *s = st + blockIdx.y;
    if (s->done) return;
    const ST *__restrict__ p0 = v.p0_at(blockIdx.y, s->iter);
    ST *__restrict__ t = v.t + blockIdx.y * v.stride;
    // FP32: a site's sum plain, a thread's and a warp's with their errors, then FP64 (grid_reduce)
    typename SiteSum<R>::type sum[1] = {}, psum = {};
    const bool lane_has_sites = threadIdx.x < spb;
    for (int k = blockIdx.x * spb + threadIdx.x; lane_has_sites && k < g.V; k += gridDim.x * spb) {
        int p, i;
        site_of_thread(k, p, i);
        cpx<R> hop[12], own[12], res[12];
        wilson_hop<R>(g, U, p0, p, i, hop);
        load_spinor<R>(p0, g.Vh, p, i, own);
        wilson_combine<R>(m4, own, hop, res);
        apply_g5(res);
        store_spinor<R>(t, g.Vh, p, i, res);
        R a0 = 0;
#pragma unroll
        for (int c = 0; c < 12; c++) a0 += norm2(res[c]);
        sum_add(sum[0], a0);
        if (OWN) {
            a0 = 0;
#pragma unroll
            for (int c = 0; c < 12; c++) a0 += norm2(own[c]);
            sum_add(psum, a0);
        }
    }
    if (OWN) add_shifted(*s, psum, sum[0]);
    grid_reduce<1>(sum, rs.row(blockIdx.y), AlphaFin<OWN>{s});
}

// r_{k+1} = r_k - alpha (gamma5 D_W(m) t + sigma0 p0) ; ||r_{k+1}||^2 -> shift scalars. Block 0 forms the shift
// scalars that need only alpha_k (ShiftScalars); it takes no sites, unless `share` is set (ms_share).
template <typename R, typename ST>
__global__ void __launch_bounds__(kBlock, MinBlocks<R>::value)
    k_ms_r_site(Geom g, const ST *__restrict__ U, R m4, MsState *st, MsBatch<ST> v, RedScratch rs, int spb, bool share) {
    MsState *s = st + blockIdx.y;
    if (s->done) return;
    typename SiteSum<R>::type sum[1] = {};
    if (blockIdx.x == 0 && threadIdx.x < 32) ShiftScalars{s}(threadIdx.x);
    if (share || blockIdx.x) {
        const int it = s->iter;
        const ST *__restrict__ p0 = v.p0_at(blockIdx.y, it);
        const ST *__restrict__ t = v.t + blockIdx.y * v.stride;
        const ST *rin = v.r_at(blockIdx.y, it);
        ST *rout = v.r_at(blockIdx.y, it + 1);
        const R ma = HopTiles<R>::minus_alpha(*s), sig0 = HopTiles<R>::sigma0(*s);
        const bool lane_has_sites = threadIdx.x < spb;
        const int first = blockIdx.x - !share, blocks = gridDim.x - !share;
        for (int k = first * spb + threadIdx.x; lane_has_sites && k < g.V; k += blocks * spb) {
            int p, i;
            site_of_thread(k, p, i);
            cpx<R> hop[12], own[12], res[12], pp[12], rv[12];
            wilson_hop<R>(g, U, t, p, i, hop);
            load_spinor<R>(t, g.Vh, p, i, own);
            wilson_combine<R>(m4, own, hop, res);
            apply_g5(res);
            load_spinor<R>(p0, g.Vh, p, i, pp);
            load_spinor<R>(rin, g.Vh, p, i, rv);
            R a0 = 0;
#pragma unroll
            for (int c = 0; c < 12; c++) {
                rv[c] = rv[c] + ma * (res[c] + sig0 * pp[c]);
                a0 += norm2(rv[c]);
            }
            sum_add(sum[0], a0);
            store_spinor<R>(rout, g.Vh, p, i, rv);
        }
    }
    grid_reduce_warp<1>(sum, rs.row(blockIdx.y), ShiftFin{s});
}

// Elementwise arithmetic on storage words: V is a word in registers, C a real coefficient in the
// word's arithmetic, made from its FP64 or its float-float value.
template <typename ST> struct Word;
template <> struct Word<double2> {
    using V = double2;
    using C = double;
    using Sum = double;
    __device__ static void add(Sum &s, double x) { s += x; }
    __device__ static V get(const double2 &w) { return w; }
    __device__ static double2 put(const V &v) { return v; }
    __device__ static C coef(double a, const float *) { return a; }
    __device__ static V fma(C a, const V &b, const V &c) {
        return make_double2(fma_r(a, b.x, c.x), fma_r(a, b.y, c.y));
    }
    __device__ static double norm2(const V &v) { return v.x * v.x + v.y * v.y; }
};
template <> struct Word<float4> {
    using V = float4;
    using C = float;
    using Sum = fsum;
    __device__ static void add(Sum &s, float x) { s.add(x); }
    __device__ static V get(const float4 &w) { return w; }
    __device__ static float4 put(const V &v) { return v; }
    __device__ static C coef(double, const float *f) { return f[0]; }
    __device__ static V fma(C a, const V &b, const V &c) {
        return make_float4(fma_r(a, b.x, c.x), fma_r(a, b.y, c.y), fma_r(a, b.z, c.z), fma_r(a, b.w, c.w));
    }
    __device__ static float norm2(const V &v) { return v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w; }
};
template <> struct Word<ffw> {
    using V = ff2;
    using C = ff2_factor;
    using Sum = ff;
    __device__ static void add(Sum &s, ff x) { s += x; }
    __device__ static V get(const ffw &w) { return ff2_load(reinterpret_cast<const float4 &>(w)); }
    __device__ static ffw put(const V &v) {
        const float4 w = ff2_word(v);
        return ffw{w.x, w.y, w.z, w.w};
    }
    __device__ static C coef(double, const float *f) { return ff2_scale(f[0], f[1]); }
    __device__ static V fma(const C &a, const V &b, const V &c) { return ff2_fma(a, b, c); }
    __device__ static ff norm2(const V &v) {
        return HopTiles<ff>::total(ff2_square_add(v, HopTiles<ff>::zero()));
    }
};

// Coefficients of the pending iterations in shared memory: the base shift's, and the list of the
// other shifts (direction l - 1, number of updates, negative while the shift stays active).
constexpr int kShiftBlocks = 3;
template <typename C>
struct ShiftList {
    C w[kMaxRing][kMaxPoles], b[kMaxRing][kMaxPoles], w0[kMaxRing];
    int idx[kMaxPoles], cnt[kMaxPoles];
    int n;
};

// The updates of NP pending iterations (the last one is iteration it - 1) on this thread's words.
template <int NP, typename ST>
__device__ __forceinline__ void shift_updates(const ShiftList<typename Word<ST>::C> &sl, const MsBatch<ST> &v, int row,
                                              int it, const typename Word<ST>::C &b0, bool go_on) {
    using W = Word<ST>;
    const int na = sl.n;
    const ST *r[NP], *p0[NP];
#pragma unroll
    for (int d = 0; d < NP; d++) {
        r[d] = v.r_at(row, it - NP + 1 + d);
        p0[d] = v.p0_at(row, it - NP + d);
    }
    ST *p0_next = v.p0_at(row, it), *y = v.y + row * v.stride, *P = v.p + row * v.prow;
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < v.stride; k += (long)gridDim.x * blockDim.x) {
        ST rw[NP], pw[NP];
#pragma unroll
        for (int d = 0; d < NP; d++) {
            rw[d] = r[d][k];
            pw[d] = p0[d][k];
        }
        typename W::V rv[NP], yv = W::get(y[k]);
#pragma unroll
        for (int d = 0; d < NP; d++) {
            rv[d] = W::get(rw[d]);
            yv = W::fma(sl.w0[d], W::get(pw[d]), yv);
        }
        if (go_on) p0_next[k] = W::put(W::fma(b0, W::get(pw[NP - 1]), rv[NP - 1]));
        for (int a0 = 0; a0 < na; a0 += 4) {
            ST w[4];
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (a0 + u < na) w[u] = P[(long)sl.idx[a0 + u] * v.stride + k];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                if (a0 + u >= na) break;
                typename W::V pv = W::get(w[u]);
                const int n = sl.cnt[a0 + u], c = n < 0 ? -n : n;
#pragma unroll
                for (int d = 0; d < NP; d++)
                    if (d < c) {
                        yv = W::fma(sl.w[d][a0 + u], pv, yv);
                        pv = W::fma(sl.b[d][a0 + u], pv, rv[d]);
                    }
                if (n < 0) P[(long)sl.idx[a0 + u] * v.stride + k] = W::put(pv);
            }
        }
        y[k] = W::put(yv);
    }
}

// The pending iterations' shift updates of right-hand side blockIdx.y, and p_0 = r_{k+1} + beta p_0.
// One wave of blocks (kShiftBlocks per SM), so that the list is made once per resident block. The shifts that were active in the first of them (later ones' sets are subsets) are compacted into
// a list in shared memory and processed four at a time: the four loads of a batch are issued before
// any store, so each thread keeps four independent memory requests in flight. A shift that has had its
// last update is not written back.
template <typename ST>
__global__ void __launch_bounds__(kBlock, kShiftBlocks) k_ms_shifts(MsState *st, MsBatch<ST> v, unsigned *counters) {
    using W = Word<ST>;
    __shared__ ShiftList<typename W::C> sl;
    const int row = blockIdx.y;
    MsState *s = st + row;
    static_assert(kBlock == kMaxRing * kMaxPoles, "one thread per coefficient");
    const int np = s->npend, it = s->iter;
    if (!np) return;   // uniform over the blocks of this right-hand side
    {
        const int d = threadIdx.x / kMaxPoles, l = threadIdx.x % kMaxPoles;
        const unsigned m0 = s->on[0][0] & ~1u, m1 = s->on[0][1];   // without the base shift
        if (d < np && ((l < 32 ? m0 : m1) >> (l & 31) & 1)) {
            const int k = l < 32 ? __popc(m0 & ((1u << l) - 1)) : __popc(m0) + __popc(m1 & ((1u << (l - 32)) - 1));
            sl.w[d][k] = W::coef(s->wa[d][l], s->wa_f[d][l]);
            sl.b[d][k] = W::coef(s->bl[d][l], s->bl_f[d][l]);
            if (d == 0) {
                int c = 0;
                for (int e = 0; e < np; e++) c += s->on[e][l / 32] >> (l & 31) & 1;
                sl.idx[k] = l - 1;
                sl.cnt[k] = s->active[l] ? -c : c;
            }
        }
        if (threadIdx.x < np) sl.w0[threadIdx.x] = W::coef(s->wa[threadIdx.x][0], s->wa_f[threadIdx.x][0]);
        if (threadIdx.x == 0) sl.n = __popc(m0) + __popc(m1);
    }
    __syncthreads();
    const bool go_on = !s->done;
    const typename W::C b0 = W::coef(s->beta_prev, s->beta_f);
    // the block that arrives last, when all have read the state, clears the pending iterations and ends
    // a finished solve
    if (grid_last_block(counters + row) && threadIdx.x == 0) {
        s->npend = 0;
        if (!go_on && s->done == 2) s->done = 1;
    }
    switch (np) {
        case 1: shift_updates<1>(sl, v, row, it, b0, go_on); break;
        case 2: shift_updates<2>(sl, v, row, it, b0, go_on); break;
        case 3: shift_updates<3>(sl, v, row, it, b0, go_on); break;
        default: shift_updates<4>(sl, v, row, it, b0, go_on); break;
    }
}

// The same with one warp per hop (hops.cuh).
template <typename R, bool OWN>
__global__ void __launch_bounds__(kHopBlock, HopBlocks<R>::value)
    k_ms_q_hops(Geom g, const typename HopTiles<R>::Link *__restrict__ U, R m4, MsState *st,
                MsBatch<typename HopTiles<R>::Store> v, RedScratch rs) {
    using H = HopTiles<R>;
    using E = typename H::Elem;
    MsState *s = st + blockIdx.y;
    if (s->done) return;
    const typename H::Store *__restrict__ p0 = v.p0_at(blockIdx.y, s->iter);
    typename H::Store *__restrict__ t = v.t + blockIdx.y * v.stride;
    typename H::Sum sum = H::zero(), psum = H::zero();
    const auto fm = H::factor(m4);
    const auto own = [&](int p, int i, int it, int e) { return H::load(p0, g.Vh, p, i, it, e); };
    hop_tiles<R>(g, blockIdx.x, gridDim.x, U, p0, own, [&](int p, int i, int it, int e, E hop, int, E o) {
        E w = H::fma(fm, o, hop);
        w = H::neg_if(w, H::upper(it));
        H::store(t, g.Vh, p, i, it, e, w);
        H::square_add(w, sum);
        if (OWN) H::square_add(o, psum);
    });
    if constexpr (OWN) add_shifted(*s, psum, sum);
    const decltype(H::total(sum)) w[1] = {H::total(sum)};
    grid_reduce<1>(w, rs.row(blockIdx.y), AlphaFin<OWN>{s});
}

template <typename R>
__global__ void __launch_bounds__(kHopBlock, HopBlocks<R>::value)
    k_ms_r_hops(Geom g, const typename HopTiles<R>::Link *__restrict__ U, R m4, MsState *st,
                MsBatch<typename HopTiles<R>::Store> v, RedScratch rs, bool share) {
    using H = HopTiles<R>;
    using E = typename H::Elem;
    MsState *s = st + blockIdx.y;
    if (s->done) return;
    const int it0 = s->iter;
    const typename H::Store *__restrict__ p0 = v.p0_at(blockIdx.y, it0);
    const typename H::Store *__restrict__ t = v.t + blockIdx.y * v.stride;
    const typename H::Store *rin = v.r_at(blockIdx.y, it0);
    typename H::Store *rout = v.r_at(blockIdx.y, it0 + 1);
    typename H::Sum sum = H::zero();
    if (blockIdx.x == 0 && threadIdx.x < 32) ShiftScalars{s}(threadIdx.x);
    const int first = share ? blockIdx.x : blockIdx.x ? blockIdx.x - 1 : g.V;   // block 0: past the last tile
    const auto fm = H::factor(m4), fa = H::minus_alpha(*s), fs = H::sigma0(*s);
    struct Own {
        E t, p0, r;
    };
    const auto own = [&](int p, int i, int it, int e) {
        return Own{H::load(t, g.Vh, p, i, it, e), H::load(p0, g.Vh, p, i, it, e), H::load_rw(rin, g.Vh, p, i, it, e)};
    };
    hop_tiles<R>(g, first, gridDim.x - !share, U, t, own, [&](int p, int i, int it, int e, E hop, int, const Own &o) {
        E w = H::fma(fm, o.t, hop);
        w = H::fma(fs, o.p0, H::neg_if(w, H::upper(it)));
        w = H::fma(fa, w, o.r);
        H::store(rout, g.Vh, p, i, it, e, w);
        H::square_add(w, sum);
    });
    const decltype(H::total(sum)) w[1] = {H::total(sum)};
    grid_reduce_warp<1>(w, rs.row(blockIdx.y), ShiftFin{s});
}

// p_0 = r_{k+1} + beta_k p_0 of right-hand side blockIdx.y
template <typename ST>
__global__ void __launch_bounds__(kBlock) k_ms_p0(const MsState *st, MsBatch<ST> v) {
    using W = Word<ST>;
    const MsState *s = st + blockIdx.y;
    if (s->done) return;
    const ST *__restrict__ r = v.r_at(blockIdx.y, s->iter), *__restrict__ p = v.p0_at(blockIdx.y, s->iter - 1);
    ST *__restrict__ o = v.p0_at(blockIdx.y, s->iter);
    const typename W::C b = W::coef(s->beta_prev, s->beta_f);
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < v.stride; k += (long)gridDim.x * blockDim.x)
        o[k] = W::put(W::fma(b, W::get(p[k]), W::get(r[k])));
}

struct InitFin {
    MsState *s;
    __device__ int before() const { return 0; }
    __device__ void operator()(const double *v, int) const {
        s->bb = v[0];
        s->rr = v[0];
        s->pp = v[0];   // p_0 = b
        if (v[0] == 0.0) s->done = 1;
        if (!isfinite(v[0])) {
            s->status = 1;
            s->done = 1;
        }
    }
};

// r = y = p_l = b ; ||b||^2 of right-hand side blockIdx.y (b: vectors v.stride words apart). One that
// needs no work (done already set) is left out: its b is a vector that its solver never wrote, and a NaN
// in it would count as a breakdown of the whole batch.
template <typename ST>
__global__ void k_ms_init(MsState *st, const ST *__restrict__ b, MsBatch<ST> v, RedScratch rs) {
    using W = Word<ST>;
    MsState *s = st + blockIdx.y;
    if (s->done) return;   // uniform over the blocks of this right-hand side: only the last to arrive sets it
    b += blockIdx.y * v.stride;
    ST *r = v.r_at(blockIdx.y, 0), *p0 = v.p0_at(blockIdx.y, 0), *y = v.y + blockIdx.y * v.stride;
    ST *P = v.p + blockIdx.y * v.prow;
    const int n = s->n;
    typename W::Sum sum{};
    for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < v.stride; k += (long)gridDim.x * blockDim.x) {
        const ST w = b[k];
        r[k] = w;
        y[k] = w;
        p0[k] = w;
        for (int l = 1; l < n; l++) P[(l - 1) * v.stride + k] = w;
        W::add(sum, W::norm2(W::get(w)));
    }
    const typename W::Sum total[1] = {sum};
    grid_reduce<1>(total, rs.row(blockIdx.y), InitFin{s});
}

inline int stream_grid(long n) {
    long b = (n + kBlock - 1) / kBlock;
    const long cap = 152L * 16;
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

// ---- 16-bit shifted directions (one thread per site: the FP16 words share a norm)
// Shift updates of one iteration (ring 1), with p_0 in FP32 and p_l (l >= 1) in FP16 with a per-site
// scale (BF = false) or in BF16 (BF = true).
template <bool BF>
__device__ __forceinline__ void load_p16(const MsVectorsH &v, int l, int Vh, int p, int i, cpx<float> pv[12]) {
    if (BF) load_spinor<float>(Bf16SpinorC{v.ph + (size_t)(l - 1) * v.words_h}, Vh, p, i, pv);
    else load_spinor<float>(HalfSpinorC{v.ph + (size_t)(l - 1) * v.words_h, v.pn + (size_t)(l - 1) * 2 * Vh}, Vh, p,
                            i, pv);
}
template <bool BF>
__device__ __forceinline__ void store_p16(const MsVectorsH &v, int l, int Vh, int p, int i, const cpx<float> pv[12]) {
    if (BF) store_spinor<float>(Bf16Spinor{v.ph + (size_t)(l - 1) * v.words_h}, Vh, p, i, pv);
    else store_spinor<float>(HalfSpinor{v.ph + (size_t)(l - 1) * v.words_h, v.pn + (size_t)(l - 1) * 2 * Vh}, Vh, p,
                             i, pv);
}

template <bool BF>
__global__ void __launch_bounds__(kBlock) k_ms_shifts_half(Geom g, MsState *s, MsVectorsH v, unsigned *counter) {
    __shared__ float sw[kMaxPoles], sb[kMaxPoles];
    __shared__ int sidx[kMaxPoles];
    __shared__ int sact;
    if (threadIdx.x == 0) {
        int na = 0;
        if (s->npend)
            for (int l = 0; l < s->n; l++)
                if (s->on[0][l / 32] >> (l & 31) & 1) {
                    sidx[na] = l;
                    sw[na] = (float)s->wa[0][l];
                    sb[na] = (float)s->bl[0][l];
                    na++;
                }
        sact = na;
    }
    __syncthreads();
    const int na = sact;
    if (!na) return;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < g.V; k += gridDim.x * blockDim.x) {
        const int p = k >= g.Vh, i = k - p * g.Vh;   // no neighbours: plain parity-major order
        cpx<float> rv[12], yv[12], pv[12];
        load_spinor<float>(v.r, g.Vh, p, i, rv);
        load_spinor<float>(v.y, g.Vh, p, i, yv);
        for (int a = 0; a < na; a++) {
            const int l = sidx[a];
            const float wl = sw[a], bl = sb[a];
            if (l == 0) load_spinor<float>(v.p0, g.Vh, p, i, pv);
            else load_p16<BF>(v, l, g.Vh, p, i, pv);
#pragma unroll
            for (int c = 0; c < 12; c++) {
                yv[c] = yv[c] + wl * pv[c];
                pv[c] = rv[c] + bl * pv[c];
            }
            if (l == 0) store_spinor<float>(v.p0, g.Vh, p, i, pv);
            else store_p16<BF>(v, l, g.Vh, p, i, pv);
        }
        store_spinor<float>(v.y, g.Vh, p, i, yv);
    }
    if (grid_last_block(counter) && threadIdx.x == 0) {
        s->npend = 0;
        if (s->done == 2) s->done = 1;
    }
}

// r = y = p_0 = b in FP32, p_l = b in FP16 or BF16 (l >= 1) ; ||b||^2
template <bool BF>
__global__ void k_ms_init_half(Geom g, MsState *s, MsVectorsH v, const float4 *__restrict__ b, int n, RedScratch rs) {
    float acc[1] = {0.f};
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < g.V; k += gridDim.x * blockDim.x) {
        const int p = k >= g.Vh, i = k - p * g.Vh;
        cpx<float> bv[12];
        load_spinor<float>(b, g.Vh, p, i, bv);
        store_spinor<float>(v.r, g.Vh, p, i, bv);
        store_spinor<float>(v.y, g.Vh, p, i, bv);
        store_spinor<float>(v.p0, g.Vh, p, i, bv);
        for (int l = 1; l < n; l++) store_p16<BF>(v, l, g.Vh, p, i, bv);
        float a = 0.f;
#pragma unroll
        for (int c = 0; c < 12; c++) a += norm2(bv[c]);
        acc[0] += a;
    }
    grid_reduce<1>(acc, rs, InitFin{s});
}

// The third kernel of an iteration: the shift updates where `flush`, else p_0 alone.
template <typename ST>
cudaError_t ms_third(const Geom &g, MsRows nrhs, MsState *s, const MsBatch<ST> &v, unsigned *counters, bool flush,
                     cudaStream_t st) {
    const int want = stream_grid(v.stride);
    if (flush)
        k_ms_shifts<ST><<<dim3(std::max(1, std::min(want, kShiftBlocks * g.nsm / nrhs.of)), nrhs.n), kBlock, 0, st>>>(s, v,
                                                                                                      counters);
    else k_ms_p0<ST><<<dim3(std::max(1, std::min(want, 16 * g.nsm / nrhs.of)), nrhs.n), kBlock, 0, st>>>(s, v);
    return cudaGetLastError();
}

// Whether block 0 of a residual kernel takes its share of a row's `turns` per block after the shift
// scalars (3 us) instead of none: a batch has few blocks a row (38 of 456 for 12 right-hand sides in FP64, 25 of
// 304 in FP32), and one without work costs as much as the row's 1/blocks. A turn takes 4 to 12 us, so the
// line is safely where a block has as many turns as there are blocks.
inline bool ms_share(long turns, int blocks) { return turns >= blocks; }

// One iteration of nrhs right-hand sides, one warp per hop.
template <typename R, typename LT, typename ST>
cudaError_t ms_stencils_hops(const Geom &g, const LT *U, double m0, MsRows nrhs, MsState *s, const MsBatch<ST> &v,
                             const RedScratch &rows, cudaStream_t st, const MsEvents &ev) {
    const int gx = hop_grid<R>(g, nrhs.of, true);
    cudaError_t e;
    if ((e = ev.record(0, st)) != cudaSuccess) return e;
    if (nrhs.of > 1 && !std::is_same<R, ff>::value)
        k_ms_q_hops<R, !std::is_same<R, ff>::value><<<dim3(gx, nrhs.n), kHopBlock, 0, st>>>(g, U, R(m0 + 4.0), s, v, rows);
    else k_ms_q_hops<R, false><<<dim3(gx, nrhs.n), kHopBlock, 0, st>>>(g, U, R(m0 + 4.0), s, v, rows);
    if ((e = ev.record(1, st)) != cudaSuccess) return e;
    // one block more for the shift scalars, within the wave
    const bool full = (long)gx * nrhs.of + nrhs.of > (long)g.nsm * HopBlocks<R>::value && gx > 1;
    const bool share = full && ms_share(hop_grid<R>(g, 1, false) / gx, gx);
    k_ms_r_hops<R><<<dim3(full ? gx : gx + 1, nrhs.n), kHopBlock, 0, st>>>(g, U, R(m0 + 4.0), s, v, rows, share);
    return ev.record(2, st);
}
// One thread per site, in FP32 and for one right-hand side in FP64 (ms_fp64_per_site). FP32: one wave of
// blocks that stride over the sites (at 32^4 thirteen waves, each block ending with a fence and an atomic,
// cost 20 us of 125; the whole FP32 sign at 32^4 14.67 ms, with the order of site_of_thread 14.17).
// FP64, ten times as long a site: as many blocks as the reduction's scratch holds, which even out what
// a last wave leaves.
template <typename R, typename ST>
cudaError_t ms_stencils_site(const Geom &g, const ST *U, R m0, MsRows nrhs, MsState *s, const MsBatch<ST> &v,
                             const RedScratch &rows, cudaStream_t st, const MsEvents &ev) {
    constexpr bool fp64 = std::is_same<R, double>::value;
    const int slots = std::max(1, g.nsm * MinBlocks<R>::value / nrhs.of);   // resident blocks of a row
    const LaunchShape q = fp64 ? balanced_shape(g.V, slots, 1, kMaxRedBlocks - 1) : balanced_shape(g.V, slots, 1, slots);
    const bool share = !fp64 && ms_share(g.V / (slots * kBlock), slots);
    const LaunchShape r = fp64 || share ? q : balanced_shape(g.V, std::max(1, slots - 1), 1, std::max(1, slots - 1));
    cudaError_t e;
    if ((e = ev.record(0, st)) != cudaSuccess) return e;
    if (!fp64 && nrhs.of > 1)
        k_ms_q_site<R, !fp64><<<dim3(q.grid, nrhs.n), q.block, 0, st>>>(g, U, m0 + (R)4, s, v, rows, q.spb);
    else k_ms_q_site<R, false><<<dim3(q.grid, nrhs.n), q.block, 0, st>>>(g, U, m0 + (R)4, s, v, rows, q.spb);
    if ((e = ev.record(1, st)) != cudaSuccess) return e;
    k_ms_r_site<R><<<dim3(r.grid + !share, nrhs.n), r.block, 0, st>>>(g, U, m0 + (R)4, s, v, rows, r.spb, share);
    return ev.record(2, st);
}
// FP64: one warp per hop, or on large lattices one thread per site. The whole sign (ms) with the one and
// the other: 24^4 126.4 / 127.9, 30^4 304.9 / 313.7, 32^4 394.8 / 382.3, 48 x 32^3 590.9 / 582.9, 64 x 32^3
// 894.9 / 872.3, 40^4 1063 / 1039; in batches, which have fewer blocks a row, 2 at 24^4 253.8 / 265.0, 8
// at 24^4 1018 / 1059, 2 at 32^4 787 / 778.
inline bool ms_fp64_per_site(const Geom &g, MsRows nrhs) { return nrhs.of == 1 && g.V >= 1 << 20; }

template <typename R, typename LT, typename ST>
cudaError_t ms_iter_t(const Geom &g, const LT *U, double m0, MsRows nrhs, MsState *s, MsBatch<ST> v, RedScratch rs,
                      unsigned *counters, bool flush, cudaStream_t st, const MsEvents &ev) {
    const RedScratch rows{rs.partials, counters};
    cudaError_t e;
    bool per_site = false;
    if constexpr (!std::is_same<R, ff>::value) {
        per_site = sizeof(R) == 4 ? g.tps32 != 4 : ms_fp64_per_site(g, nrhs);
        if (per_site) e = ms_stencils_site<R>(g, U, (R)m0, nrhs, s, v, rows, st, ev);
    }
    if (!per_site) e = ms_stencils_hops<R>(g, U, m0, nrhs, s, v, rows, st, ev);
    if (e != cudaSuccess || (e = ms_third(g, nrhs, s, v, counters, flush, st)) != cudaSuccess ||
        (e = ev.record(3, st)) != cudaSuccess)
        return e;
    count_launches(3);
    return cudaGetLastError();
}
template <typename ST>
cudaError_t ms_init_t(MsRows nrhs, MsState *s, const MsBatch<ST> &v, const ST *b, RedScratch rs, unsigned *counters,
                      cudaStream_t st) {
    const int gx = std::max(1, red_grid(v.stride) / nrhs.of);
    k_ms_init<ST><<<dim3(gx, nrhs.n), kBlock, 0, st>>>(s, b, v, RedScratch{rs.partials, counters});
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace

cudaError_t ms_init(const Geom &g, MsRows nrhs, MsState *s, MsBatch<double2> v, const double2 *b, RedScratch rs,
                    unsigned *counters, cudaStream_t st) {
    return ms_init_t(nrhs, s, v, b, rs, counters, st);
}
cudaError_t ms_init(const Geom &g, MsRows nrhs, MsState *s, MsBatch<float4> v, const float4 *b, RedScratch rs,
                    unsigned *counters, cudaStream_t st) {
    return ms_init_t(nrhs, s, v, b, rs, counters, st);
}
cudaError_t ms_init(const Geom &g, MsRows nrhs, MsState *s, MsBatch<ffw> v, const ffw *b, RedScratch rs,
                    unsigned *counters, cudaStream_t st) {
    return ms_init_t(nrhs, s, v, b, rs, counters, st);
}
cudaError_t ms_iter(const Geom &g, const double2 *U, double m0, MsRows nrhs, MsState *s, MsBatch<double2> v, RedScratch rs,
                    unsigned *counters, bool flush, cudaStream_t st, const MsEvents &ev) {
    return ms_iter_t<double>(g, U, m0, nrhs, s, v, rs, counters, flush, st, ev);
}
cudaError_t ms_iter(const Geom &g, const float4 *U, double m0, MsRows nrhs, MsState *s, MsBatch<float4> v, RedScratch rs,
                    unsigned *counters, bool flush, cudaStream_t st, const MsEvents &ev) {
    return ms_iter_t<float>(g, U, m0, nrhs, s, v, rs, counters, flush, st, ev);
}
// float-float: the scalar recurrences stay FP64 on the device
cudaError_t ms_iter(const Geom &g, const ffl *U, double m0, MsRows nrhs, MsState *s, MsBatch<ffw> v, RedScratch rs,
                    unsigned *counters, bool flush, cudaStream_t st, const MsEvents &ev) {
    return ms_iter_t<ff>(g, U, m0, nrhs, s, v, rs, counters, flush, st, ev);
}

}  // namespace ovl

namespace ovl {
cudaError_t ms_init_half(const Geom &g, int n, MsState *s, MsVectorsH v, const float4 *b, RedScratch rs, bool bf16,
                         cudaStream_t st) {
    if (bf16) k_ms_init_half<true><<<red_grid(g.V), kBlock, 0, st>>>(g, s, v, b, n, rs);
    else k_ms_init_half<false><<<red_grid(g.V), kBlock, 0, st>>>(g, s, v, b, n, rs);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t ms_iter_half(const Geom &g, const float4 *U, double m0, MsState *s, MsVectorsH v, RedScratch rs, bool bf16,
                         cudaStream_t st, const MsEvents &ev) {
    const MsBatch<float4> w{v.r, v.p0, v.t, v.y, nullptr, v.words, 0, 1};
    cudaError_t e = ms_stencils_site<float>(g, U, (float)m0, 1, s, w, RedScratch{rs.partials, rs.counter}, st, ev);
    if (e != cudaSuccess) return e;
    const int gsh = balanced_shape(g.V, g.nsm, 2, 1 << 30).grid;
    if (bf16) k_ms_shifts_half<true><<<gsh, kBlock, 0, st>>>(g, s, v, rs.counter);
    else k_ms_shifts_half<false><<<gsh, kBlock, 0, st>>>(g, s, v, rs.counter);
    if ((e = ev.record(3, st)) != cudaSuccess) return e;
    count_launches(3);
    return cudaGetLastError();
}
}  // namespace ovl
