// Schwarz alternating procedure (SAP) for the Wilson-Dirac operator D_W(m0):
// the smoother of the inexact Wilson preconditioner.
//
// The paper preconditions with D_W(m0_prec)^{-1} applied inexactly (Sec. 5.1) by
// DD-alpha-AMG, whose smoother is a red-black multiplicative Schwarz method. Here the
// Schwarz method itself preconditions a short flexible GMRES on D_W(m0_prec):
//
//   blocks: the lattice is cut into blocks of b0 x b1 x b2 x b3 sites, coloured by the
//           parity of the block coordinates (red-black over blocks);
//   one cycle, x <- x + sum over colour c of the block corrections:
//       r = v - D_W x                       (full-lattice stencil)
//       for every block B of colour c: solve D_BB e_B = r_B approximately,
//       x_B += e_B
//   where D_BB is D_W restricted to the block (hops leaving the block dropped).
//
// Block solve: a fixed number of minimal-residual steps, one CTA per block, the block's residual
// and links held in shared memory:
//   e = 0, s = r_B;  repeat:  q = D_BB s,  alpha = <q, s>/<q, q>,  e += alpha s,  s -= alpha q.
// FP64: one thread per block site; FP32: two (k_sap_block32).
#include "internal.h"
#include "reduce.cuh"
#include "sap.h"
#include "wilson_site.cuh"

namespace ovl {

namespace {

// FP64: shared-memory copies of a block's spinor and forward links in the word layouts of global
// memory, spinor double2 [12][nb] and links double2 [4][9][nb]: consecutive threads read
// consecutive words (no bank conflicts).
constexpr int kSapSpinor64 = 12, kSapLink64 = 9;
__device__ __forceinline__ void sm_load_sp(const double2 *s, int nb, int t, cpx<double> v[12]) {
#pragma unroll
    for (int c = 0; c < 12; c++) {
        const double2 w = s[c * nb + t];
        v[c] = cpx<double>{w.x, w.y};
    }
}
__device__ __forceinline__ void sm_store_sp(double2 *s, int nb, int t, const cpx<double> v[12]) {
#pragma unroll
    for (int c = 0; c < 12; c++) s[c * nb + t] = make_double2(v[c].re, v[c].im);
}
__device__ __forceinline__ void sm_load_link(const double2 *u, int nb, int mu, int t, cpx<double> m[3][3]) {
    const double2 *b = u + mu * 9 * nb + t;
#pragma unroll
    for (int c = 0; c < 9; c++) {
        const double2 w = b[c * nb];
        m[c / 3][c % 3] = cpx<double>{w.x, w.y};
    }
}
// The link words of U_mu at (p, i) in global memory, copied to block site t.
__device__ __forceinline__ void sm_copy_link(double2 *u, int nb, int mu, int t, const double2 *__restrict__ U, int Vh,
                                             int p, int i) {
    constexpr int W = kSapLink64;
    const double2 *gw = U + ((size_t)(p * 4 + mu) * W) * Vh + i;
#pragma unroll
    for (int c = 0; c < W; c++) u[(mu * W + c) * nb + t] = __ldg(gw + (size_t)c * Vh);
}

// q = D_BB s at local site t (local coords l, extents bx), links of the block in smem.
template <typename R, typename LT, typename ST>
__device__ __forceinline__ void block_apply(const ST *s, const LT *u, int nb, int t, const int l[4], const int bx[4],
                                            const int stride[4], R m4, cpx<R> q[12]) {
    cpx<R> acc[12];
#pragma unroll
    for (int c = 0; c < 12; c++) acc[c] = cpx<R>{0, 0};
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        if (l[mu] + 1 < bx[mu]) {
            cpx<R> v[12], h0[3], h1[3], a0[3], a1[3], m[3][3];
            sm_load_sp(s, nb, t + stride[mu], v);
            sm_load_link(u, nb, mu, t, m);
            proj_fwd(mu, v, h0, h1);
            su3_mul(m, h0, a0);
            su3_mul(m, h1, a1);
            acc_fwd<false>(mu, acc, a0, a1);
        }
        if (l[mu] > 0) {
            cpx<R> v[12], h0[3], h1[3], a0[3], a1[3], m[3][3];
            sm_load_sp(s, nb, t - stride[mu], v);
            sm_load_link(u, nb, mu, t - stride[mu], m);
            proj_bwd(mu, v, h0, h1);
            su3_dag_mul(m, h0, a0);
            su3_dag_mul(m, h1, a1);
            acc_bwd(mu, acc, a0, a1);
        }
    }
    cpx<R> own[12];
    sm_load_sp(s, nb, t, own);
    wilson_combine<R>(m4, own, acc, q);
}

// MR step of a block solve: the block sums of Re<q, s>, Im<q, s> and |q|^2 (per warp by
// shuffles, then over warps in a fixed order by thread 0, all in R) and alpha = <q, s>/|q|^2,
// computed once by thread 0 and broadcast. Returns false when |q|^2 is not positive
// (uniform over the CTA). Every thread of the CTA must call it.
template <typename R>
__device__ __forceinline__ bool mr_alpha(R a0, R a1, R a2, cpx<R> &alpha) {
    __shared__ R red[3][32];
    __shared__ R bc[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a0 += __shfl_down_sync(0xffffffffu, a0, off);
        a1 += __shfl_down_sync(0xffffffffu, a1, off);
        a2 += __shfl_down_sync(0xffffffffu, a2, off);
    }
    if (lane == 0) {
        red[0][warp] = a0;
        red[1][warp] = a1;
        red[2][warp] = a2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        R s0 = 0, s1 = 0, s2 = 0;
        for (int w = 0; w < nw; w++) {
            s0 += red[0][w];
            s1 += red[1][w];
            s2 += red[2][w];
        }
        const bool ok = s2 > (R)0;
        bc[0] = ok ? s0 / s2 : (R)0;
        bc[1] = ok ? s1 / s2 : (R)0;
        bc[2] = ok ? (R)1 : (R)0;
    }
    __syncthreads();
    alpha = cpx<R>{bc[0], bc[1]};
    return bc[2] > (R)0;
}

// One CTA per block of the given colour.
//   RES = false: the block residual is r_B = v_B (x = 0 everywhere before this sweep);
//   RES = true:  r_B = v_B - (D_W x)_B is formed here from global x (own sites and the
//                neighbours across the block faces, which have the other colour and are
//                not written during this launch).
// colour_grid = true: the grid holds only the blocks of this colour (blocks per direction
// all even); otherwise it holds all blocks and the other colour's CTAs return at once.
template <typename R, typename LT, typename ST, bool RES>
__global__ void __launch_bounds__(kBlock, 1) k_sap_block(Geom g, SapGeom sg, const LT *__restrict__ U, const ST *__restrict__ v, ST *x, R m4,
                            int colour, int mr_iters, bool colour_grid) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nb = sg.nb;
    // block coordinates of this CTA
    int B[4], rem = blockIdx.x;
    if (colour_grid) {
        const int h3 = sg.nblk[3] / 2;
        const int b3h = rem % h3; rem /= h3;
        B[2] = rem % sg.nblk[2]; rem /= sg.nblk[2];
        B[1] = rem % sg.nblk[1];
        B[0] = rem / sg.nblk[1];
        B[3] = 2 * b3h + ((B[0] + B[1] + B[2] + colour) & 1);
    } else {
        B[3] = rem % sg.nblk[3]; rem /= sg.nblk[3];
        B[2] = rem % sg.nblk[2]; rem /= sg.nblk[2];
        B[1] = rem % sg.nblk[1];
        B[0] = rem / sg.nblk[1];
        if (((B[0] + B[1] + B[2] + B[3]) & 1) != colour) return;   // uniform over the CTA
    }
    ST *s = reinterpret_cast<ST *>(smem_raw);
    LT *u = reinterpret_cast<LT *>(s + kSapSpinor64 * nb);
    // the CTA is padded to whole warps; threads t >= nb hold no site but join the reductions
    const bool act = threadIdx.x < nb;
    const int t = act ? threadIdx.x : 0;
    int l[4], rr = t;
    l[3] = rr % sg.b[3]; rr /= sg.b[3];
    l[2] = rr % sg.b[2]; rr /= sg.b[2];
    l[1] = rr % sg.b[1];
    l[0] = rr / sg.b[1];
    int xg[4];
#pragma unroll
    for (int mu = 0; mu < 4; mu++) xg[mu] = B[mu] * sg.b[mu] + l[mu];
    const int p = (xg[0] + xg[1] + xg[2] + xg[3]) & 1;
    const int i = eo_index(g, xg);
    // links U_mu(x) of the block sites (forward links; backward ones are the neighbours')
    if (act)
#pragma unroll
        for (int mu = 0; mu < 4; mu++) sm_copy_link(u, nb, mu, t, U, g.Vh, p, i);
    cpx<R> res[12], e[12], q[12];
#pragma unroll
    for (int c = 0; c < 12; c++) {
        e[c] = cpx<R>{0, 0};
        res[c] = cpx<R>{0, 0};
        q[c] = cpx<R>{0, 0};
    }
    if (act) {
        load_spinor<R>(v, g.Vh, p, i, res);
        if (RES) {   // res = v - D_W x at this site
            cpx<R> hop[12], own[12], dx[12];
            wilson_hop<R>(g, U, x, p, i, hop);
            load_spinor<R>(x, g.Vh, p, i, own);
            wilson_combine<R>(m4, own, hop, dx);
#pragma unroll
            for (int c = 0; c < 12; c++) res[c] = res[c] - dx[c];
        }
    }
    for (int it = 0; it < mr_iters; it++) {
        if (act) sm_store_sp(s, nb, t, res);
        __syncthreads();
        if (act) block_apply<R, LT, ST>(s, u, nb, t, l, sg.b, sg.stride, m4, q);
        R a0 = 0, a1 = 0, a2 = 0;   // per-site and block sums in the arithmetic type
#pragma unroll
        for (int c = 0; c < 12; c++) {
            a0 += q[c].re * res[c].re + q[c].im * res[c].im;   // Re <q, s>
            a1 += q[c].re * res[c].im - q[c].im * res[c].re;   // Im <q, s>
            a2 += norm2(q[c]);
        }
        cpx<R> alpha;
        if (!mr_alpha<R>(a0, a1, a2, alpha)) break;   // uniform over the CTA
#pragma unroll
        for (int c = 0; c < 12; c++) {
            e[c] = e[c] + alpha * res[c];
            res[c] = res[c] - alpha * q[c];
        }
    }
    __syncthreads();   // every thread of the CTA has finished reading x before any writes it
    if (!act) return;
    cpx<R> xv[12];
    load_spinor<R>(x, g.Vh, p, i, xv);
#pragma unroll
    for (int c = 0; c < 12; c++) xv[c] = xv[c] + e[c];
    store_spinor<R>(x, g.Vh, p, i, xv);
}

// ---------------------------------------------------------------------------------
// FP32: two threads per block site. Lanes 0-15 of a warp hold spins 0 and 2 of 16 sites, lanes
// 16-31 spins 1 and 3: thread k forms component k of each projected half spinor, multiplies it by
// the link and adds it to its upper spin; the lower spins get +-1 or +-i times the two components,
// in place for directions 0 and 3 and crossed for 1 and 2, so one exchange between the two lanes
// of a site at the end of the eight hops completes them.
//
// Bound: shared memory, 8 x (48 B spinor + 72 B link / 2) of reads per thread and MR step (4^4:
// 2700 clocks a step at 128 B per clock); the links are kept as all 18 reals, since rebuilding the
// third row in every step costs more issue slots than the 24 B cost bandwidth, and the two lanes of
// a site read the same words. One thread per site left an SM with eight warps, bound by latency, and
// two or four threads per site by direction moved all partial sums through shared memory. One colour
// of 4^4 blocks with 6 MR steps at 16^4 (128 CTAs), best of the three forms -> this one: 28.8 -> 23.9
// us from a given residual, 34.0 -> 32.1 (27.3 with x = 0 on the colour) with the residual formed in
// the kernel. Right-hand sides of a batch are grid rows: four at 16 x 8^3 (16 blocks per colour) took
// four launches of 28 us and now take one. Spins are stored as (colour 0, colour 1) and colour 2, so that a
// spin takes one 16-byte and one 8-byte access.
// Rows are S sites long whatever the block's size (64 or 256), so that all offsets are constants:
// address arithmetic was a tenth of the instructions.
template <int S>
struct Sap32 {
    float4 uA[16][S];   // [4 mu][4] entries 0-7 of the link, row by row, two to a word
    float4 sA[4][S];    // [4 spins] colours 0 and 1
    float2 uB[4][S];    // [4 mu] entry 8
    float2 sB[4][S];    // [4 spins] colour 2
};

template <int S>
__device__ __forceinline__ void sap_spin(const Sap32<S> &m, int spin, int t, cpx<float> v[3]) {
    const float4 a = m.sA[spin][t];
    const float2 b = m.sB[spin][t];
    v[0] = cpx<float>{a.x, a.y};
    v[1] = cpx<float>{a.z, a.w};
    v[2] = cpx<float>{b.x, b.y};
}
template <int S>
__device__ __forceinline__ void sap_put_spin(Sap32<S> &m, int spin, int t, const cpx<float> v[3]) {
    m.sA[spin][t] = make_float4(v[0].re, v[0].im, v[1].re, v[1].im);
    m.sB[spin][t] = make_float2(v[2].re, v[2].im);
}
template <int S>
__device__ __forceinline__ void sap_link(const Sap32<S> &m, int mu, int t, cpx<float> u[3][3]) {
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const float4 w = m.uA[4 * mu + c][t];
        u[(2 * c) / 3][(2 * c) % 3] = cpx<float>{w.x, w.y};
        u[(2 * c + 1) / 3][(2 * c + 1) % 3] = cpx<float>{w.z, w.w};
    }
    const float2 w = m.uB[mu][t];
    u[2][2] = cpx<float>{w.x, w.y};
}
// One spin of site (p, i) of an FP32 spinor in global memory: complex numbers 3 spin .. 3 spin + 2,
// three halves of two words.
__device__ __forceinline__ void glob_spin(const float4 *f, int Vh, int p, int i, int spin, cpx<float> v[3]) {
    const float4 *b = f + (size_t)(p * 6 + 3 * (spin >> 1) + (spin & 1)) * Vh + i;
    const float4 a = b[0], d = b[Vh];
    v[0] = spin & 1 ? cpx<float>{a.z, a.w} : cpx<float>{a.x, a.y};
    v[1] = spin & 1 ? cpx<float>{d.x, d.y} : cpx<float>{a.z, a.w};
    v[2] = spin & 1 ? cpx<float>{d.z, d.w} : cpx<float>{d.x, d.y};
}
__device__ __forceinline__ void glob_put_spin(float4 *f, int Vh, int p, int i, int spin, const cpx<float> v[3]) {
    float2 *f2 = reinterpret_cast<float2 *>(f);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const int w = 3 * spin + c;
        f2[2 * ((size_t)(p * 6 + w / 2) * Vh + i) + (w & 1)] = make_float2(v[c].re, v[c].im);
    }
}

// The hop from a neighbour whose spins k and 2 + k or 3 - k are (up, low), with link u (of the site
// for FWD, of the neighbour otherwise): added, times weight (0 or 1), to the upper spin, and to the
// lower spin of this thread (in place) or of the other one (crossed).
template <int MU, bool FWD>
__device__ __forceinline__ void sap_hop(const cpx<float> up[3], const cpx<float> low[3], const cpx<float> u[3][3], int k,
                                        bool flip, float weight, cpx<float> au[3], cpx<float> al[3]) {
    constexpr bool turn = MU == 1 || MU == 3;
    // h = up + c low with c = +-1 or +-i: its sign, the same for both lanes of a site in directions
    // 0 and 1, opposite in 2 and 3 (a factor of a fused multiply-add there instead of sign flips)
    const float sg = (MU == 0 ? -1.f : MU == 1 || !k ? 1.f : -1.f) * (FWD ? 1.f : -1.f);
    const float sw = sg * weight;
    cpx<float> h[3], a[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        h[c].re = up[c].re + (turn ? -sg * low[c].im : sg * low[c].re);
        h[c].im = up[c].im + (turn ? sg * low[c].re : sg * low[c].im);
        if (MU == 0) h[c] = cpx<float>{flip_sign(h[c].re, flip), flip_sign(h[c].im, flip)};
    }
    if (FWD) su3_mul(u, h, a);
    else su3_dag_mul(u, h, a);
#pragma unroll
    for (int c = 0; c < 3; c++) {   // lower spin: conj(c) a
        au[c].re += weight * a[c].re;
        au[c].im += weight * a[c].im;
        al[c].re += turn ? sw * a[c].im : sw * a[c].re;
        al[c].im += turn ? -sw * a[c].re : sw * a[c].im;
    }
}

// Lower spins: the crossed sums of the site's other lane added to this one's.
__device__ __forceinline__ void sap_exchange(cpx<float> al[3], const cpx<float> ax[3]) {
#pragma unroll
    for (int c = 0; c < 3; c++) {
        al[c].re += __shfl_xor_sync(0xffffffffu, ax[c].re, 16);
        al[c].im += __shfl_xor_sync(0xffffffffu, ax[c].im, 16);
    }
}

template <int MU, int S>
__device__ __forceinline__ void sap_block_dir(const Sap32<S> &m, int t, int k, const int l[4], const SapGeom &sg,
                                              cpx<float> au[3], cpx<float> al[3]) {
    const int low_spin = MU == 0 || MU == 3 ? 2 + k : 3 - k;
    cpx<float> up[3], low[3], u[3][3];
    // x0 and x1 are mostly the same in a warp, whose 16 sites are consecutive: a hop that leaves the
    // block is skipped. Along x2 and x3 some lanes of every warp have the hop, so it is done without
    // a branch, with weight 0 where it leaves: the loads of the next hops then overlap with it.
    const bool fwd = l[MU] + 1 < sg.b[MU], bwd = l[MU] > 0;
    if (MU >= 2 || fwd) {
        const int n = MU < 2 || fwd ? t + sg.stride[MU] : t;
        sap_spin(m, k, n, up);
        sap_spin(m, low_spin, n, low);
        sap_link(m, MU, t, u);
        sap_hop<MU, true>(up, low, u, k, false, MU < 2 || fwd ? 1.f : 0.f, au, al);
    }
    if (MU >= 2 || bwd) {
        const int n = MU < 2 || bwd ? t - sg.stride[MU] : t;
        sap_spin(m, k, n, up);
        sap_spin(m, low_spin, n, low);
        sap_link(m, MU, n, u);
        sap_hop<MU, false>(up, low, u, k, false, MU < 2 || bwd ? 1.f : 0.f, au, al);
    }
}

// Hops of the global field x at a block site; OUT: only those that leave the block.
template <int MU, bool OUT, int S>
__device__ __forceinline__ void sap_glob_dir(const Geom &g, const Sap32<S> &m, const float4 *__restrict__ U, const float4 *x,
                                             int p, const int xg[4], int t, int k, const int l[4], const SapGeom &sg,
                                             cpx<float> au[3], cpx<float> al[3]) {
    const int low_spin = MU == 0 || MU == 3 ? 2 + k : 3 - k;
    cpx<float> up[3], low[3], u[3][3];
    int y[4] = {xg[0], xg[1], xg[2], xg[3]};
    if (!OUT || l[MU] + 1 == sg.b[MU]) {
        y[MU] = xg[MU] + 1 == g.L[MU] ? 0 : xg[MU] + 1;
        const int j = eo_index(g, y);
        glob_spin(x, g.Vh, 1 - p, j, k, up);
        glob_spin(x, g.Vh, 1 - p, j, low_spin, low);
        sap_link(m, MU, t, u);
        sap_hop<MU, true>(up, low, u, k, g.antiperiodic && xg[0] == g.L[0] - 1, 1.f, au, al);
    }
    if (!OUT || l[MU] == 0) {
        y[MU] = xg[MU] == 0 ? g.L[MU] - 1 : xg[MU] - 1;
        const int j = eo_index(g, y);
        glob_spin(x, g.Vh, 1 - p, j, k, up);
        glob_spin(x, g.Vh, 1 - p, j, low_spin, low);
        if (l[MU] == 0) load_link<float>(U, g.Vh, 1 - p, MU, j, u);
        else sap_link(m, MU, t - sg.stride[MU], u);
        sap_hop<MU, false>(up, low, u, k, g.antiperiodic && xg[0] == 0, 1.f, au, al);
    }
}

// What is known of x before a block solve: the residual is v itself, v minus the hops from the
// neighbouring blocks (the block's own x is zero and is assigned), or v - D_W x.
enum SapStart { kSapFresh, kSapOwnZero, kSapFull };

// One CTA per block of the colour and right-hand side; ADD: x += e instead of x = e.
template <int S, int START, bool ADD>
__global__ void __launch_bounds__(2 * S, 1)
    k_sap_block32(Geom g, SapGeom sg, const float4 *__restrict__ U, const float4 *__restrict__ v, float4 *x, long stride,
                  RowList rows, float m4, int colour, int mr_iters, bool colour_grid) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float4 red[2 * kBlock / 32];
    int B[4], rem = blockIdx.x;
    if (colour_grid) {
        const int h3 = sg.nblk[3] / 2;
        const int b3h = rem % h3; rem /= h3;
        B[2] = rem % sg.nblk[2]; rem /= sg.nblk[2];
        B[1] = rem % sg.nblk[1];
        B[0] = rem / sg.nblk[1];
        B[3] = 2 * b3h + ((B[0] + B[1] + B[2] + colour) & 1);
    } else {
        B[3] = rem % sg.nblk[3]; rem /= sg.nblk[3];
        B[2] = rem % sg.nblk[2]; rem /= sg.nblk[2];
        B[1] = rem % sg.nblk[1];
        B[0] = rem / sg.nblk[1];
        if (((B[0] + B[1] + B[2] + B[3]) & 1) != colour) return;   // uniform over the CTA
    }
    v += rows.row[blockIdx.y] * stride;
    x += rows.row[blockIdx.y] * stride;
    const int nb = sg.nb;
    Sap32<S> &m = *reinterpret_cast<Sap32<S> *>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int k = lane >> 4, site = warp * 16 + (lane & 15);
    const bool act = site < nb;   // the CTA is padded to whole warps; the others join the reductions
    const int t = act ? site : 0;
    int l[4], rr = t;
    l[3] = rr % sg.b[3]; rr /= sg.b[3];
    l[2] = rr % sg.b[2]; rr /= sg.b[2];
    l[1] = rr % sg.b[1];
    l[0] = rr / sg.b[1];
    int xg[4];
#pragma unroll
    for (int mu = 0; mu < 4; mu++) xg[mu] = B[mu] * sg.b[mu] + l[mu];
    const int p = (xg[0] + xg[1] + xg[2] + xg[3]) & 1;
    const int i = eo_index(g, xg);
    if (act)
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int mu = 2 * k + h;
            cpx<float> u[3][3];
            load_link<float>(U, g.Vh, p, mu, i, u);
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const cpx<float> e0 = u[(2 * c) / 3][(2 * c) % 3], e1 = u[(2 * c + 1) / 3][(2 * c + 1) % 3];
                m.uA[4 * mu + c][t] = make_float4(e0.re, e0.im, e1.re, e1.im);
            }
            m.uB[mu][t] = make_float2(u[2][2].re, u[2][2].im);
        }
    cpx<float> ru[3], rl[3], eu[3], el[3];   // residual and correction: spins k and 2 + k
#pragma unroll
    for (int c = 0; c < 3; c++) eu[c] = el[c] = ru[c] = rl[c] = cpx<float>{0.f, 0.f};
    if (act) {
        glob_spin(v, g.Vh, p, i, k, ru);
        glob_spin(v, g.Vh, p, i, 2 + k, rl);
    }
    if (START != kSapFresh) {
        __syncthreads();   // links
        cpx<float> au[3], al[3], ax[3];
#pragma unroll
        for (int c = 0; c < 3; c++) au[c] = al[c] = ax[c] = cpx<float>{0.f, 0.f};
        constexpr bool OUT = START == kSapOwnZero;
        sap_glob_dir<0, OUT>(g, m, U, x, p, xg, t, k, l, sg, au, al);
        sap_glob_dir<1, OUT>(g, m, U, x, p, xg, t, k, l, sg, au, ax);
        sap_glob_dir<2, OUT>(g, m, U, x, p, xg, t, k, l, sg, au, ax);
        sap_glob_dir<3, OUT>(g, m, U, x, p, xg, t, k, l, sg, au, al);
        __syncwarp();
        sap_exchange(al, ax);
        if (act) {
            cpx<float> xu[3], xl[3];
            if (!OUT) {
                glob_spin(x, g.Vh, p, i, k, xu);
                glob_spin(x, g.Vh, p, i, 2 + k, xl);
            }
#pragma unroll
            for (int c = 0; c < 3; c++) {
                if (!OUT) {
                    au[c] = cpx<float>{fma_r(m4, xu[c].re, au[c].re), fma_r(m4, xu[c].im, au[c].im)};
                    al[c] = cpx<float>{fma_r(m4, xl[c].re, al[c].re), fma_r(m4, xl[c].im, al[c].im)};
                }
                ru[c] = ru[c] - au[c];
                rl[c] = rl[c] - al[c];
            }
        }
    }
    for (int it = 0; it < mr_iters; it++) {
        if (act) {
            sap_put_spin(m, k, t, ru);
            sap_put_spin(m, 2 + k, t, rl);
        }
        __syncthreads();   // s and, in the first step, the links
        cpx<float> qu[3], ql[3], qx[3];
#pragma unroll
        for (int c = 0; c < 3; c++) qu[c] = ql[c] = qx[c] = cpx<float>{0.f, 0.f};
        sap_block_dir<0>(m, t, k, l, sg, qu, ql);
        sap_block_dir<1>(m, t, k, l, sg, qu, qx);
        sap_block_dir<2>(m, t, k, l, sg, qu, qx);
        sap_block_dir<3>(m, t, k, l, sg, qu, ql);
        __syncwarp();
        sap_exchange(ql, qx);
        float a0 = 0.f, a1 = 0.f, a2 = 0.f;   // Re<q, s>, Im<q, s>, |q|^2
#pragma unroll
        for (int c = 0; c < 3; c++) {
            qu[c] = cpx<float>{fma_r(m4, ru[c].re, qu[c].re), fma_r(m4, ru[c].im, qu[c].im)};
            ql[c] = cpx<float>{fma_r(m4, rl[c].re, ql[c].re), fma_r(m4, rl[c].im, ql[c].im)};
            a0 += qu[c].re * ru[c].re + qu[c].im * ru[c].im + ql[c].re * rl[c].re + ql[c].im * rl[c].im;
            a1 += qu[c].re * ru[c].im - qu[c].im * ru[c].re + ql[c].re * rl[c].im - ql[c].im * rl[c].re;
            a2 += norm2(qu[c]) + norm2(ql[c]);
        }
        if (!act) a0 = a1 = a2 = 0.f;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, off);
            a1 += __shfl_xor_sync(0xffffffffu, a1, off);
            a2 += __shfl_xor_sync(0xffffffffu, a2, off);
        }
        if (lane == 0) red[warp] = make_float4(a0, a1, a2, 0.f);
        __syncthreads();   // also: every thread is done reading s
        // every warp sums the (at most 16) warps' values in the same order
        const float4 w = (lane & 15) < nw ? red[lane & 15] : make_float4(0.f, 0.f, 0.f, 0.f);
        a0 = w.x;
        a1 = w.y;
        a2 = w.z;
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, off);
            a1 += __shfl_xor_sync(0xffffffffu, a1, off);
            a2 += __shfl_xor_sync(0xffffffffu, a2, off);
        }
        if (!(a2 > 0.f)) break;   // uniform over the CTA
        const cpx<float> alpha{a0 / a2, a1 / a2};
#pragma unroll
        for (int c = 0; c < 3; c++) {
            eu[c] = eu[c] + alpha * ru[c];
            el[c] = el[c] + alpha * rl[c];
            ru[c] = ru[c] - alpha * qu[c];
            rl[c] = rl[c] - alpha * ql[c];
        }
    }
    // x of this colour is read (kSapFull) by its own block only: every thread has passed a barrier since
    if (START == kSapFull && mr_iters == 0) __syncthreads();
    if (!act) return;
    if (ADD) {
        cpx<float> xu[3], xl[3];
        glob_spin(x, g.Vh, p, i, k, xu);
        glob_spin(x, g.Vh, p, i, 2 + k, xl);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            eu[c] = xu[c] + eu[c];
            el[c] = xl[c] + el[c];
        }
    }
    glob_put_spin(x, g.Vh, p, i, k, eu);
    glob_put_spin(x, g.Vh, p, i, 2 + k, el);
}

}  // namespace

// Grants the dynamic shared memory of kernel f once per size (per process).
template <typename K>
static cudaError_t grant_smem(K f, size_t smem, size_t &granted) {
    if (smem <= 48 * 1024 || smem <= granted) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e;
    }
    granted = smem;
    return cudaSuccess;
}

// Blocks of one colour: all of them with an even number of blocks in every direction (then the
// colours alternate across every face, also through the periodic boundary, so that one colour's
// blocks can form their own residuals in place and the grid can hold only that colour).
struct SapGrid {
    bool even;
    int blocks;
};
static SapGrid sap_grid(const SapGeom &sg) {
    const int n = sg.nblk[0] * sg.nblk[1] * sg.nblk[2] * sg.nblk[3];
    const bool even = !(sg.nblk[0] & 1) && !(sg.nblk[1] & 1) && !(sg.nblk[2] & 1) && !(sg.nblk[3] & 1);
    return SapGrid{even, even ? n / 2 : n};
}

template <int S, int START, bool ADD>
static cudaError_t launch_sap32_s(const Geom &g, const SapGeom &sg, const SapGrid &sp, const float4 *U, const float4 *v,
                                  float4 *x, long stride, const RowList &rows, float m4, int colour, int mr_iters,
                                  cudaStream_t st) {
    static size_t granted = 0;
    constexpr size_t smem = sizeof(Sap32<S>);
    cudaError_t e = grant_smem(k_sap_block32<S, START, ADD>, smem, granted);
    if (e != cudaSuccess) return e;
    const int threads = (sg.nb + 15) / 16 * 32;
    k_sap_block32<S, START, ADD><<<dim3(sp.blocks, rows.n), threads, smem, st>>>(g, sg, U, v, x, stride, rows, m4,
                                                                                 colour, mr_iters, sp.even);
    count_launches(1);
    return cudaGetLastError();
}
template <int START, bool ADD>
static cudaError_t launch_sap32(const Geom &g, const SapGeom &sg, const SapGrid &sp, const float4 *U, const float4 *v,
                                float4 *x, long stride, const RowList &rows, float m4, int colour, int mr_iters,
                                cudaStream_t st) {
    // blocks of up to 64 sites take 25 KB instead of 98, so that more of them fit on an SM
    return sg.nb <= 64 ? launch_sap32_s<64, START, ADD>(g, sg, sp, U, v, x, stride, rows, m4, colour, mr_iters, st)
                       : launch_sap32_s<256, START, ADD>(g, sg, sp, U, v, x, stride, rows, m4, colour, mr_iters, st);
}

cudaError_t sap_f32_rows(const Geom &g, const SapGeom &sg, const float4 *U, const float4 *v, float4 *x, float4 *r,
                         long stride, int n, const char *act, float m0, int cycles, int mr_iters, cudaStream_t st) {
    const SapGrid sp = sap_grid(sg);
    const float m4 = m0 + 4.f;
    const size_t bytes = (size_t)g.V * 6 * sizeof(float4);
    RowList rows{};
    cudaError_t e;
    for (int y = 0; y < n; y++) {
        if (!act || act[y]) rows.row[rows.n++] = y;
        if ((act && !act[y]) || !sp.even)
            if ((e = cudaMemsetAsync(x + y * stride, 0, bytes, st)) != cudaSuccess) return e;
    }
    if (!rows.n) return cudaSuccess;
    for (int cyc = 0; cyc < cycles; cyc++) {
        for (int colour = 0; colour < 2; colour++) {
            if (sp.even) {
                if (cyc == 0 && colour == 0)
                    e = launch_sap32<kSapFresh, false>(g, sg, sp, U, v, x, stride, rows, m4, colour, mr_iters, st);
                else if (cyc == 0)
                    e = launch_sap32<kSapOwnZero, false>(g, sg, sp, U, v, x, stride, rows, m4, colour, mr_iters, st);
                else
                    e = launch_sap32<kSapFull, true>(g, sg, sp, U, v, x, stride, rows, m4, colour, mr_iters, st);
                if (e != cudaSuccess) return e;
                continue;
            }
            if (cyc == 0 && colour == 0) {   // x = 0: the residual is v
                if ((e = launch_sap32<kSapFresh, true>(g, sg, sp, U, v, x, stride, rows, m4, colour, mr_iters, st)) !=
                    cudaSuccess)
                    return e;
                continue;
            }
            for (int k = 0; k < rows.n; k++) {   // r = v - D_W x on the whole lattice, then the block solves from r
                RowList one{};
                one.n = 1;
                const long off = rows.row[k] * stride;
                if ((e = wilson_f32(g, U, x + off, r, m0, 0, -1.f, v + off, 1.f, st)) != cudaSuccess) return e;
                if ((e = launch_sap32<kSapFresh, true>(g, sg, sp, U, r, x + off, 0, one, m4, colour, mr_iters, st)) !=
                    cudaSuccess)
                    return e;
            }
        }
    }
    return cudaSuccess;
}
cudaError_t sap_f32(const Geom &g, const SapGeom &sg, const float4 *U, const float4 *v, float4 *x, float4 *r,
                    float m0, int cycles, int mr_iters, cudaStream_t st) {
    return sap_f32_rows(g, sg, U, v, x, r, 0, 1, nullptr, m0, cycles, mr_iters, st);
}

template <bool RES>
static cudaError_t launch_sap64(const Geom &g, const SapGeom &sg, const SapGrid &sp, const double2 *U, const double2 *v,
                                double2 *x, double m4, int colour, int mr_iters, cudaStream_t st) {
    static size_t granted = 0;
    const size_t smem = (size_t)sg.nb * (kSapSpinor64 + 4 * kSapLink64) * sizeof(double2);
    cudaError_t e = grant_smem(k_sap_block<double, double2, double2, RES>, smem, granted);
    if (e != cudaSuccess) return e;
    const int threads = (sg.nb + 31) / 32 * 32;
    k_sap_block<double, double2, double2, RES><<<sp.blocks, threads, smem, st>>>(g, sg, U, v, x, m4, colour, mr_iters,
                                                                                 sp.even);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t sap_f64(const Geom &g, const SapGeom &sg, const double2 *U, const double2 *v, double2 *x, double2 *r,
                    double m0, int cycles, int mr_iters, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(x, 0, (size_t)g.V * 24 * sizeof(double), st);
    if (e != cudaSuccess) return e;
    const SapGrid sp = sap_grid(sg);
    const double m4 = m0 + 4.0;
    bool x_zero = true;
    for (int cyc = 0; cyc < cycles; cyc++) {
        for (int colour = 0; colour < 2; colour++) {
            if (x_zero) {
                e = launch_sap64<false>(g, sg, sp, U, v, x, m4, colour, mr_iters, st);
            } else if (sp.even) {
                e = launch_sap64<true>(g, sg, sp, U, v, x, m4, colour, mr_iters, st);
            } else {
                // r = v - D_W x on the whole lattice, then the block solves from r
                if ((e = wilson_f64(g, U, x, r, m0, 0, -1.0, v, 1.0, st)) != cudaSuccess) return e;
                e = launch_sap64<false>(g, sg, sp, U, r, x, m4, colour, mr_iters, st);
            }
            if (e != cudaSuccess) return e;
            x_zero = false;
        }
    }
    return cudaSuccess;
}

}  // namespace ovl
