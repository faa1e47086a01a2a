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
// One thread per block site.
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

// FP32 (k_sap_site32): spinor float4 [6][nb], links float4 [4][3][nb], row 2 rebuilt in registers.
constexpr int kSapSpinor32 = 6, kSapLink32 = 3;
__device__ __forceinline__ void sm_load_sp(const float4 *s, int nb, int t, cpx<float> v[12]) {
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const float4 w = s[c * nb + t];
        v[2 * c] = cpx<float>{w.x, w.y};
        v[2 * c + 1] = cpx<float>{w.z, w.w};
    }
}
__device__ __forceinline__ void sm_load_link(const float4 *u, int nb, int mu, int t, cpx<float> m[3][3]) {
    const float4 *b = u + mu * kSapLink32 * nb + t;
#pragma unroll
    for (int c = 0; c < kSapLink32; c++) {
        const float4 w = b[c * nb];
        m[(2 * c) / 3][(2 * c) % 3] = cpx<float>{w.x, w.y};
        m[(2 * c + 1) / 3][(2 * c + 1) % 3] = cpx<float>{w.z, w.w};
    }
    reconstruct_row2(m);
}
// The one hop of a site of a 2^4 block in direction mu, to site n, forward or backward: with sg = -1 forward and +1
// backward, h = up + sg c low and the lower spins sg c^* a; the link is the site's, or the neighbour's
// adjoint. The same sums in the same order as the two branches of block_apply.
__device__ __forceinline__ void sap_one_hop(const float4 *s, const float4 *u, int nb, int mu, int t, int n, bool fwd,
                                            cpx<float> acc[12]) {
    const float sg = fwd ? -1.f : 1.f;
    cpx<float> v[12], h0[3], h1[3], a0[3], a1[3], m[3][3];
    sm_load_sp(s, nb, n, v);
    sm_load_link(u, nb, mu, fwd ? t : n, m);
    const bool cross = mu == 1 || mu == 2, turn = mu == 1 || mu == 3;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const cpx<float> low0 = v[(cross ? 9 : 6) + c], low1 = v[(cross ? 6 : 9) + c];
        const float s0 = mu == 0 ? sg : -sg, s1 = mu == 1 ? -sg : sg;
        h0[c] = v[c] + s0 * (turn ? mul_i(low0) : low0);
        h1[c] = v[3 + c] + s1 * (turn ? mul_i(low1) : low1);
    }
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = a; b < 3; b++) {
            const cpx<float> x = m[a][b], y = m[b][a];
            m[a][b] = cpx<float>{fwd ? x.re : y.re, fwd ? x.im : -y.im};
            m[b][a] = cpx<float>{fwd ? y.re : x.re, fwd ? y.im : -x.im};
        }
    su3_mul(m, h0, a0);
    su3_mul(m, h1, a1);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const cpx<float> l2 = cross ? a1[c] : a0[c], l3 = cross ? a0[c] : a1[c];
        acc[c] = acc[c] + a0[c];
        acc[3 + c] = acc[3 + c] + a1[c];
        acc[6 + c] = acc[6 + c] + sg * (turn ? mul_i(l2) : l2);
        acc[9 + c] = acc[9 + c] + (mu >= 2 ? -sg : sg) * (turn ? mul_i(l3) : l3);
    }
}

// q = D_BB s at local site t (local coords l, extents bx), links of the block in smem. TWO (FP32): all
// extents are 2, where a site has one hop per direction and its warp would run through both branches.
template <typename R, typename LT, typename ST, bool TWO = false>
__device__ __forceinline__ void block_apply(const ST *s, const LT *u, int nb, int t, const int l[4], const int bx[4],
                                            const int stride[4], R m4, cpx<R> q[12]) {
    cpx<R> acc[12];
#pragma unroll
    for (int c = 0; c < 12; c++) acc[c] = cpx<R>{0, 0};
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        if constexpr (TWO) {
            sap_one_hop(s, u, nb, mu, t, t ^ (8 >> mu), l[mu] == 0, acc);
            continue;
        }
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

// Block coordinates of CTA `rem`; false if the block has the other colour (a grid of all blocks).
__device__ __forceinline__ bool sap_block_of(const SapGeom &sg, int rem, int colour, bool colour_grid, int B[4]) {
    if (colour_grid) {
        const int h3 = sg.nblk[3] / 2;
        const int b3h = rem % h3; rem /= h3;
        B[2] = rem % sg.nblk[2]; rem /= sg.nblk[2];
        B[1] = rem % sg.nblk[1];
        B[0] = rem / sg.nblk[1];
        B[3] = 2 * b3h + ((B[0] + B[1] + B[2] + colour) & 1);
        return true;
    }
    B[3] = rem % sg.nblk[3]; rem /= sg.nblk[3];
    B[2] = rem % sg.nblk[2]; rem /= sg.nblk[2];
    B[1] = rem % sg.nblk[1];
    B[0] = rem / sg.nblk[1];
    return ((B[0] + B[1] + B[2] + B[3]) & 1) == colour;
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
    int B[4];
    if (!sap_block_of(sg, blockIdx.x, colour, colour_grid, B)) return;   // uniform over the CTA
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

// What is known of x before a block solve: the residual is v itself, v minus the hops from the
// neighbouring blocks (the block's own x is zero and is assigned), or v - D_W x.
enum SapStart { kSapFresh, kSapOwnZero, kSapFull };

// The hops of the global field x in direction MU that leave the block.
template <int MU>
__device__ __forceinline__ void sap_out_dir(const Geom &g, const SapGeom &sg, const float4 *__restrict__ U, const float4 *x,
                                            int p, int i, const int xg[4], const int l[4], cpx<float> acc[12]) {
    cpx<float> v[12], h0[3], h1[3], a0[3], a1[3], m[3][3];
    int y[4] = {xg[0], xg[1], xg[2], xg[3]};
    if (l[MU] + 1 == sg.b[MU]) {
        y[MU] = xg[MU] + 1 == g.L[MU] ? 0 : xg[MU] + 1;
        load_spinor<float>(x, g.Vh, 1 - p, eo_index(g, y), v);
        load_link<float>(U, g.Vh, p, MU, i, m);
        proj_fwd(MU, v, h0, h1);
        if (MU == 0) flip_half(h0, h1, g.antiperiodic && xg[0] == g.L[0] - 1);
        su3_mul(m, h0, a0);
        su3_mul(m, h1, a1);
        acc_fwd<false>(MU, acc, a0, a1);
    }
    if (l[MU] == 0) {
        y[MU] = xg[MU] == 0 ? g.L[MU] - 1 : xg[MU] - 1;
        const int j = eo_index(g, y);
        load_spinor<float>(x, g.Vh, 1 - p, j, v);
        load_link<float>(U, g.Vh, 1 - p, MU, j, m);
        proj_bwd(MU, v, h0, h1);
        if (MU == 0) flip_half(h0, h1, g.antiperiodic && xg[0] == 0);
        su3_dag_mul(m, h0, a0);
        su3_dag_mul(m, h1, a1);
        acc_bwd(MU, acc, a0, a1);
    }
}
// FP32: one CTA per block of the colour and right-hand side, one thread per block site; ADD: x += e
// instead of x = e. Bound: shared memory (a hop reads 96 B of spinor and 48 B of link) and, up to one
// CTA per SM, latency. Two CTAs of 256 threads share an SM (74 KB each: links as rows 0 and 1, the third
// rebuilt), so that one computes while the other loads its links, forms its residual or sums. Two
// threads per site by spin (all 18 reals of a link, read by both) filled an SM with one CTA and were
// slower from one CTA per SM on; four or two by direction moved all partial sums through shared
// memory. What the launch knows of x saves passes over it: x = 0 before the first colour, zero on the
// second colour's blocks. Right-hand sides of a batch are grid rows. One Schwarz application (two
// cycles, 6 MR steps), one thread per site without these savings -> two threads per site with them ->
// this form: 16^4 183 -> 142 -> 139 us, 24^4 621 -> 586 -> 492, 32^4 1593 -> 1632 -> 1254.
template <int START, bool ADD, bool TWO>
__global__ void __launch_bounds__(kBlock, 2)
    k_sap_site32(Geom g, SapGeom sg, const float4 *__restrict__ U, const float4 *__restrict__ v, float4 *x, long stride,
                 RowList rows, float m4, int colour, int mr_iters, bool colour_grid) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nb = TWO ? 16 : sg.nb;
    int B[4];
    if (!sap_block_of(sg, blockIdx.x, colour, colour_grid, B)) return;   // uniform over the CTA
    v += rows.row[blockIdx.y] * stride;
    x += rows.row[blockIdx.y] * stride;
    float4 *s = reinterpret_cast<float4 *>(smem_raw), *u = s + kSapSpinor32 * nb;
    const bool act = threadIdx.x < nb;   // the CTA is padded to whole warps; the others join the sums
    const int t = act ? threadIdx.x : 0;
    int l[4], rr = t, xg[4];
    l[3] = rr % sg.b[3]; rr /= sg.b[3];
    l[2] = rr % sg.b[2]; rr /= sg.b[2];
    l[1] = rr % sg.b[1];
    l[0] = rr / sg.b[1];
#pragma unroll
    for (int mu = 0; mu < 4; mu++) xg[mu] = B[mu] * sg.b[mu] + l[mu];
    const int p = (xg[0] + xg[1] + xg[2] + xg[3]) & 1;
    const int i = eo_index(g, xg);
    if (act) {
        const float4 *gu = U + (size_t)p * 4 * kSapLink32 * g.Vh + i;
#pragma unroll
        for (int c = 0; c < 4 * kSapLink32; c++) u[c * nb + t] = __ldg(gu + (size_t)c * g.Vh);
    }
    cpx<float> res[12], e[12], q[12];
#pragma unroll
    for (int c = 0; c < 12; c++) e[c] = res[c] = q[c] = cpx<float>{0.f, 0.f};
    if (act) {
        load_spinor<float>(v, g.Vh, p, i, res);
        if (START == kSapFull) {   // v - D_W x
            cpx<float> hop[12], own[12], dx[12];
            wilson_hop<float>(g, U, x, p, i, hop);
            load_spinor<float>(x, g.Vh, p, i, own);
            wilson_combine<float>(m4, own, hop, dx);
#pragma unroll
            for (int c = 0; c < 12; c++) res[c] = res[c] - dx[c];
        } else if (START == kSapOwnZero) {
            cpx<float> hop[12];
#pragma unroll
            for (int c = 0; c < 12; c++) hop[c] = cpx<float>{0.f, 0.f};
            sap_out_dir<0>(g, sg, U, x, p, i, xg, l, hop);
            sap_out_dir<1>(g, sg, U, x, p, i, xg, l, hop);
            sap_out_dir<2>(g, sg, U, x, p, i, xg, l, hop);
            sap_out_dir<3>(g, sg, U, x, p, i, xg, l, hop);
#pragma unroll
            for (int c = 0; c < 12; c++) res[c] = res[c] - hop[c];
        }
    }
    for (int it = 0; it < mr_iters; it++) {
        if (act)
#pragma unroll
            for (int c = 0; c < 6; c++)
                s[c * nb + t] = make_float4(res[2 * c].re, res[2 * c].im, res[2 * c + 1].re, res[2 * c + 1].im);
        __syncthreads();
        if (act) block_apply<float, float4, float4, TWO>(s, u, nb, t, l, sg.b, sg.stride, m4, q);
        float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
        for (int c = 0; c < 12; c++) {
            a0 += q[c].re * res[c].re + q[c].im * res[c].im;   // Re <q, s>
            a1 += q[c].re * res[c].im - q[c].im * res[c].re;   // Im <q, s>
            a2 += norm2(q[c]);
        }
        cpx<float> alpha;
        if (!mr_alpha<float>(a0, a1, a2, alpha)) break;   // uniform over the CTA
#pragma unroll
        for (int c = 0; c < 12; c++) {
            e[c] = e[c] + alpha * res[c];
            res[c] = res[c] - alpha * q[c];
        }
    }
    __syncthreads();   // every thread of the CTA has finished reading x before any writes it
    if (!act) return;
    if (ADD) {
        cpx<float> xv[12];
        load_spinor<float>(x, g.Vh, p, i, xv);
#pragma unroll
        for (int c = 0; c < 12; c++) e[c] = xv[c] + e[c];
    }
    store_spinor<float>(x, g.Vh, p, i, e);
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

template <int START, bool ADD, bool TWO>
static cudaError_t launch_sap32_form(const Geom &g, const SapGeom &sg, const SapGrid &sp, const float4 *U, const float4 *v,
                                float4 *x, long stride, const RowList &rows, float m4, int colour, int mr_iters,
                                cudaStream_t st) {
    static size_t granted = 0;
    const size_t smem = (size_t)sg.nb * (kSapSpinor32 + 4 * kSapLink32) * sizeof(float4);
    cudaError_t e = grant_smem(k_sap_site32<START, ADD, TWO>, smem, granted);
    if (e != cudaSuccess) return e;
    k_sap_site32<START, ADD, TWO><<<dim3(sp.blocks, rows.n), (sg.nb + 31) / 32 * 32, smem, st>>>(
        g, sg, U, v, x, stride, rows, m4, colour, mr_iters, sp.even);
    count_launches(1);
    return cudaGetLastError();
}

template <int START, bool ADD>
static cudaError_t launch_sap32(const Geom &g, const SapGeom &sg, const SapGrid &sp, const float4 *U, const float4 *v,
                                float4 *x, long stride, const RowList &rows, float m4, int colour, int mr_iters,
                                cudaStream_t st) {
    // blocks of 16 sites are 2^4. One cycle (us) with the best of one, two and four threads per site, with
    // the general form, and with the one for 2^4: 4^4 30 / 37 / 25, 8^4 35 / 37 / 28, 12^4 47 / 47 / 35, 16^4
    // 82 / 76 / 54, 24^4 332 / 316 / 223. A CTA is one warp there, bound by fetching its instructions.
    return sg.nb == 16 ? launch_sap32_form<START, ADD, true>(g, sg, sp, U, v, x, stride, rows, m4, colour, mr_iters, st)
               : launch_sap32_form<START, ADD, false>(g, sg, sp, U, v, x, stride, rows, m4, colour, mr_iters, st);
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
