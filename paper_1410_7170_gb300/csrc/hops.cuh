// Wilson stencil with one warp per hop: a block of eight warps takes a tile of 32 consecutive
// sites, warp w computes the hop of direction mu = w / 2 (forward for even w, backward for odd)
// of every site of the tile and leaves the link times half spinor products in shared memory;
// after a barrier the eight warps share out the components of the sites, sum the eight
// contributions in the order of the one-thread-per-site stencil (the same results bit for bit)
// and run the caller's epilogue.
//
// Used for small lattices in FP32 (the autotuner's choice: 8^4 5.8 -> 4.2 us a stencil, 16^4 8.3 -> 12.4,
// where the shared memory traffic costs more than the extra warps give), at all sizes in float-float (about
// 10k FP32 operations per site), and in FP64 (2 lanes per clock and SM on GB300, so a warp's FP64
// instruction holds the SM's unit for 16 clocks) but for some large lattices, where one thread per
// site is up to 3% faster (wilson_f64, ms_fp64_per_site):
//   * the work of a tile is spread evenly over the four schedulers. One thread per site fills
//     them only from about 150 x 2 x 256 sites on; at 8^4 its 304 blocks of 14 sites used two
//     schedulers of each SM with 14 of 32 lanes live;
//   * no thread holds the 24 accumulators of a site while it computes a hop, so three blocks
//     fit on an SM at 80 registers instead of two of one-thread-per-site blocks at 128;
//   * the direction is uniform in a warp: no divergence and no multiplications by spin units.
// The sum of the FP64 instructions per site is that of the one-thread form, 888 with the epilogue. One
// stencil, one thread per site -> one warp per hop (us): FP64 4^4 33 -> 8, 8^4 33 -> 12, 12^4 51 -> 39,
// 16^4 111 -> 109, 32^4 1687 -> 1680; float-float 8^4 25 -> 6, 16^4 38 -> 29, 24^4 194 -> 138, 32^4 535 ->
// 418. 32^4 in FP64 is 0.88 of the units' 2 lanes a clock (1479 us at the 2070 MHz of the run), 1.76 lanes;
// ovl_fma_peak's chains of fused multiply-adds reach 1.68 and are no bound for it.
#pragma once
#include "reduce.cuh"
#include "wilson_site.cuh"

namespace ovl {

constexpr int kHopBlock = 256;  // one warp per hop

// ---------------------------------------------------------------- packed float-float
// Two float-float numbers side by side, (a, b), as two FP32 pairs: the packed FP32 instructions
// of sm_100 and later (fma.rn.f32x2 and so on) round each half as the scalar ones do, issue once
// for both and so halve the issue slots and the length of the dependent chains.
struct f2 {
    unsigned long long v;
};
__device__ __forceinline__ f2 f2_pack(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_unpack(f2 x, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// sign bits of both halves flipped by masks of 0 or 0x80000000
__device__ __forceinline__ f2 f2_flip(f2 x, unsigned ma, unsigned mb) {
    float a, b;
    f2_unpack(x, a, b);
    return f2_pack(__uint_as_float(__float_as_uint(a) ^ ma), __uint_as_float(__float_as_uint(b) ^ mb));
}

struct ff2 {
    f2 hi, lo;
};
__device__ __forceinline__ ff2 ff2_load(float4 w) { return ff2{f2_pack(w.x, w.y), f2_pack(w.z, w.w)}; }
__device__ __forceinline__ float4 ff2_word(ff2 x) {
    float4 w;
    f2_unpack(x.hi, w.x, w.y);
    f2_unpack(x.lo, w.z, w.w);
    return w;
}
__device__ __forceinline__ ff2 ff2_flip(ff2 x, unsigned ma, unsigned mb) {
    return ff2{f2_flip(x.hi, ma, mb), f2_flip(x.lo, ma, mb)};
}
__device__ __forceinline__ ff2 f2_two_sum(f2 a, f2 b) {
    const f2 s = f2_add(a, b), bv = f2_sub(s, a);
    return ff2{s, f2_add(f2_sub(a, f2_sub(s, bv)), f2_sub(b, bv))};
}
__device__ __forceinline__ ff2 f2_fast_two_sum(f2 a, f2 b) {
    const f2 s = f2_add(a, b);
    return ff2{s, f2_sub(b, f2_sub(s, a))};
}
__device__ __forceinline__ ff2 ff2_add(ff2 a, ff2 b) {
    const ff2 s = f2_two_sum(a.hi, b.hi);
    return f2_fast_two_sum(s.hi, f2_add(s.lo, f2_add(a.lo, b.lo)));
}
// without the renormalisation (cadd_acc of wilson_site.cuh)
__device__ __forceinline__ ff2 ff2_add_lazy(ff2 a, ff2 b) {
    const ff2 s = f2_two_sum(a.hi, b.hi);
    return ff2{s.hi, f2_add(s.lo, f2_add(a.lo, b.lo))};
}

// One float-float factor, copied to both halves. The packed instructions have no negated
// operands, so the rounding errors of products are formed negated, which takes -hi and -lo.
struct ff2_factor {
    f2 hi, nhi, nlo;
};
__device__ __forceinline__ ff2_factor ff2_scale(float hi, float lo) {
    return ff2_factor{f2_pack(hi, hi), f2_pack(-hi, -hi), f2_pack(-lo, -lo)};
}
__device__ __forceinline__ ff2_factor ff2_scale(ff x) { return ff2_scale(x.hi, x.lo); }
// a b + c (ff_fma)
__device__ __forceinline__ ff2 ff2_fma(const ff2_factor &a, ff2 b, ff2 c) {
    const f2 p = f2_mul(a.hi, b.hi);
    f2 ne = f2_fma(a.nhi, b.hi, p);
    ne = f2_fma(a.nhi, b.lo, ne);
    ne = f2_fma(a.nlo, b.hi, ne);
    const ff2 s = f2_two_sum(p, c.hi);
    return f2_fast_two_sum(s.hi, f2_add(s.lo, f2_sub(c.lo, ne)));
}
// a b
__device__ __forceinline__ ff2 ff2_mul(const ff2_factor &a, ff2 b) {
    const f2 p = f2_mul(a.hi, b.hi);
    f2 ne = f2_fma(a.nhi, b.hi, p);
    ne = f2_fma(a.nhi, b.lo, ne);
    ne = f2_fma(a.nlo, b.hi, ne);
    const f2 s = f2_sub(p, ne);
    return ff2{s, f2_sub(f2_sub(p, s), ne)};
}
// x x + c, both halves
__device__ __forceinline__ ff2 ff2_square_add(ff2 x, ff2 c) {
    float a, b, d, e;
    f2_unpack(x.hi, a, b);
    f2_unpack(x.lo, d, e);
    return ff2_fma(ff2_factor{x.hi, f2_pack(-a, -b), f2_pack(-d, -e)}, x, c);
}
// Dot product of factors with pairs (ff_dot of wilson_site.cuh, the error sum negated).
struct ff2_dot {
    f2 s, ne;
    __device__ __forceinline__ void first(const ff2_factor &a, ff2 b) {
        s = f2_mul(a.hi, b.hi);
        ne = f2_fma(a.nhi, b.hi, s);
        ne = f2_fma(a.nhi, b.lo, ne);
        ne = f2_fma(a.nlo, b.hi, ne);
    }
    __device__ __forceinline__ void add(const ff2_factor &a, ff2 b) {
        const f2 p = f2_mul(a.hi, b.hi);
        const f2 nep = f2_fma(a.nhi, b.hi, p);
        const ff2 t = f2_two_sum(s, p);
        s = t.hi;
        ne = f2_sub(ne, f2_sub(t.lo, nep));
        ne = f2_fma(a.nhi, b.lo, ne);
        ne = f2_fma(a.nlo, b.hi, ne);
    }
    __device__ __forceinline__ ff2 done() const {
        const f2 r = f2_sub(s, ne);
        return ff2{r, f2_sub(f2_sub(s, r), ne)};
    }
};

// ---------------------------------------------------------------- one hop
// Neighbour of the site with coordinates x in direction mu: its checkerboard index, and
// whether the hop crosses the antiperiodic boundary.
__device__ __forceinline__ int hop_neighbour(const Geom &g, const int x[4], int mu, bool fwd, bool &flip) {
    int y[4];
#pragma unroll
    for (int m = 0; m < 4; m++) {
        const int to = fwd ? (x[m] + 1 == g.L[m] ? 0 : x[m] + 1) : (x[m] == 0 ? g.L[m] - 1 : x[m] - 1);
        y[m] = m == mu ? to : x[m];
    }
    flip = mu == 0 && g.antiperiodic && x[0] == (fwd ? g.L[0] - 1 : 0);
    return eo_index(g, y);
}

// Tile<R>: shared memory word, the hop of one warp, and the components of a tile.
template <typename R> struct HopTiles;

// FP64. A tile is 16 sites: lanes 0-15 of a hop's warp form h0 of the half spinor, lanes 16-31 h1,
// and leave 12 reals per site, [h0, h1][colour][re, im]. In the second part item r is complex
// component r of the spinor, its real part in lanes 0-15 and its imaginary part in lanes 16-31.
template <> struct HopTiles<double> {
    using Word = double;
    using Elem = double;
    using Factor = double;
    using Store = double2;
    using Link = double2;
    static constexpr int tile = 16, words = 12, items = 12;

    template <int MU, bool FWD>
    __device__ static void hop(const Geom &g, const double2 *__restrict__ U, const double2 *__restrict__ in, int p, int i,
                               const int x[4], int k, Word *out) {
        bool flip;
        const int j = hop_neighbour(g, x, MU, FWD, flip);
        // h = s_k + c s_l with l = 2 + k or 3 - k, c one of +-1, +-i (proj_fwd, proj_bwd)
        constexpr bool cross = MU == 1 || MU == 2, turn = MU == 1 || MU == 3;
        const bool neg = (MU == 0 || (MU >= 2 && k)) != !FWD;
        const double2 *f = in + (size_t)(1 - p) * 12 * g.Vh + j;
        const int up = 3 * k, low = 6 + 3 * (cross ? 1 - k : k);
        cpx<double> h[3], a[3], u[3][3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double2 s = __ldg(f + (size_t)(up + c) * g.Vh), l = __ldg(f + (size_t)(low + c) * g.Vh);
            h[c].re = s.x + flip_sign(turn ? l.y : l.x, turn ? !neg : neg);
            h[c].im = s.y + flip_sign(turn ? l.x : l.y, neg);
            if (MU == 0) h[c] = cpx<double>{flip_sign(h[c].re, flip), flip_sign(h[c].im, flip)};
        }
        if (FWD) {
            load_link<double>(U, g.Vh, p, MU, i, u);
            su3_mul(u, h, a);
        } else {
            load_link<double>(U, g.Vh, 1 - p, MU, j, u);
            su3_dag_mul(u, h, a);
        }
#pragma unroll
        for (int c = 0; c < 3; c++) {
            out[(6 * k + 2 * c) * tile] = a[c].re;
            out[(6 * k + 2 * c + 1) * tile] = a[c].im;
        }
    }
    // out: this hop's words of the lane's site, `tile` apart; sub = lane / tile
    __device__ static void hop(const Geom &g, const Link *__restrict__ U, const Store *__restrict__ in, int p, int i,
                               const int x[4], int w, int sub, Word *out) {
        switch (w) {
            case 0: hop<0, true>(g, U, in, p, i, x, sub, out); break;
            case 1: hop<0, false>(g, U, in, p, i, x, sub, out); break;
            case 2: hop<1, true>(g, U, in, p, i, x, sub, out); break;
            case 3: hop<1, false>(g, U, in, p, i, x, sub, out); break;
            case 4: hop<2, true>(g, U, in, p, i, x, sub, out); break;
            case 5: hop<2, false>(g, U, in, p, i, x, sub, out); break;
            case 6: hop<3, true>(g, U, in, p, i, x, sub, out); break;
            default: hop<3, false>(g, U, in, p, i, x, sub, out); break;
        }
    }
    // Item `it` summed over the hops; part: the words of the lane's site.
    __device__ static Elem sum(const Word *part, int it, int im) {
        const int spin = it / 3, c = it - 3 * spin, k = spin & 1;
        const bool low = spin >= 2;
        Elem acc = 0.0;
#pragma unroll
        for (int h = 0; h < 8; h++) {
            const int mu = h >> 1;
            // lower spins are +-1 or +-i times h0 or h1 (acc_fwd, acc_bwd)
            const bool cross = mu == 1 || mu == 2, turn = mu == 1 || mu == 3;
            int half = k, q = im;
            bool neg = false;
            if (low) {
                half = cross ? 1 - k : k;
                q = turn ? 1 - im : im;
                neg = mu == 0 ? true : mu == 1 ? im != 0 : mu == 2 ? k == 0 : (im != 0) != (k != 0);
                if (h & 1) neg = !neg;
            }
            const double v = flip_sign(part[(h * words + 6 * half + 2 * c + q) * tile], neg);
            acc = h == 0 ? v : acc + v;
        }
        return acc;
    }
    __device__ static bool upper(int it) { return it < 6; }
    __device__ static size_t at(int Vh, int p, int i, int it, int im) {
        return 2 * ((size_t)(p * 12 + it) * Vh + i) + im;
    }
    __device__ static Elem load(const Store *f, int Vh, int p, int i, int it, int im) {
        return __ldg(reinterpret_cast<const double *>(f) + at(Vh, p, i, it, im));
    }
    __device__ static Elem load_rw(const Store *f, int Vh, int p, int i, int it, int im) {
        return reinterpret_cast<const double *>(f)[at(Vh, p, i, it, im)];
    }
    __device__ static void store(Store *f, int Vh, int p, int i, int it, int im, Elem v) {
        reinterpret_cast<double *>(f)[at(Vh, p, i, it, im)] = v;
    }
    // component `it` of site s of a boundary vector ([s][12] complex doubles)
    __device__ static void store_lex(double *f, int s, int it, int im, Elem v) { f[24 * (size_t)s + 2 * it + im] = v; }
    __device__ static Factor factor(double a) { return a; }
    __device__ static Factor minus_alpha(const MsState &s) { return -s.alpha; }
    __device__ static Factor sigma0(const MsState &s) { return s.sigma[0]; }
    __device__ static Elem fma(Factor a, Elem b, Elem c) { return __fma_rn(a, b, c); }
    __device__ static Elem mul(Factor a, Elem b) { return a * b; }
    __device__ static Elem neg_if(Elem x, bool n) { return flip_sign(x, n); }
    using Sum = double;
    __device__ static void square_add(Elem x, Sum &s) { s = __fma_rn(x, x, s); }
    __device__ static Sum zero() { return 0.0; }
    __device__ static double total(Sum s) { return s; }
};

// FP32. A tile is 32 sites; a hop leaves 12 reals per site, [h0, h1][colour][re, im]; item j is
// storage word j, complex components 2 j and 2 j + 1 (six items: two of the eight warps idle in the
// second part, which is a tenth of the work).
template <> struct HopTiles<float> {
    using Word = float;
    using Elem = float4;
    using Factor = float;
    using Store = float4;
    using Link = float4;
    static constexpr int tile = 32, words = 12, items = 6;

    template <int MU, bool FWD>
    __device__ static void hop(const Geom &g, const float4 *__restrict__ U, const float4 *__restrict__ in, int p, int i,
                               const int x[4], Word *out) {
        bool flip;
        const int j = hop_neighbour(g, x, MU, FWD, flip);
        cpx<float> s[12], h0[3], h1[3], a0[3], a1[3], u[3][3];
        load_spinor<float>(in, g.Vh, 1 - p, j, s);
        if (FWD) load_link<float>(U, g.Vh, p, MU, i, u);
        else load_link<float>(U, g.Vh, 1 - p, MU, j, u);
        if (FWD) proj_fwd(MU, s, h0, h1);
        else proj_bwd(MU, s, h0, h1);
        if (MU == 0) flip_half(h0, h1, flip);
        if (FWD) {
            su3_mul(u, h0, a0);
            su3_mul(u, h1, a1);
        } else {
            su3_dag_mul(u, h0, a0);
            su3_dag_mul(u, h1, a1);
        }
#pragma unroll
        for (int c = 0; c < 3; c++) {
            out[(2 * c) * tile] = a0[c].re;
            out[(2 * c + 1) * tile] = a0[c].im;
            out[(6 + 2 * c) * tile] = a1[c].re;
            out[(7 + 2 * c) * tile] = a1[c].im;
        }
    }
    __device__ static void hop(const Geom &g, const Link *__restrict__ U, const Store *__restrict__ in, int p, int i,
                               const int x[4], int w, int, Word *out) {
        switch (w) {
            case 0: hop<0, true>(g, U, in, p, i, x, out); break;
            case 1: hop<0, false>(g, U, in, p, i, x, out); break;
            case 2: hop<1, true>(g, U, in, p, i, x, out); break;
            case 3: hop<1, false>(g, U, in, p, i, x, out); break;
            case 4: hop<2, true>(g, U, in, p, i, x, out); break;
            case 5: hop<2, false>(g, U, in, p, i, x, out); break;
            case 6: hop<3, true>(g, U, in, p, i, x, out); break;
            default: hop<3, false>(g, U, in, p, i, x, out); break;
        }
    }
    __device__ static Elem sum(const Word *part, int it, int) {
        float acc[4];
#pragma unroll
        for (int d = 0; d < 2; d++) {
            const int cix = 2 * it + d, spin = cix / 3, c = cix - 3 * spin, k = spin & 1;
            const bool low = spin >= 2;
#pragma unroll
            for (int h = 0; h < 8; h++) {
                const int mu = h >> 1;
                // lower spins are +-1 or +-i times h0 or h1 (acc_fwd, acc_bwd)
                const bool cross = mu == 1 || mu == 2, turn = mu == 1 || mu == 3;
                const int half = low && cross ? 1 - k : k;
                const float *b = part + (h * words + 6 * half + 2 * c) * tile;
                float re = b[0], im = b[tile];
                if (low) {
                    const bool sre = (mu == 0 || (mu == 2 && k == 0) || (mu == 3 && k == 1)) != ((h & 1) != 0);
                    const bool sim = (mu == 0 || mu == 1 || (mu == 2 && k == 0) || (mu == 3 && k == 0)) != ((h & 1) != 0);
                    const float a = turn ? im : re, e = turn ? re : im;
                    re = flip_sign(a, sre);
                    im = flip_sign(e, sim);
                }
                acc[2 * d] = h == 0 ? re : acc[2 * d] + re;
                acc[2 * d + 1] = h == 0 ? im : acc[2 * d + 1] + im;
            }
        }
        return make_float4(acc[0], acc[1], acc[2], acc[3]);
    }
    __device__ static bool upper(int it) { return it < 3; }
    __device__ static size_t at(int Vh, int p, int i, int it) { return (size_t)(p * 6 + it) * Vh + i; }
    __device__ static Elem load(const Store *f, int Vh, int p, int i, int it, int) { return __ldg(f + at(Vh, p, i, it)); }
    __device__ static Elem load_rw(const Store *f, int Vh, int p, int i, int it, int) { return f[at(Vh, p, i, it)]; }
    __device__ static void store(Store *f, int Vh, int p, int i, int it, int, Elem v) { f[at(Vh, p, i, it)] = v; }
    __device__ static Factor factor(float a) { return a; }
    __device__ static Factor minus_alpha(const MsState &s) { return -s.alpha_f[0]; }
    __device__ static Factor sigma0(const MsState &s) { return s.sigma0_f[0]; }
    __device__ static Elem fma(Factor a, Elem b, Elem c) {
        return make_float4(__fmaf_rn(a, b.x, c.x), __fmaf_rn(a, b.y, c.y), __fmaf_rn(a, b.z, c.z), __fmaf_rn(a, b.w, c.w));
    }
    __device__ static Elem mul(Factor a, Elem b) { return make_float4(a * b.x, a * b.y, a * b.z, a * b.w); }
    __device__ static Elem neg_if(Elem x, bool n) {
        return make_float4(flip_sign(x.x, n), flip_sign(x.y, n), flip_sign(x.z, n), flip_sign(x.w, n));
    }
    using Sum = fsum;   // over all tiles of a block: at 32^4 with one warp per hop 54 of them
    __device__ static void square_add(Elem x, Sum &s) { s.add(x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w); }
    __device__ static Sum zero() { return Sum(); }
    __device__ static Sum total(const Sum &s) { return s; }
};

// Float-float. A word is a pair of float-float numbers, the same real of two spins, so that one
// link entry multiplies both: a hop leaves six words per site, [colour][re, im] of (h0, h1), and a
// spinor has twelve, [upper, lower spin pair][colour][re, im].
template <> struct HopTiles<ff> {
    using Word = float4;
    using Elem = ff2;
    using Factor = ff2_factor;
    using Store = ffw;
    using Link = ffl;
    static constexpr int tile = 32, words = 6, items = 12;

    // o[c] = sum_b u[c][b] h[b] (DAG: the adjoint link), h and o as [colour][re, im]
    // row: the link's first row (DAG: column). The next one is loaded before a row is used, and the first
    // one before the spinor's words are added up: a row's three loads cost an L2 round trip of their own
    // otherwise (24^4 144.7 -> 137.2 us; a multishift iteration at 16^4 2%).
    template <bool DAG>
    __device__ static void su3(const float4 *__restrict__ U, size_t Vh, const ff2 h[6], float4 row[3], Word *out) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            float4 next[3];
            if (a < 2) {
#pragma unroll
                for (int b = 0; b < 3; b++) next[b] = __ldg(U + (DAG ? 3 * b + a + 1 : 3 * a + 3 + b) * Vh);
            }
            ff2_dot re, im;
#pragma unroll
            for (int b = 0; b < 3; b++) {
                const float4 u = row[b];
                const ff2_factor ur = ff2_scale(u.x, u.y), ui = ff2_scale(u.z, u.w), mi = ff2_scale(-u.z, -u.w);
                if (b == 0) {
                    re.first(ur, h[0]);
                    im.first(ur, h[1]);
                } else {
                    re.add(ur, h[2 * b]);
                    im.add(ur, h[2 * b + 1]);
                }
                re.add(DAG ? ui : mi, h[2 * b + 1]);
                im.add(DAG ? mi : ui, h[2 * b]);
            }
            out[(2 * a) * tile] = ff2_word(re.done());
            out[(2 * a + 1) * tile] = ff2_word(im.done());
#pragma unroll
            for (int b = 0; b < 3; b++) row[b] = next[b];
        }
    }
    __device__ static void hop(const Geom &g, const Link *__restrict__ U, const Store *__restrict__ in, int p, int i,
                               const int x[4], int w, int, Word *out) {
        const int mu = w >> 1;
        const bool fwd = !(w & 1);
        bool flip;
        const int j = hop_neighbour(g, x, mu, fwd, flip);
        const float4 *f = reinterpret_cast<const float4 *>(in) + (size_t)(1 - p) * 12 * g.Vh + j;
        const float4 *l = reinterpret_cast<const float4 *>(U) +
                          (size_t)((fwd ? p : 1 - p) * 4 + mu) * kLink64Words * g.Vh + (fwd ? i : j);
        float4 row[3];
#pragma unroll
        for (int b = 0; b < 3; b++) row[b] = __ldg(l + (size_t)(fwd ? b : 3 * b) * g.Vh);
        // h = (s0, s1) + c (s2, s3) or c (s3, s2), c one of +-1, +-i per half (proj_fwd, proj_bwd)
        const bool cross = mu == 1 || mu == 2, turn = mu == 1 || mu == 3;
        const unsigned bit = 0x80000000u;
        // signs of c for h0 and h1: forward -1 -1, +i +i, +1 -1, +i -i
        unsigned s0 = mu == 0 ? bit : 0u, s1 = mu == 1 ? 0u : bit;
        if (!fwd) {
            s0 ^= bit;
            s1 ^= bit;
        }
        const unsigned r0 = turn ? s0 ^ bit : s0, r1 = turn ? s1 ^ bit : s1;   // real parts: i (a + i b) = -b + i a
        ff2 h[6];
#pragma unroll
        for (int c = 0; c < 3; c++) {
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const ff2 up = ff2_load(__ldg(f + (size_t)(2 * c + q) * g.Vh));
                float4 lw = __ldg(f + (size_t)(6 + 2 * c + (turn ? 1 - q : q)) * g.Vh);
                if (cross) lw = make_float4(lw.y, lw.x, lw.w, lw.z);
                h[2 * c + q] = ff2_add(up, q == 0 ? ff2_flip(ff2_load(lw), r0, r1) : ff2_flip(ff2_load(lw), s0, s1));
            }
        }
        if (mu == 0) {
            const unsigned m = flip ? bit : 0u;
#pragma unroll
            for (int k = 0; k < 6; k++) h[k] = ff2_flip(h[k], m, m);
        }
        if (fwd) su3<false>(l, g.Vh, h, row, out);
        else su3<true>(l, g.Vh, h, row, out);
    }
    __device__ static Elem sum(const Word *part, int it, int) {
        const int low = it >= 6, cq = low ? it - 6 : it, im = cq & 1;
        const unsigned bit = 0x80000000u;
        Elem acc = zero();
#pragma unroll
        for (int h = 0; h < 8; h++) {
            const int mu = h >> 1;
            ff2 v;
            if (!low) {
                v = ff2_load(part[((size_t)h * words + cq) * tile]);
            } else {   // forward: -(h0, h1), -i (h1, h0), (-h1, h0), (-i h0, i h1); backward negated
                const bool cross = mu == 1 || mu == 2, turn = mu == 1 || mu == 3;
                float4 lw = part[((size_t)h * words + (turn ? cq ^ 1 : cq)) * tile];
                if (cross) lw = make_float4(lw.y, lw.x, lw.w, lw.z);
                unsigned m0 = mu == 0 || mu == 2 || im ? bit : 0u;
                unsigned m1 = mu == 0 ? bit : mu == 1 ? (im ? bit : 0u) : mu == 2 ? 0u : (im ? 0u : bit);
                if (h & 1) {
                    m0 ^= bit;
                    m1 ^= bit;
                }
                v = ff2_flip(ff2_load(lw), m0, m1);
            }
            acc = h == 0 ? v : ff2_add_lazy(acc, v);
        }
        return acc;
    }
    __device__ static bool upper(int it) { return it < 6; }
    __device__ static size_t at(int Vh, int p, int i, int it) { return (size_t)(p * 12 + it) * Vh + i; }
    __device__ static Elem load(const Store *f, int Vh, int p, int i, int it, int) {
        return ff2_load(__ldg(reinterpret_cast<const float4 *>(f) + at(Vh, p, i, it)));
    }
    __device__ static Elem load_rw(const Store *f, int Vh, int p, int i, int it, int) {
        return ff2_load(reinterpret_cast<const float4 *>(f)[at(Vh, p, i, it)]);
    }
    __device__ static void store(Store *f, int Vh, int p, int i, int it, int, Elem v) {
        reinterpret_cast<float4 *>(f)[at(Vh, p, i, it)] = ff2_word(v);
    }
    __device__ static Factor factor(ff a) { return ff2_scale(a); }
    __device__ static Factor minus_alpha(const MsState &s) { return ff2_scale(-s.alpha_f[0], -s.alpha_f[1]); }
    __device__ static Factor sigma0(const MsState &s) { return ff2_scale(s.sigma0_f[0], s.sigma0_f[1]); }
    __device__ static Elem fma(const Factor &a, Elem b, Elem c) { return ff2_fma(a, b, c); }
    __device__ static Elem mul(const Factor &a, Elem b) { return ff2_mul(a, b); }
    __device__ static Elem neg_if(Elem x, bool n) { return ff2_flip(x, n ? 0x80000000u : 0u, n ? 0x80000000u : 0u); }
    using Sum = ff2;
    __device__ static void square_add(Elem x, Sum &s) { s = ff2_square_add(x, s); }
    __device__ static Sum zero() { return ff2{f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)}; }
    __device__ static ff total(Sum s) {
        float a, b, c, d;
        f2_unpack(s.hi, a, b);
        f2_unpack(s.lo, c, d);
        return ff(a, c) + ff(b, d);
    }
};

// Blocks resident per SM that the kernels are compiled for.
template <typename R> struct HopBlocks;
template <> struct HopBlocks<double> { static constexpr int value = 3; };
template <> struct HopBlocks<ff> { static constexpr int value = 3; };
template <> struct HopBlocks<float> { static constexpr int value = 4; };

// Tiles first, first + step, ... : epi(p, i, item, sub, hop, s, o) is called for each of the warp's items in
// every lane that holds a site, with the hopping sum (times -1/2, the stored links' factor), the
// site's lexicographic index and o = own(p, i, item, sub): what the epilogue reads at the site, loaded
// for the warp's first item before the barrier (float-float iteration at 16^4 0.7% less).
template <typename R, typename Own, typename Epi>
__device__ __forceinline__ void hop_tiles(const Geom &g, int first, int step,
                                          const typename HopTiles<R>::Link *__restrict__ U,
                                          const typename HopTiles<R>::Store *__restrict__ in, Own own, Epi epi) {
    using H = HopTiles<R>;
    __shared__ typename H::Word part[8 * H::words * H::tile];
    const int lane = threadIdx.x % H::tile, sub = (threadIdx.x & 31) / H::tile, w = threadIdx.x >> 5;
    const int tiles = (g.V + H::tile - 1) / H::tile;
    for (int tile = first; tile < tiles; tile += step) {
        const int t = tile * H::tile + lane;
        const bool live = t < g.V;
        int p, i, x[4];
        site_of_thread(live ? t : 0, p, i);
        eo_coords(g, p, i, x);
        H::hop(g, U, in, p, i, x, w, sub, part + (size_t)w * H::words * H::tile + lane);
        auto o = own(p, i, min(w, H::items - 1), sub);   // the last warps may have no item
        __syncthreads();
#pragma unroll
        for (int it = w; it < H::items; it += 8) {
            if (it != w) o = own(p, i, it, sub);
            const typename H::Elem hop = H::sum(part + lane, it, sub);
            if (live) epi(p, i, it, sub, hop, 2 * i + (x[3] & 1), o);
        }
        if (tile + step < tiles) __syncthreads();   // the next tile overwrites part
    }
}

// Blocks for the tiles of a lattice: one each in a plain stencil; where a reduction follows
// (wave = true), one wave of resident blocks that take the tiles in turn, because a block ends with a
// fence and an atomic whose round trip its slot then waits for (float-float at 16^4: 47 us with 2048
// blocks of one tile).
template <typename R>
inline int hop_grid(const Geom &g, int rows, bool wave) {
    const int tiles = (g.V + HopTiles<R>::tile - 1) / HopTiles<R>::tile;
    if (!wave) return tiles;
    const int most = g.nsm * HopBlocks<R>::value / rows;
    return tiles < most ? tiles : (most < 1 ? 1 : most);
}

}  // namespace ovl
