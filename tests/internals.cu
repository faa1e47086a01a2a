// Host functions of the library that no entry point reaches alone, with C linkage for the tests.
#include "../paper_1410_7170_gb300/csrc/internal.h"
#include "../paper_1410_7170_gb300/csrc/sap.h"

using namespace ovl;

static Geom geom(const int *dims) {
    Geom g{};
    g.set_dims(dims);
    g.antiperiodic = 1;
    g.tps32 = 1;
    g.mrhs32 = g.mrhs32l = 1;
    g.nsm = device_sm_count();
    return g;
}
static int done(cudaError_t e) {
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    return (int)e;
}

// ms_init of nrhs FP64 vectors of `words` complex numbers with one pole, those with skip[y] != 0 marked as
// needing no work; status[y] and bb[y]: the solver's status and ||b_y||^2
extern "C" int t_ms_init(int nrhs, long words, const void *b, const int *skip, int *status, double *bb) {
    double2 *d = nullptr;
    MsState *s = nullptr;
    double *part = nullptr;
    MsState *h = new MsState[nrhs]();
    for (int y = 0; y < nrhs; y++) {
        h[y].n = 1;
        h[y].done = skip[y];
    }
    cudaError_t e = cudaMalloc(&d, (size_t)words * nrhs * ms_vectors(1, 1) * sizeof(double2));
    if (e == cudaSuccess) e = cudaMalloc(&s, sizeof(MsState) * nrhs);
    if (e == cudaSuccess) e = cudaMalloc(&part, sizeof(double) * 4 * kMaxRedBlocks * nrhs + 256);
    if (e == cudaSuccess) {
        const long v = words * nrhs;
        unsigned *cnt = (unsigned *)(part + (size_t)4 * kMaxRedBlocks * nrhs);
        const MsBatch<double2> w{d, d + v, d + 2 * v, d + 3 * v, d + 4 * v, words, 0, 1};
        cudaMemset(cnt, 0, 256);
        cudaMemcpy(s, h, sizeof(MsState) * nrhs, cudaMemcpyHostToDevice);
        e = ms_init(Geom{}, nrhs, s, w, (const double2 *)b, RedScratch{part, cnt}, cnt, 0);
        cudaMemcpy(h, s, sizeof(MsState) * nrhs, cudaMemcpyDeviceToHost);
        for (int y = 0; y < nrhs; y++) {
            status[y] = h[y].status;
            bb[y] = h[y].bb;
        }
    }
    const int st = done(e);
    cudaFree(d);
    cudaFree(s);
    cudaFree(part);
    delete[] h;
    return st;
}

// x (+)= sum_i c_i v_i of n_rows right-hand sides with cols[y] of m columns each (FP64, gs_combine)
extern "C" int t_gs_combine_f64(const double *base, long stride, int m, const double *c, const int *cols, double *x, int add,
                                long n, int n_rows) {
    RowList rows{n_rows, {}};
    RowColumns rc{};
    for (int y = 0; y < n_rows; y++) {
        rows.row[y] = y;
        rc.n[y] = cols[y];
    }
    return done(gs_combine<double>(base, stride, m, c, x, add != 0, n, rows, rc, 0));
}

// gs_dots of n_rows right-hand sides, all of them; out: n_rows records of gs_record(m) doubles
extern "C" int t_gs_dots_f32(const float *base, long stride, int m, const float *w, long n, int n_rows, double *out,
                             double *partials, unsigned *counters) {
    RowList rows{n_rows, {}};
    for (int y = 0; y < n_rows; y++) rows.row[y] = y;
    return done(gs_dots<float>(base, stride, m, w, n, rows, out, gs_record(m), false, nullptr, partials, counters, 0));
}

// nrhs multishift solves with shifts sigma0 and sigma0 + 1, stopped after `iters` iterations: scal = 5 doubles per
// right-hand side (||b||^2, ||r||^2, ||p_0||^2 as the solver has it, alpha of the last iteration, status);
// t, r, p0: the vectors' last values.
template <typename ST, typename LT>
static int ms_probe(const Geom &g, const LT *U, int nrhs, int ring, long words, const ST *b, int iters,
                    double sigma0, double *scal, ST *t, ST *r, ST *p0) {
    const int n = 2;
    ST *d = nullptr;
    MsState *s = nullptr;
    double *part = nullptr;
    MsState *h = new MsState[nrhs]();
    for (int y = 0; y < nrhs; y++) {
        h[y].n = n;
        h[y].tol = 1e-14;
        h[y].alpha_prev = 1.0;
        h[y].sigma[0] = sigma0;
        h[y].sigma[1] = sigma0 + 1.0;
        h[y].sigma0_f[0] = (float)sigma0;
        h[y].sigma0_f[1] = (float)(sigma0 - (double)(float)sigma0);
        for (int l = 0; l < n; l++) h[y].w[l] = h[y].crit[l] = h[y].zeta[l] = h[y].zeta_prev[l] = 1.0, h[y].active[l] = 1;
    }
    const long v = words * nrhs;
    cudaError_t e = cudaMalloc(&d, (size_t)v * ms_vectors(n, ring) * sizeof(ST));
    if (e == cudaSuccess) e = cudaMalloc(&s, sizeof(MsState) * nrhs);
    if (e == cudaSuccess) e = cudaMalloc(&part, sizeof(double) * kMaxRedBlocks * nrhs + 256);
    if (e == cudaSuccess) {
        unsigned *cnt = (unsigned *)(part + (size_t)kMaxRedBlocks * nrhs);
        const MsBatch<ST> w{d, d + v * ring, d + 2 * v * ring, d + (2 * ring + 1) * v, d + (2 * ring + 2) * v, words,
                            words * (n - 1), ring};
        cudaMemset(cnt, 0, 256);
        cudaMemcpy(s, h, sizeof(MsState) * nrhs, cudaMemcpyHostToDevice);
        e = ms_init(g, nrhs, s, w, b, RedScratch{part, cnt}, cnt, 0);
        for (int k = 0; k < iters && e == cudaSuccess; k++)
            e = ms_iter(g, U, -1.0, nrhs, s, w, RedScratch{part, cnt}, cnt, (k + 1) % ring == 0 || k == iters - 1, 0, MsEvents{});
        cudaMemcpy(h, s, sizeof(MsState) * nrhs, cudaMemcpyDeviceToHost);
        for (int y = 0; y < nrhs; y++) {
            const MsState &q = h[y];
            const double o[5] = {q.bb, q.rr, q.pp, q.alpha, (double)q.status};
            for (int k = 0; k < 5; k++) scal[5 * y + k] = o[k];
            cudaMemcpy(t + y * words, w.t + y * words, words * sizeof(ST), cudaMemcpyDeviceToDevice);
            cudaMemcpy(r + y * words, w.r_at(y, iters), words * sizeof(ST), cudaMemcpyDeviceToDevice);
            cudaMemcpy(p0 + y * words, w.p0_at(y, iters), words * sizeof(ST), cudaMemcpyDeviceToDevice);
        }
    }
    const int st = done(e);
    cudaFree(d);
    cudaFree(s);
    cudaFree(part);
    delete[] h;
    return st;
}
extern "C" int t_ms_probe(const int *dims, const double *gauge, int fp64, int tps32, int nrhs, int ring, const void *b, int iters,
                          double sigma0, double *scal, void *t, void *r, void *p0) {
    Geom g = geom(dims);
    g.tps32 = tps32;
    double2 *u64 = nullptr;
    float4 *u32 = nullptr;
    int *bad = nullptr;
    cudaError_t e = cudaMalloc(&u64, (size_t)g.V * 4 * kLink64Words * sizeof(double2));
    if (e == cudaSuccess) e = cudaMalloc(&u32, (size_t)g.V * 4 * 3 * sizeof(float4));
    if (e == cudaSuccess) e = cudaMalloc(&bad, sizeof(int));
    if (e == cudaSuccess) e = pack_gauge(g, gauge, u64, u32, bad, 1e-10, 0);
    int st = done(e);
    if (!st && fp64)
        st = ms_probe<double2>(g, u64, nrhs, ring, 12L * g.V, (const double2 *)b, iters, sigma0, scal, (double2 *)t, (double2 *)r,
                               (double2 *)p0);
    else if (!st)
        st = ms_probe<float4>(g, u32, nrhs, ring, 6L * g.V, (const float4 *)b, iters, sigma0, scal, (float4 *)t, (float4 *)r,
                              (float4 *)p0);
    cudaFree(u64);
    cudaFree(u32);
    cudaFree(bad);
    return st;
}

// One Schwarz application to n boundary vectors (device memory, back to back) as the batched solvers make
// it: rows with act[y] = 0 are left out
extern "C" int t_sap_rows_f32(const int *dims, const double *gauge, const int *block, const double *in, double *out,
                              const char *act, int n, double m0, int cycles, int mr_iters) {
    const Geom g = geom(dims);
    const long words = 6L * g.V;
    double2 *u64 = nullptr;
    float4 *u32 = nullptr, *v = nullptr;
    int *bad = nullptr;
    cudaError_t e = cudaMalloc(&u64, (size_t)g.V * 4 * kLink64Words * sizeof(double2));
    if (e == cudaSuccess) e = cudaMalloc(&u32, (size_t)g.V * 4 * 3 * sizeof(float4));
    if (e == cudaSuccess) e = cudaMalloc(&v, (size_t)words * (2 * n + 1) * sizeof(float4));
    if (e == cudaSuccess) e = cudaMalloc(&bad, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(v, 0xff, (size_t)words * (2 * n + 1) * sizeof(float4));   // NaN
    if (e == cudaSuccess) e = pack_gauge(g, gauge, u64, u32, bad, 1e-10, 0);
    if (e == cudaSuccess) e = spinor_in(g, v, words, in, n, InputFlags{nullptr, nullptr}, 0);
    float4 *x = v + words * n, *r = x + words * n;
    if (e == cudaSuccess) e = sap_f32_rows(g, make_sap_geom(g, block), u32, v, x, r, words, n, act, (float)m0, cycles, mr_iters, 0);
    if (e == cudaSuccess) e = spinor_out(g, out, x, words, n, nullptr, 0);
    const int st = done(e);
    cudaFree(u64);
    cudaFree(u32);
    cudaFree(v);
    cudaFree(bad);
    return st;
}
