// Host functions of the library that no entry point reaches alone, with C linkage for the tests.
#include "../paper_1410_7170_gb300/csrc/internal.h"

using namespace ovl;

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
