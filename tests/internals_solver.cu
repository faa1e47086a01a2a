// A Krylov solver inside another one, which the entry points only use on unit vectors: FGMRES on
// D_W(m0) preconditioned by wilson_solve, both from x = 0 without a final residual check.
#include "../paper_1410_7170_gb300/csrc/solver.cu"

using namespace ovl;

extern "C" int t_nested_solve_f32(ovl_ctx *ctx, double *x, const double *b, double m0, double tol) {
    Ctx *c = reinterpret_cast<Ctx *>(ctx);
    ST(ensure_f32_buffers(c));
    ST(c->import_vec(b, (float4 *)c->f_a));
    ST(ensure_krylov<float>(c, c->kry_inner, 8, true));
    auto mv = [&](const float *a, float *o, double) -> ovl_status {
        CK(Ops<float>::wilson(c, a, o, m0));
        return OVL_OK;
    };
    auto pc = [&](const float *a, float *o) -> ovl_status { return wilson_solve<float>(c, c->kry_wil32, a, o, m0, 0.1); };
    KrylovResult r;
    ST(fgmres<float>(c, c->kry_inner, c->f_b, c->f_a, tol, 100, true, mv, &pc, &r, false));
    return c->export_vec((const float4 *)c->f_b, x);
}
