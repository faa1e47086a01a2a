"""The FGMRES solvers' device-resident Gram-Schmidt at its edges: zero right-hand sides alone and
among others, right-hand sides of very different size, restarts, iteration caps, lattices smaller
than one block of the kernels. Solutions against dense LU (1e-8, as the other solve tests) and
Wilson solves against their residual (1.5 tol)."""
import numpy as np
import pytest

import synth
from oracle import dense, sparse

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1410_7170_gb300 as ovl  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_7170_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("precision,precond,restart", [(ovl.OVL_FP64, ovl.OVL_PREC_NONE, 100),
                                                       (ovl.OVL_FP64, ovl.OVL_PREC_WILSON, 3),
                                                       (ovl.OVL_MIXED_FP32, ovl.OVL_PREC_RECURSIVE, 100),
                                                       (ovl.OVL_MIXED_FP32, ovl.OVL_PREC_WILSON, 4)])
@pytest.mark.parametrize("n", [1, 5])
def test_solves_with_zero_and_scaled_right_hand_sides(precision, precond, restart, n):
    dims = (2, 2, 4, 4)
    U = synth.gauge_field(dims, 0.3, 900)
    rho = dense.rho_from_mu(0.05, -1.0)
    DN, S, w = dense.overlap_dense(U, dims, rho, -1.0)
    aw = np.abs(w)
    op = ovl.Overlap(U, dims, 1.0, 0.05, ovl.params_default(
        lambda_min=0.98 * aw.min(), lambda_max=1.02 * aw.max(), precision=precision, precond=precond,
        sap_block=(2, 2, 2, 2), restart=restart, rhs_block=4))
    b = synth.rhs_gaussian(dims, 901, n_rhs=n)
    if n > 1:
        b[1] = 0
        b[2] *= 1e-6
        b[3] *= 1e6
    x = torch.zeros_like(dev(b))
    op.ovl_solve(x, dev(b), n, 1e-11)
    for k in range(n):
        if not b[k].any():
            assert not bool(x[k].any())
            continue
        ref = dense.overlap_solve_dense(DN, b[k])
        assert np.linalg.norm(x[k].cpu().numpy() - ref) < 1e-8 * np.linalg.norm(ref)
    z = torch.zeros_like(x[0])
    st, stats = op.ovl_solve(z, torch.zeros_like(z), 1, 1e-11)
    assert st == ovl.OVL_OK and not bool(z.any()) and stats["outer_iters"] == 0
    op.close()


@pytest.mark.parametrize("precision,tol", [(ovl.OVL_FP64, 1e-10), (ovl.OVL_MIXED_FP32, 1e-5)])
@pytest.mark.parametrize("restart", [2, 5, 120])
def test_wilson_solve_restarts_caps_and_zero(precision, tol, restart):
    dims = (4, 4, 4, 8)
    U = synth.gauge_field(dims, 0.5, 902, stout_steps=3)
    b = synth.rhs_gaussian(dims, 903)
    op = ovl.Overlap(U, dims, 1.0, 0.05, ovl.params_default(lambda_min=0.05, lambda_max=8.0, precision=precision,
                                                            sap_block=(2, 2, 2, 2), prec_restart=restart,
                                                            prec_max_iter=400))
    x = np.ones_like(b)
    assert op.wilson_solve(x, b, -0.3, tol) > 1
    r = b - sparse.wilson(x, U, dims, -0.3)
    assert np.linalg.norm(r) < 1.5 * tol * np.linalg.norm(b)
    assert op.wilson_solve(x, np.zeros_like(b), -0.3, tol) == 0 and not x.any()
    op.close()
    op = ovl.Overlap(U, dims, 1.0, 0.05, ovl.params_default(lambda_min=0.05, lambda_max=8.0, precision=precision,
                                                            sap_block=(2, 2, 2, 2), prec_restart=restart,
                                                            prec_max_iter=1))
    assert op.wilson_solve(x, b, -0.3, tol) == 1   # capped: one step's answer
    r = b - sparse.wilson(x, U, dims, -0.3)
    assert tol < np.linalg.norm(r) / np.linalg.norm(b) < 1
    op.close()
