"""A Krylov solver whose preconditioner is a Krylov solver, on a right-hand side that is no unit vector:
residual at most 1.5 times the requested one, as for the other Wilson solves."""
import ctypes

import numpy as np
import pytest

import synth
from oracle import sparse

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1410_7170_gb300 as ovl  # noqa: E402
from internals import load  # noqa: E402


@pytest.mark.parametrize("scale", [1.0, 1e-3, 1e4])
def test_nested_solvers_keep_their_norms(scale):
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    lib = load("internals_solver")
    dims = (4, 4, 4, 8)
    U = synth.gauge_field(dims, 0.5, 71, stout_steps=3)
    b = scale * synth.rhs_gaussian(dims, 72)
    x = np.zeros_like(b)
    op = ovl.Overlap(U, dims, 1.0, 0.05, ovl.params_default(lambda_min=0.2, lambda_max=8.0, precision=ovl.OVL_MIXED_FP32,
                                                            sap_block=(2, 2, 2, 2)))
    D = ctypes.c_double
    assert lib.t_nested_solve_f32(op.ctx, ovl._ptr(x), ovl._ptr(b), D(-0.3), D(1e-4)) == 0
    r = b - sparse.wilson(x, U, dims, -0.3)
    assert np.linalg.norm(r) < 1.5e-4 * np.linalg.norm(b)
    op.close()
