"""FP64 on lattices of 2^19 sites and more, where the stencil and the multishift have a second form (one thread
per site): the stencil against the oracle's on host buffers, which take it, and on device buffers,
which don't (1e-13 of the largest value, as for the other stencils); the sign of one vector against
the rows of a batch (1e-11, two evaluations to 1e-12)."""
import numpy as np
import pytest

import synth
from oracle import sparse

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1410_7170_gb300 as ovl  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_7170_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def _op(dims):
    U = synth.gauge_field(dims, 0.5, 81, stout_steps=2, device="cuda")
    return U, ovl.Overlap(U, dims, 1.0, 0.05, ovl.params_default(lambda_min=0.2, lambda_max=8.0, mrhs_kernel=1))


@pytest.mark.parametrize("dims", [(28, 28, 28, 28), (26, 28, 30, 28), (30, 30, 26, 28)])
def test_stencil_forms(dims):
    U, op = _op(dims)
    b = synth.rhs_gaussian(dims, 82)
    ref = sparse.wilson(b, U, dims, -0.7)
    out, dev = np.empty_like(b), torch.empty(b.shape, dtype=torch.complex128, device="cuda")
    op.wilson_apply(out, b, -0.7)
    bd = torch.from_numpy(b).cuda()
    torch.cuda.synchronize()
    op.wilson_apply(dev, bd, -0.7)
    for o in (out, dev.cpu().numpy()):
        assert np.abs(o - ref).max() < 1e-13 * np.abs(ref).max()
    op.close()


@pytest.mark.parametrize("dims", [(32, 32, 32, 32), (34, 30, 32, 34)])
def test_sign_forms(dims):
    U, op = _op(dims)
    b = torch.from_numpy(synth.rhs_gaussian(dims, 83, n_rhs=2)).cuda()
    rows, one = torch.empty_like(b), torch.empty_like(b[0])
    torch.cuda.synchronize()
    op.ovl_apply_n(rows, b, 2, 1e-12)
    for k in range(2):
        op.ovl_apply(one, b[k], 1e-12)
        assert ((rows[k] - one).norm() / one.norm()).item() < 1e-11
    op.close()
