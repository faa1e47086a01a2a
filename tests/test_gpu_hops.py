"""The warp-per-hop stencil (FP64, float-float) where its tiles, grid rows and scalar recurrences
have their edges: lattices below one tile, with a partial last tile, and with more tiles per
right-hand side than blocks; vectors whose squared norm is near the bottom of the FP64 range.

Tolerances: one Wilson application 1e-13 of the largest value (as for the other stencils); two
sign evaluations of one vector to tol = 1e-13 differ by rounding, 1e-11 relative (100 tol).
"""
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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _op(dims, **kw):
    U = synth.gauge_field(dims, 0.5, 500 + sum(dims), stout_steps=2)
    return U, ovl.Overlap(U, dims, 1.0, 0.05, ovl.params_default(lambda_min=0.2, lambda_max=8.0, **kw))


@pytest.mark.parametrize("ap", [0, 1])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 2, 4), (2, 4, 2, 6), (6, 2, 10, 4), (2, 2, 2, 66), (12, 4, 6, 2)])
@pytest.mark.parametrize("arith", [ovl.OVL_ARITH_FP64, ovl.OVL_ARITH_FF])
def test_stencil_at_tile_edges(dims, arith, ap):
    U, op = _op(dims, antiperiodic=ap)
    b = synth.rhs_gaussian(dims, 31)
    out = torch.empty_like(dev(b))
    op.wilson_apply_arith(out, dev(b), 0.3, arith)
    ref = sparse.wilson(b, U, dims, 0.3, antiperiodic=bool(ap))
    assert np.abs(out.cpu().numpy() - ref).max() < 1e-13 * np.abs(ref).max()
    op.close()


@pytest.mark.parametrize("dims,n", [((2, 2, 2, 6), 3), ((6, 4, 10, 8), 12), ((8, 8, 8, 10), 5)])
def test_rows_of_a_batch_equal_single_vectors(dims, n):
    U, op = _op(dims)
    b = dev(synth.rhs_gaussian(dims, 32, n_rhs=n))
    b[1] *= 1e-3
    out, one = torch.empty_like(b), torch.empty_like(b)
    op.ovl_apply_n(out, b, n, 1e-13)
    for k in range(n):
        op.ovl_apply(one[k], b[k], 1e-13)
        assert ((out[k] - one[k]).norm() / one[k].norm()).item() < 1e-11
    op.close()


@pytest.mark.parametrize("power", [-270, -400, 300])
def test_sign_scales_with_its_argument(power):
    """||b||^2 around 1e-160, 1e-238 and 1e183: the drop rule and the CG scalars use reciprocals of
    squared norms, scaled where they would leave the FP64 range."""
    dims = (4, 4, 4, 6)
    U, op = _op(dims)
    b = dev(synth.rhs_gaussian(dims, 33))
    ref, out = torch.empty_like(b), torch.empty_like(b)
    op.sign_apply(ref, b, 1e-13)
    op.sign_apply(out, b * 2.0 ** power, 1e-13)
    assert ((out * 2.0 ** -power - ref).norm() / ref.norm()).item() < 1e-11
    op.close()


def test_batches_of_both_arithmetics_share_vectors():
    """The mixed solve's float-float batches and D_N's FP64 batches use the same vectors, which
    grow with the batch: results are the same before and after the other has moved them."""
    dims = (4, 4, 4, 8)
    U, op = _op(dims, precision=ovl.OVL_MIXED_FP32, precond=ovl.OVL_PREC_RECURSIVE, sap_block=(2, 2, 2, 2))
    b = dev(synth.rhs_gaussian(dims, 34, n_rhs=9))

    def solve(n):
        x = torch.zeros_like(b[:n])
        op.ovl_solve(x, b[:n], n, 1e-10)
        return x

    def apply(n):
        y = torch.empty_like(b[:n])
        op.ovl_apply_n(y, b[:n], n, 1e-12)
        return y

    x2, y2, x3, y9 = solve(2), apply(2), solve(3), apply(9)
    assert torch.equal(solve(2), x2) and torch.equal(solve(3), x3)
    assert torch.equal(apply(2), y2) and torch.equal(apply(9), y9)
    r = torch.empty_like(x3)
    op.ovl_apply_n(r, x3, 3, 1e-13)
    assert ((r - b[:3]).norm() / b[:3].norm()).item() < 2e-10
    op.close()


@pytest.mark.parametrize("tps", [1, 4])
@pytest.mark.parametrize("arith,tol,bar", [(ovl.OVL_ARITH_FP64, 1e-12, 1e-12), (ovl.OVL_ARITH_FF, 1e-11, 1e-11),
                                           (ovl.OVL_ARITH_FP32, 1e-5, 2e-5)])
def test_chunk_lengths_and_pending_updates(arith, tol, bar, tps):
    """The shift updates are done four iterations at a time (two in a batch), and at the end of every
    chunk of check_every iterations: any chunk length, captured or not, stops after the same iteration
    and gives the same result up to the rounding of y (2e-5: 100 FP32 roundings, more in FP64 bars)."""
    dims = (6, 4, 4, 10)
    b = dev(synth.rhs_gaussian(dims, 35, n_rhs=3))
    ref, its = None, None
    for every, graphs in ((8, 1), (1, 1), (2, 0), (3, 1), (5, 0), (7, 1), (64, 1)):
        U, op = _op(dims, check_every=every, use_graphs=graphs, stencil_tps=tps)
        out = torch.empty_like(b)
        op.prof_enable(True)
        op.sign_apply_arith(out[0], b[0], tol, arith)
        n = {k: v["launches"] for k, v in op.prof_get(reset=True).items() if k.startswith("ms_shifts")}
        op.prof_enable(False)
        if arith == ovl.OVL_ARITH_FP64:
            op.ovl_apply_n(out, b, 3, tol)
        op.close()
        if ref is None:
            ref, its = out.clone(), n
            continue
        assert n == its, (every, n, its)
        m = 3 if arith == ovl.OVL_ARITH_FP64 else 1
        assert ((out[:m] - ref[:m]).norm() / ref[:m].norm()).item() < bar, (every, graphs)
