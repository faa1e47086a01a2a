"""Boundary vectors (lexicographic, complex128) into and out of the internal formats: lattices
below one 64-site tile, with a partial last tile, and of whole tiles; one and several vectors;
host and device memory; NaN and Inf on device buffers, where the check is made at the end of
the call and the output must stay as it was.

Tolerances on the largest error over the largest value: 1e-13 in FP64 and float-float; FP32
3e-6, about 20 roundings of 2^-24 in a row on terms whose absolute sum is 2.5 times the result.
"""
import numpy as np
import pytest

import synth
from oracle import sparse

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1410_7170_gb300 as ovl  # noqa: E402

TOL = {ovl.OVL_ARITH_FP64: 1e-13, ovl.OVL_ARITH_FF: 1e-13, ovl.OVL_ARITH_FP32: 3e-6}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_7170_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _op(dims, tps=0):
    U = synth.gauge_field(dims, 0.5, 300 + sum(dims))
    return U, ovl.Overlap(U, dims, 1.0, 0.05, ovl.params_default(lambda_min=0.05, lambda_max=8.0, stencil_tps=tps))


@pytest.mark.parametrize("tps", [1, 4])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 4, 6), (2, 6, 6, 10), (4, 4, 4, 4), (4, 4, 6, 8), (12, 10, 8, 6)])
@pytest.mark.parametrize("arith", list(TOL))
def test_formats_on_partial_tiles(dims, arith, tps):
    U, op = _op(dims, tps)
    for n in (1,) if arith == ovl.OVL_ARITH_FF else (1, 3, 13):
        b = synth.rhs_gaussian(dims, 400 + n, n_rhs=n)
        ref = np.stack([sparse.wilson(b[k], U, dims, -0.7) for k in range(n)])
        for to in (dev, np.copy):
            out = to(np.zeros_like(b))
            if n == 1:
                op.wilson_apply_arith(out, to(b), -0.7, arith)
            else:
                op.wilson_apply_n_arith(out, to(b), n, -0.7, arith)
            o = out.cpu().numpy() if to is dev else out
            assert np.abs(o - ref).max() < TOL[arith] * np.abs(ref).max()
    op.close()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 6, 10), (4, 4, 4, 4)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("tps", [1, 4])
def test_nonfinite_device_input_leaves_output_and_context_alone(dims, bad, tps):
    U, op = _op(dims, tps)
    b = synth.rhs_gaussian(dims, 77, n_rhs=2)
    ref = sparse.wilson(b[0], U, dims, -0.7)
    at = dev(b)
    at[1, -1, 3, 2] = complex(0.5, bad)   # last component of the last vector
    out = torch.full_like(at, 7.0)
    calls = [lambda: op.wilson_apply(out[1], at[1], -0.7), lambda: op.wilson_apply_n(out, at, 2, -0.7),
             lambda: op.wilson_apply_n_arith(out, at, 2, -0.7, ovl.OVL_ARITH_FP32)]
    calls += [lambda a=a: op.wilson_apply_arith(out[1], at[1], -0.7, a) for a in range(5)]
    if all(d % 4 == 0 for d in dims):
        calls.append(lambda: op.sap_apply(out[1], at[1], -0.7))
    for call in calls:
        with pytest.raises(ovl.OvlError) as e:
            call()
        assert e.value.status == ovl.OVL_EINVAL
        assert bool((out == 7.0).all())
        good = torch.empty_like(at[0])
        op.wilson_apply(good, at[0], -0.7)   # the next call is not affected
        assert np.abs(good.cpu().numpy() - ref).max() < 1e-13 * np.abs(ref).max()
    op.close()
