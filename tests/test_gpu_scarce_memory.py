"""Calls that find little device memory left: what fails reports it and leaves the context as it was.
The lattice is 48^4 (a vector of FP64 is 1.0 GB), so that hundreds of MB stay free for the CUDA runtime
while an allocation of the library does not fit. Links are the identity; nothing here tests numbers."""
import contextlib

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1410_7170_gb300 as ovl  # noqa: E402

DIMS = (48, 48, 48, 48)
V = 48 ** 4
VEC = V * 12 * 16   # bytes of one FP64 vector


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1410_7170_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    yield
    torch.cuda.empty_cache()


@contextlib.contextmanager
def scarce(left):
    """All but `left` bytes of the free device memory taken."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del held
        torch.cuda.empty_cache()


def _op(**kw):
    u = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V, 4, 3, 3).contiguous()
    torch.cuda.synchronize()   # the library works on a stream of its own
    return ovl.Overlap(u, DIMS, 1.0, 0.05, ovl.params_default(lambda_min=0.2, lambda_max=8.0, mrhs_kernel=1, **kw))


def status(f, op, *args):
    return f(op.ctx, *[ovl._ptr(a) if isinstance(a, torch.Tensor) else a for a in args])


@pytest.mark.parametrize("precision", [ovl.OVL_FP64, ovl.OVL_MIXED_FP32])
def test_refused_call_leaves_no_trace_in_the_next_one(precision):
    """The Schwarz application's scratch vector does not fit: bad input is reported first, and the flags
    that it set are gone when the next call comes."""
    op = _op(precision=precision, sap_block=(4, 4, 4, 4))
    good = torch.ones((V, 4, 3), dtype=torch.complex128, device="cuda")
    bad, out = good.clone(), torch.full_like(good, 7.0)
    bad[-1, 3, 2] = float("nan")
    if precision != ovl.OVL_FP64:   # the FP32 vectors of the call, so that its scratch vector comes next
        op.wilson_apply_arith(torch.empty_like(good), good, -0.3, ovl.OVL_ARITH_FP32)
    f = ovl.lib().wilson_sap_apply
    with scarce(VEC // 4):
        assert status(f, op, out, bad, -0.3) == ovl.OVL_EINVAL
        assert status(f, op, out, good, -0.3) == ovl.OVL_ENOMEM
    assert bool((out == 7.0).all())
    assert status(f, op, out, good, -0.3) == ovl.OVL_OK
    op.close()
