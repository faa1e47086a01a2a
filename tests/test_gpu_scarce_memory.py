"""Calls that find little device memory left: what fails reports it and leaves the context as it was, and
what is there for speed alone is left out before a call fails. The lattice is 48^4 (a vector of FP64 is 1.0 GB), so that hundreds of MB stay free for the CUDA runtime
while an allocation of the library does not fit. Links are the identity.

Bars: two evaluations with another order of the shift updates differ by rounding, 1e-11 in FP64 and
float-float, 2e-5 in FP32 (as for the other tests of the update order)."""
import contextlib

import numpy as np
import pytest

import synth

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


# vectors of a multishift solve with n poles and rings of one (n + 3), in units of an FP64 vector
POLES = 4
SIGNS = {ovl.OVL_ARITH_FP64: (1.0, 1e-11), ovl.OVL_ARITH_FF: (1.0, 1e-11), ovl.OVL_ARITH_FP32: (0.5, 2e-5)}


@pytest.mark.parametrize("arith", list(SIGNS))
def test_sign_with_room_for_the_smallest_rings(arith):
    size, tol = SIGNS[arith]
    gen = torch.Generator("cuda")
    gen.manual_seed(51)
    b = torch.view_as_complex(torch.randn((V, 4, 3, 2), dtype=torch.float64, device="cuda", generator=gen))
    ref, out = torch.empty_like(b), torch.empty_like(b)
    op = _op(n_poles=POLES)
    op.sign_apply_arith(ref, b, 1e-5, arith)
    op.close()
    op = _op(n_poles=POLES)
    op.wilson_apply_arith(out, b, -1.0, arith)   # what the call needs besides
    f = ovl.lib().sign_apply_arith
    with scarce(int((POLES + 3 + 0.8) * size * VEC)):
        assert status(f, op, out, b, 1e-5, arith) == ovl.OVL_OK
    out -= ref
    assert (out.norm() / ref.norm()).item() < tol
    op.close()


def test_batch_with_room_for_the_smallest_rings():
    b = torch.randn((2, V, 4, 3), dtype=torch.complex128, device="cuda")
    ref, out = torch.empty_like(b), torch.empty_like(b)
    op = _op(n_poles=POLES)
    op.ovl_apply_n(ref, b, 2, 1e-5)
    op.close()
    op = _op(n_poles=POLES)
    op.wilson_apply_n(out, b, 2, -1.0)
    with scarce(int((2 * (POLES + 3) + 0.8) * VEC)):
        assert status(ovl.lib().ovl_apply_n, op, out, b, 2, 1e-5) == ovl.OVL_OK
    out -= ref
    assert (out.norm() / ref.norm()).item() < 1e-11
    op.close()


@pytest.mark.parametrize("n", [1, 3])
def test_budget_of_the_smallest_rings_admits(n):
    """A budget that holds a request with rings of one serves it."""
    dims = (8, 8, 8, 8)
    U = synth.gauge_field(dims, 0.5, 52, stout_steps=3)
    p = ovl.params_default(precond=ovl.OVL_PREC_RECURSIVE, precision=ovl.OVL_MIXED_FP32, rhs_block=4)
    one, batch = 6 * 1.5, 2 * 1.5 * (n if n > 1 else 0)   # vectors of the larger rings, FP64 and half as much in FP32
    budget = ovl.request_bytes(dims, n, p) - int(1.1 * (one + batch) * 8 ** 4 * 192) + (1 << 20)
    b = synth.rhs_gaussian(dims, 53, n_rhs=n)
    x = np.zeros_like(b)
    srv = ovl.Server(slots=1, hbm_budget=budget)
    res = srv.wait(srv.submit(U, dims, 1.0, 0.05, b, x, n, 1e-8, p))
    srv.close()
    assert res["status"] == ovl.OVL_OK, res["message"]
    op = ovl.Overlap(U, dims, 1.0, 0.05, p)
    for k in range(n):
        ax = np.empty_like(x[k])
        op.ovl_apply(ax, x[k], 1e-12)
        assert np.linalg.norm(b[k] - ax) / np.linalg.norm(b[k]) < 1.5e-8
    op.close()


def test_served_batch_in_parts_gives_the_same_bits():
    """The float-float batch of a served request whose vectors don't fit all at once."""
    dims, n = (16, 16, 16, 16), 4
    U = torch.from_numpy(synth.gauge_field(dims, 0.5, 54, stout_steps=2, device="cuda")).cuda()
    b = torch.from_numpy(synth.rhs_gaussian(dims, 55, n_rhs=n)).cuda()
    p = ovl.params_default(precond=ovl.OVL_PREC_RECURSIVE, precision=ovl.OVL_MIXED_FP32, rhs_block=n, restart=8,
                           restart_inner=16, prec_restart=8, lambda_min=0.15, lambda_max=8.0, m0_prec=0.0, relax_factor=0.3)
    vec = 16 ** 4 * 192

    def served(left):
        x = torch.zeros_like(b)
        srv = ovl.Server(slots=1)
        with scarce(left) if left else contextlib.nullcontext():
            free = torch.cuda.mem_get_info()[0]
            res = srv.wait(srv.submit(U, dims, 1.0, 0.05, b, x, n, 1e-9, p, gauge_key=7))
            used = free - torch.cuda.mem_get_info()[0]   # the resident context still holds its memory
        srv.close()
        assert res["status"] == ovl.OVL_OK, res["message"]
        return x, used

    ref, used = served(0)
    batch = n * (2 * 2 + 2 + 19) * vec   # the float-float batch's vectors: 20 poles, rings of two
    assert used > batch
    x, less = served(used - batch // 4)
    assert less < used - batch // 4
    assert torch.equal(x, ref)
