"""The FP32 Schwarz application as the batched solvers make it: several right-hand sides, some of them left
out, even and odd numbers of blocks per direction, blocks of 2^4 sites (which have a
form of their own) and larger ones, one and several cycles. Each row against the oracle's smoother, 5e-6 relative
as for one right-hand side; a row that is left out is zero."""
import ctypes

import numpy as np
import pytest

import synth
from oracle import sap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from internals import load  # noqa: E402


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((6, 4, 4, 4), (2, 2, 2, 2)), ((8, 4, 4, 8), (4, 2, 2, 4)),
                                        ((4, 8, 12, 4), (2, 4, 4, 2)), ((8, 8, 8, 8), (4, 4, 4, 4)),
                                        ((12, 8, 8, 4), (4, 4, 4, 2))])
@pytest.mark.parametrize("act", [(1,), (1, 0, 1)])
@pytest.mark.parametrize("cycles", [1, 3])
def test_rows_match_oracle(dims, block, act, cycles):
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    lib = load()
    n, m0, mr = len(act), -0.3, 4
    U = synth.gauge_field(dims, 0.5, 91 + sum(dims), stout_steps=1)
    v = synth.rhs_gaussian(dims, 92, n_rhs=n)
    ud, vd = torch.from_numpy(U).cuda(), torch.from_numpy(v).cuda()
    out = torch.zeros_like(vd)
    torch.cuda.synchronize()
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    I4 = ctypes.c_int * 4
    assert lib.t_sap_rows_f32(I4(*dims), P(ud), I4(*block), P(vd), P(out), (ctypes.c_char * n)(*act), n, ctypes.c_double(m0),
                              cycles, mr) == 0
    for y in range(n):
        got = out[y].cpu().numpy()
        if not act[y]:
            assert not got.any()
            continue
        ref = sap.sap_apply(U, dims, m0, v[y], block, cycles, mr)
        assert np.linalg.norm(got - ref) < 5e-6 * np.linalg.norm(ref), y
