"""Rounding errors of the FP32 kernels' sums of squares and dot products against FP64 sums of the same
vectors, at sizes where a thread adds many terms.

Bars. A sum is made of plain FP32 sums of at most `chain` products; each has a relative error of about
2^-24 sqrt(chain) / 3 of random sign (2^-24 / sqrt(3) the standard deviation of one rounding to nearest,
chain / 3 the mean square of the partial sums), and the groups are added with smaller errors, so that the
whole sum's is that over the root of the number of groups. The bars are six times that.
"""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from internals import load  # noqa: E402


@pytest.fixture(scope="module")
def lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return load()


def P(t):
    return ctypes.c_void_p(t.data_ptr())


def L(k):
    return ctypes.c_long(k)


def bar(chain, terms):
    return 6 * 2.0 ** -24 * chain ** 0.5 / 3 / (terms / chain) ** 0.5


@pytest.mark.parametrize("sites,m,rows", [(32 ** 4, 1, 1), (32 ** 4, 16, 1), (32 ** 4, 30, 1), (24 ** 4, 80, 1),
                                          (16 ** 4, 32, 12), (8 ** 4, 5, 3), (16, 2, 2)])
def test_gram_schmidt_dots_f32(lib, sites, m, rows):
    n = 24 * sites
    gen = torch.Generator("cuda")
    gen.manual_seed(21)
    v = torch.randn((m, rows, n), dtype=torch.float32, device="cuda", generator=gen)
    w = torch.randn((rows, n), dtype=torch.float32, device="cuda", generator=gen)
    rec = 2 * m + 6
    out = torch.zeros((rows, rec), dtype=torch.float64, device="cuda")
    part = torch.empty(128 * 256 * 2, dtype=torch.float64, device="cuda")
    cnt = torch.zeros(32, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert lib.t_gs_dots_f32(P(v), L(rows * n), m, P(w), L(n), rows, P(out), P(part), P(cnt)) == 0
    tol = bar(16, n)
    for y in range(rows):
        wd = w[y].double()
        ww = wd.square().sum()
        assert abs(out[y, 2 * m] / ww - 1) < tol
        wc = torch.view_as_complex(wd.view(-1, 2))
        for i in range(m):
            vd = v[i, y].double()
            h = torch.vdot(torch.view_as_complex(vd.view(-1, 2)), wc)
            err = abs(complex(out[y, 2 * i].item(), out[y, 2 * i + 1].item()) - h.item())
            assert err < tol * (ww.sqrt() * vd.norm()).item()
