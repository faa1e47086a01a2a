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


def multishift(lib, dims, dtype, tps, rows, ring, iters, seed, sigma0=0.01, b=None):
    """ms_probe on random links (and vectors unless given): (scalars [rows][5], t, r, p_0 as [rows][24 V])."""
    V = dims[0] * dims[1] * dims[2] * dims[3]
    gen = torch.Generator("cuda")
    gen.manual_seed(seed)
    u = torch.linalg.qr(torch.complex(*torch.randn((2, 4096, 4, 3, 3), dtype=torch.float64, device="cuda", generator=gen)))[0]
    u = u / torch.linalg.det(u).pow(1 / 3)[..., None, None]
    u = u[torch.randint(0, 4096, (V,), device="cuda", generator=gen)].contiguous()
    if b is None:
        b = torch.randn((rows, 24 * V), dtype=dtype, device="cuda", generator=gen)
    t, r, p = torch.zeros_like(b), torch.zeros_like(b), torch.zeros_like(b)
    scal = (ctypes.c_double * (5 * rows))()
    torch.cuda.synchronize()
    assert lib.t_ms_probe((ctypes.c_int * 4)(*dims), P(u), int(dtype == torch.float64), tps, rows, ring, P(b), iters,
                          ctypes.c_double(sigma0), scal, P(t), P(r), P(p)) == 0
    return torch.tensor(list(scal), dtype=torch.float64).view(rows, 5), b, t, r, p


def squares(x):
    return torch.stack([v.double().square().sum() for v in x]).cpu()


@pytest.mark.parametrize("dims,tps,rows", [((32, 32, 32, 32), 1, 1), ((32, 32, 32, 32), 1, 12), ((32, 32, 32, 32), 4, 3),
                                           ((16, 16, 16, 16), 1, 12), ((6, 4, 10, 8), 1, 5), ((6, 4, 10, 8), 4, 5)])
def test_multishift_sums_f32(lib, dims, tps, rows):
    """||b||^2, ||Q p_0||^2 (from alpha) and ||r_1||^2 of one iteration. One plain FP32 sum runs over a site's
    24 products (four in ||b||^2)."""
    scal, b, t, r, _ = multishift(lib, dims, torch.float32, tps, rows, 2, 1, 31)
    n = b.shape[1]
    assert bool((scal[:, 4] == 0).all())
    bb = squares(b)
    assert (scal[:, 0] / bb - 1).abs().max() < bar(4, n)
    assert (scal[:, 1] / squares(r) - 1).abs().max() < bar(24, n)
    tt = scal[:, 0] / scal[:, 3] - 0.01 * scal[:, 0]
    assert (tt / squares(t) - 1).abs().max() < bar(24, n) + 0.01 * bar(4, n)


@pytest.mark.parametrize("dtype,tps", [(torch.float32, 1), (torch.float32, 4), (torch.float64, 1)])
@pytest.mark.parametrize("dims,rows", [((16, 16, 16, 16), 3), ((6, 4, 10, 8), 12)])
def test_direction_norm_of_a_batch(lib, dtype, tps, dims, rows):
    """||p_0||^2 in alpha of a later iteration of several right-hand sides, with a shift as large as Q^2: it is
    summed from the vector, not carried from iteration to iteration."""
    k, sigma0 = 6, 16.0
    before, b, _, _, p = multishift(lib, dims, dtype, tps, rows, 2, k, 41, sigma0)
    after, _, t, _, _ = multishift(lib, dims, dtype, tps, rows, 2, k + 1, 41, sigma0)
    tt, pp = squares(t), squares(p)
    got = (before[:, 1] / after[:, 3] - tt) / sigma0
    eps = bar(24, b.shape[1]) if dtype == torch.float32 else 1e-14
    assert ((got / pp - 1).abs() < eps * (1 + tt / (sigma0 * pp))).all()


@pytest.mark.parametrize("dtype,tps,dims", [(torch.float64, 1, (14, 12, 12, 12)), (torch.float64, 1, (12, 10, 10, 10)),
                                            (torch.float32, 1, (20, 20, 20, 20)), (torch.float32, 1, (16, 16, 16, 16)),
                                            (torch.float32, 4, (20, 20, 20, 20))])
def test_rows_of_a_batch_cover_the_lattice(lib, dtype, tps, dims):
    """r, t and p_0 of twelve right-hand sides after three iterations against one alone, on either side of the
    size from which block 0 takes sites too. The scalars differ by rounding: 100 units of the arithmetic."""
    _, b, t, r, p = multishift(lib, dims, dtype, tps, 12, 2, 3, 61)
    for y in (0, 11):
        _, _, t1, r1, p1 = multishift(lib, dims, dtype, tps, 1, 2, 3, 61, b=b[y:y + 1].contiguous())
        for x, x1 in ((t[y], t1[0]), (r[y], r1[0]), (p[y], p1[0])):
            assert (x - x1).abs().max() < 100 * torch.finfo(dtype).eps * x1.abs().max()
