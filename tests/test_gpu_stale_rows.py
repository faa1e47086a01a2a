"""Right-hand sides of a batch that are done while others go on: their vectors are not written any more and
may hold anything, NaN among it, which must not reach a status or an answer."""
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


@pytest.mark.parametrize("words", [12 * 16, 12 * 4096])
def test_multishift_leaves_rows_without_work_alone(lib, words):
    gen = torch.Generator("cuda")
    gen.manual_seed(11)
    b = torch.randn((4, 2 * words), dtype=torch.float64, device="cuda", generator=gen)
    b[1] = float("nan")
    b[3] = float("inf")
    skip, status, bb = (ctypes.c_int * 4)(0, 1, 0, 1), (ctypes.c_int * 4)(), (ctypes.c_double * 4)()
    torch.cuda.synchronize()
    assert lib.t_ms_init(4, ctypes.c_long(words), P(b), skip, status, bb) == 0
    assert list(status) == [0, 0, 0, 0]
    for y in (0, 2):
        assert abs(bb[y] / b[y].square().sum().item() - 1) < 1e-13


@pytest.mark.parametrize("add", [0, 1])
@pytest.mark.parametrize("n", [24 * 16, 24 * 5000])
def test_solution_from_own_columns(lib, n, add):
    """Rows of 5, 2, 0 and 3 columns; the basis past a row's columns is NaN. Bar: 20 roundings of numbers up to
    40 (sums of five products of Gaussian numbers)."""
    m, cols = 5, [5, 2, 0, 3]
    gen = torch.Generator("cuda")
    gen.manual_seed(12)
    v = torch.randn((m, 4, n // 2), dtype=torch.complex128, device="cuda", generator=gen)
    c = torch.randn((4, m), dtype=torch.complex128, device="cuda", generator=gen)
    x = torch.randn((4, n // 2), dtype=torch.complex128, device="cuda", generator=gen)
    ref = x * add
    for y, k in enumerate(cols):
        ref[y] += (c[y, :k, None] * v[:k, y]).sum(0)
        v[k:, y] = complex(float("nan"), float("nan"))
        c[y, k:] = 0
    torch.cuda.synchronize()
    assert lib.t_gs_combine_f64(P(v), ctypes.c_long(4 * n), m, P(c), (ctypes.c_int * 4)(*cols), P(x), add, ctypes.c_long(n),
                                4) == 0
    assert (x - ref).abs().max().item() < 20 * 40 * 2.0 ** -53
