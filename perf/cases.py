"""The work that users of the library have it do, as cases that can be timed and compared.

A case is one call of a public entry point on inputs that a program has in hand: a context on a
gauge field (made once per field, as every program does) and right-hand sides on the GPU.
The calls are the library's own layers, from one Wilson operator to a whole overlap solve:

    wilson   D_W on one or several vectors, in FP64, float-float or FP32 arithmetic
    sign     sign(Q) of one vector, in FP64, float-float or FP32 arithmetic
    overlap  D_N of several vectors in lock-step (FP64)
    precond  the inexact Wilson solve that preconditions the overlap solvers (FP32, Schwarz)
    solve    the overlap solve itself, FP64 outer and lower-precision inner iterations

Lattices run from 4^4 to 64 x 32^3, the smallest and the largest of the workloads that the
library is tested and benchmarked on, with unequal extents and numbers of right-hand sides
among them. Links are exp(i 0.5 H) of random traceless Hermitian H; the calls that depend on
the spectrum of Q get them smoothed by three stout steps, as the solves do everywhere else.

Answers that were computed in FP32 arithmetic are kept as complex64, the precision that a
program which asks for that arithmetic has use for; all others are complex128 as returned.
"""
import math

import numpy as np
import torch

import paper_1410_7170_gb300 as ovl

ARITH = {"fp64": ovl.OVL_ARITH_FP64, "ff": ovl.OVL_ARITH_FF, "fp32": ovl.OVL_ARITH_FP32}
PRECISION = {"fp32": ovl.OVL_MIXED_FP32, "half": ovl.OVL_MIXED_HALF}
RHO, MU = 1.0, 0.01


def _case(call, dims, rhs=1, arith="fp64", tol=0.0, name=None):
    c = {"call": call, "l0": dims[0], "l1": dims[1], "l2": dims[2], "l3": dims[3], "rhs": rhs, "arith": arith, "tol": tol}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a single operator on the smallest lattice that the tests use: a program that builds its
        # own solver calls it thousands of times
        _case("wilson", (4, 4, 4, 4), name="wilson_4"),
        # FP64 operator on a lattice of unequal extents, no power of two among them
        _case("wilson", (22, 6, 14, 10), name="wilson_ragged"),
        # the operator in the arithmetic of the solver's tight products
        _case("wilson", (24, 24, 24, 24), arith="ff", name="wilson_ff_24"),
        # the operator in the preconditioner's arithmetic on the largest configuration
        _case("wilson", (64, 32, 32, 32), arith="fp32", name="wilson_f32_64"),
        # twelve spin-colour sources of one propagator
        _case("wilson", (32, 32, 32, 32), rhs=12, arith="fp32", name="wilson12_f32_32"),
        # sign function in plain FP64 on the smallest lattice of the serving mix
        _case("sign", (8, 8, 8, 8), tol=1e-12, name="sign_f64_8"),
        # the outer solver's tight sign product
        _case("sign", (16, 16, 16, 16), arith="ff", tol=1e-10, name="sign_ff_16"),
        # a relaxed sign product of the inner solver on a lattice that does not fit the L2 cache
        _case("sign", (32, 32, 32, 32), arith="fp32", tol=1e-4, name="sign_f32_32"),
        # overlap operator on several vectors at once
        _case("overlap", (8, 8, 8, 8), rhs=5, tol=1e-10, name="overlap5_f64_8"),
        # the Wilson preconditioner as the overlap solvers call it
        _case("precond", (16, 16, 16, 16), arith="fp32", tol=1e-1, name="precond_16"),
        # a small served request with several right-hand sides, and the benchmark's solve
        _case("solve", (16, 8, 8, 8), rhs=4, arith="fp32", tol=1e-10, name="solve4_16_8"),
        _case("solve", (16, 16, 16, 16), arith="fp32", tol=1e-10, name="solve_16"),
    ]


def _dims(rng, low, high, step):
    """Extents (multiples of step) of a lattice whose volume is spread over its logarithm."""
    want = math.exp(rng.uniform(math.log(low), math.log(high)))
    while True:
        d = [step * rng.randint(max(1, 4 // step), max(2, 64 // step)) for _ in range(4)]
        k = (want / math.prod(d)) ** 0.25
        d = tuple(max(max(4, step), step * round(x * k / step)) for x in d)
        if low <= math.prod(d) <= high and max(d) <= 8 * min(d):
            return d


def draw(rng):
    call = rng.choice(["wilson", "wilson", "sign", "sign", "overlap", "precond", "solve"])
    if call == "wilson":
        arith = rng.choice(["fp64", "ff", "fp32"])
        rhs = 1 if arith == "ff" else rng.choice([1, 1, rng.randint(2, 12)])
        top = {"fp64": 32 ** 4, "ff": 24 ** 4, "fp32": 64 * 32 ** 3}[arith]
        return _case(call, _dims(rng, 4 ** 4, top // rhs, 2), rhs, arith)
    if call == "sign":
        arith = rng.choice(["fp64", "ff", "fp32"])
        top = {"fp64": 16 ** 4, "ff": 24 ** 4, "fp32": 32 ** 4}[arith]
        tol = rng.choice([1e-2, 1e-3, 1e-4, 1e-5] if arith == "fp32" else [1e-8, 1e-10, 1e-12])
        return _case(call, _dims(rng, 8 ** 4, top, 2), 1, arith, tol)
    if call == "overlap":
        rhs = rng.randint(2, 12)
        return _case(call, _dims(rng, 6 ** 4, 16 ** 4 // rhs, 2), rhs, "fp64", rng.choice([1e-8, 1e-10]))
    if call == "precond":
        return _case(call, _dims(rng, 8 ** 4, 32 ** 4, 4), 1, "fp32", rng.choice([1e-1, 1e-2]))
    rhs = rng.choice([1, 1, 2, 3, 4])
    return _case(call, _dims(rng, 8 ** 4, 16 ** 4 if rhs == 1 else 32768 // rhs, 4), rhs, rng.choice(["fp32", "half"]), 1e-10)


# ------------------------------------------------------------------ inputs
def _mul(a, b):
    """Products of 3 x 3 matrices."""
    o = a[..., :, 0:1] * b[..., 0:1, :]
    for k in (1, 2):
        o += a[..., :, k:k + 1] * b[..., k:k + 1, :]
    return o


def _dag(a):
    return a.conj().transpose(-1, -2)


def _exp(z, s):
    """exp of anti-Hermitian 3 x 3 matrices: Taylor series of exp(z / 2^s), squared s times."""
    z = z / 2.0 ** s
    term = z
    o = torch.eye(3, dtype=z.dtype, device=z.device) + z
    for k in range(2, 13):
        term = _mul(term, z) / k
        o += term
    for _ in range(s):
        o = _mul(o, o)
    return o


def _traceless(m):
    """The traceless anti-Hermitian part."""
    b = 0.5 * (m - _dag(m))
    return b - (torch.diagonal(b, dim1=-2, dim2=-1).sum(-1) / 3.0)[..., None, None] * torch.eye(3, dtype=b.dtype, device=b.device)


def _links(dims, gen, stout):
    """[V][4][3][3]: exp(i 0.5 H) of random H, then `stout` stout steps with parameter 0.1."""
    n = tuple(dims) + (4, 3, 3)
    a = torch.complex(torch.randn(n, dtype=torch.float64, device="cuda", generator=gen),
                      torch.randn(n, dtype=torch.float64, device="cuda", generator=gen))
    u = _exp(0.5 * _traceless(1j * a), 4)
    del a
    for _ in range(stout):
        new = torch.empty_like(u)
        for mu in range(4):
            um = u[..., mu, :, :]
            s = torch.zeros_like(um)
            for nu in range(4):
                if nu != mu:
                    un = u[..., nu, :, :]
                    s += _mul(_mul(un, torch.roll(um, -1, nu)), _dag(torch.roll(un, -1, mu)))
                    ub = torch.roll(un, 1, nu)
                    s += _mul(_mul(_dag(ub), torch.roll(um, 1, nu)), torch.roll(ub, -1, mu))
            new[..., mu, :, :] = _mul(_exp(0.1 * _traceless(_mul(s, _dag(um))), 2), um)
        u = new
    return u.reshape(-1, 4, 3, 3).contiguous()


def _spectral(case):
    return case["call"] in ("sign", "overlap", "solve")


def _mass(case):
    """Mass of the Wilson operator: the overlap kernel's, or the preconditioner's."""
    return -0.25 if case["call"] == "precond" else -RHO


def _inputs(case, seed):
    dims = tuple(case["l%d" % m] for m in range(4))
    gen = torch.Generator("cuda")
    gen.manual_seed(seed)
    u = _links(dims, gen, 0 if case["call"] == "wilson" else 3)
    n = (case["rhs"], math.prod(dims), 4, 3)
    b = torch.complex(torch.randn(n, dtype=torch.float64, device="cuda", generator=gen),
                      torch.randn(n, dtype=torch.float64, device="cuda", generator=gen))
    return dims, u, b


def prepare(case, seed):
    dims, u, b = _inputs(case, seed)
    kw = {}
    if not _spectral(case):   # nothing of these calls depends on the interval of |Q|: no estimate
        kw.update(lambda_min=0.05, lambda_max=8.0)
    if case["call"] == "precond":
        kw.update(precision=ovl.OVL_MIXED_FP32, precond=ovl.OVL_PREC_WILSON, m0_prec=-0.25)
    if case["call"] == "solve":
        # the benchmark's parameters: relaxation 0.3, preconditioner mass 0
        kw.update(precision=PRECISION[case["arith"]], precond=ovl.OVL_PREC_RECURSIVE, relax_factor=0.3, m0_prec=0.0)
    # one stream for the library's calls and for what torch does between them
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    op = ovl.Overlap(u, dims, RHO, MU, ovl.params_default(**kw), stream=stream.cuda_stream)
    return {"case": case, "op": op, "b": b, "out": torch.empty_like(b), "stream": stream}


def run(state):
    c, op, b, out = state["case"], state["op"], state["b"], state["out"]
    with torch.cuda.stream(state["stream"]):
        if c["call"] == "wilson":
            if c["rhs"] > 1:
                op.wilson_apply_n_arith(out, b, c["rhs"], -RHO, ARITH[c["arith"]])
            elif c["arith"] == "fp64":
                op.wilson_apply(out, b, -RHO)
            else:
                op.wilson_apply_arith(out, b, -RHO, ARITH[c["arith"]])
        elif c["call"] == "sign":
            if c["arith"] == "fp64":
                op.sign_apply(out, b, c["tol"])
            else:
                op.sign_apply_arith(out, b, c["tol"], ARITH[c["arith"]])
        elif c["call"] == "overlap":
            op.ovl_apply_n(out, b, c["rhs"], c["tol"])
        elif c["call"] == "precond":
            op.wilson_solve(out, b, _mass(c), c["tol"])
        else:
            out.zero_()   # the initial guess
            op.ovl_solve(out, b, c["rhs"], c["tol"])
            return out
        return out.to(torch.complex64) if c["arith"] == "fp32" else out


def work(case):
    """Vectors in and out and the links once; floating-point operations of the Wilson operator (1368
    a site), twice for each step of a conjugate gradient iteration to the tolerance asked for."""
    v = math.prod(case["l%d" % m] for m in range(4))
    link = 4 * 12 * 4 if case["arith"] in ("fp32", "half") else 4 * 18 * 8
    steps = {"wilson": 1.0, "precond": 20.0}.get(case["call"])
    if steps is None:   # condition number of |Q| on these fields: about 13
        steps = 2 * 6.5 * math.log(2 / case["tol"]) * (6 if case["call"] == "solve" else 1)
    return {"bytes": float(v * (2 * 192 * case["rhs"] + link)), "flops": 1368.0 * v * case["rhs"] * steps}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch
def _gammas():
    i2 = np.eye(2)
    sig = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])]
    z = np.zeros((2, 2))
    return [np.block([[z, i2], [i2, z]])] + [np.block([[z, -1j * s], [1j * s, z]]) for s in sig]


def _dw(u, psi, m0):
    """D_W(m0) psi for psi [...]: links u [T][X][Y][Z][4][3][3], psi [T][X][Y][Z][4][3],
    antiperiodic in the first direction."""
    out = (m0 + 4.0) * psi
    for mu, g in enumerate(_gammas()):
        g = torch.tensor(g, dtype=psi.dtype, device=psi.device)
        one = torch.eye(4, dtype=psi.dtype, device=psi.device)
        um = u[..., mu, :, :]
        f = torch.roll(psi, -1, mu)
        b = torch.roll(_mul(psi, um.conj()), 1, mu)   # U^H psi at its own site, then moved on
        if mu == 0:
            f[-1] *= -1
            b[0] *= -1
        f = _mul(f, um.transpose(-1, -2))
        out -= 0.5 * (torch.matmul(one - g, f) + torch.matmul(one + g, b))
    return out


def _zolotarev(k, n):
    """Zolotarev's best approximation of 1 on [1, 1/k], x sum_l w_l / (x^2 + c_l); sn = sin(amplitude) by the AGM."""
    a, b, ratio = 1.0, k, []
    while abs(a - b) > 1e-16 * a and len(ratio) < 40:
        a, b, c = 0.5 * (a + b), math.sqrt(a * b), 0.5 * (a - b)
        ratio.append(c / a)
    quarter = math.pi / (2 * a)

    def amplitude(x):
        phi = 2 ** len(ratio) * a * x
        for q in reversed(ratio):
            phi = 0.5 * (phi + math.asin(q * math.sin(phi)))
        return phi

    c = np.array([math.tan(amplitude(m * quarter / (2 * n))) ** 2 for m in range(1, 2 * n)])   # sn^2 / (1 - sn^2)
    odd, even = c[0::2], c[1::2]
    w = np.array([np.prod(even - odd[m]) / np.prod(np.delete(odd, m) - odd[m]) for m in range(n)])
    x = np.exp(np.linspace(0.0, -math.log(k), 20001))
    r = x * sum(w[m] / (x * x + odd[m]) for m in range(n))
    return 2 * w / (r.max() + r.min()), odd


def _sign(u, psi, accuracy):
    """sign(Q) psi, Q = gamma5 D_W(-RHO): multishift conjugate gradients on Q^2."""
    g5 = torch.tensor([-1.0, -1.0, 1.0, 1.0], dtype=torch.float64, device=psi.device)[:, None]
    low, high = 0.03, 7.001      # |Q| <= |m0 + 4| + 4
    w, c = _zolotarev(low / high, 16 if accuracy > 1e-9 else 28)
    sig = torch.tensor(c * low * low, device=psi.device)
    n = len(c)
    shape = (n,) + (1,) * psi.dim()
    ds = (sig - sig[0])
    x, r = torch.zeros_like(psi), psi.clone()
    p0, ps = psi.clone(), psi.expand((n,) + psi.shape).clone()
    wl = torch.tensor(w * low, device=psi.device)
    z, q = torch.ones(n, dtype=torch.float64, device=psi.device), torch.ones(n, dtype=torch.float64, device=psi.device)
    one = torch.ones((), dtype=torch.float64, device=psi.device)
    al_o, be_o, rr = one, 0 * one, torch.view_as_real(r).square().sum()
    end = accuracy ** 2 * float(rr)
    for k in range(1, 3001):   # z: a shift's residual over the base residual, q: its change in a step
        t = g5 * _dw(u, p0, -RHO)
        ap = g5 * _dw(u, t, -RHO) + sig[0] * p0
        al = rr / (torch.view_as_real(p0) * torch.view_as_real(ap)).sum()
        q = al_o / (al * be_o * (1 - q) + al_o * (1 + ds * al))
        z = z * q
        x += ((wl * al * q).to(psi.dtype).reshape(shape) * ps).sum(0)
        r -= al * ap
        new = torch.view_as_real(r).square().sum()
        be = new / rr
        p0 = r + be * p0
        ps *= (be * q * q).reshape(shape)
        for m in range(n):
            ps[m] += z[m] * r
        al_o, be_o, rr = al, be, new
        if k % 10 == 0 and float(rr) <= end:
            break
    return g5 * _dw(u, x, -RHO)


def exact(case, seed):
    v = math.prod(case["l%d" % m] for m in range(4))
    if case["call"] in ("precond", "solve"):   # an inexact solve; a solve of many sign functions
        return None
    if case["call"] != "wilson" and v * case["rhs"] > (32 if case["arith"] == "fp32" else 24) ** 4:
        return None
    dims, u, b = _inputs(case, seed)
    u = u.reshape(dims + (4, 3, 3))
    out = torch.empty_like(b)
    rho = (-MU / 2 - RHO) / (MU / 2 - RHO)
    for k in range(case["rhs"]):
        psi = b[k].reshape(dims + (4, 3))
        if case["call"] == "wilson":
            y = _dw(u, psi, -RHO)
        else:
            y = _sign(u, psi, 1e-8 if case["arith"] == "fp32" else 1e-14)
            if case["call"] == "overlap":
                y[..., :2, :] *= -1   # gamma5
                y += rho * psi
        out[k] = y.reshape(out[k].shape)
    return out
