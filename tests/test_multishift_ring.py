"""The order of the shifted-direction updates in the multishift kernels, in numpy FP64 on a small Hermitian
matrix: residuals and base directions in rings of `ring` vectors that are written over, the coefficients
of the pending iterations kept, and the updates of all of them done together in every ring-th iteration
and at a chunk's end. A ring slot that is written over before its update is done, a coefficient of the wrong
iteration or a shift that is updated after its last iteration shows against the iteration-by-iteration
form (same updates, other order of the additions to y: 1e-12 relative)."""
import numpy as np
import pytest

from test_multishift_schedule import _problem, _three_kernel, _zeta_next


def _ring(A, b, sigma, w, crit, tol, iters, drop, ring, chunk):
    n = len(sigma)
    nan = np.full(len(b), np.nan + 0j)
    r, p0 = [nan.copy() for _ in range(ring)], [nan.copy() for _ in range(ring)]
    r[0], p0[0], y = b.copy(), b.copy(), b.copy()
    P = [None] + [b.copy() for _ in range(n - 1)]
    rr = pp = bb = np.vdot(b, b).real
    z, zp, ap, bp = np.ones(n), np.ones(n), 1.0, 0.0
    active, pending, done = [True] * n, [], False   # pending: (wa, bl) of each shift that took part
    for k in range(iters):
        p = p0[k % ring]
        t = A @ p
        a = rr / (np.vdot(p, t).real + sigma[0] * pp)
        new = r[k % ring] - a * (t + sigma[0] * p)
        r[(k + 1) % ring] = new                     # in place for ring = 1
        rr_new = np.vdot(new, new).real
        beta = rr_new / rr
        coef, live = {}, False
        for l in range(n):
            if not active[l]:
                continue
            zn = 1.0 if l == 0 else _zeta_next(z[l], zp[l], a, ap, bp, sigma[l] - sigma[0])
            coef[l] = (w[l] * (a * zn), beta * (zn / z[l] if z[l] != 0.0 else 0.0))
            zp[l], z[l] = z[l], zn
            if not drop or crit[l] * abs(zn) * np.sqrt(rr_new) > tol * np.sqrt(bb):
                live = True
            elif l > 0:
                active[l] = False
        pending.append(coef)
        done = not live
        ap, bp, pp, rr = a, beta, rr_new + beta * beta * pp, rr_new
        in_chunk = k % chunk
        if (in_chunk + 1) % ring == 0 or in_chunk == chunk - 1 or done or k == iters - 1:
            m = len(pending)
            rs = [r[(k + 1 - m + 1 + d) % ring] for d in range(m)]
            ps = [p0[(k + 1 - m + d) % ring] for d in range(m)]
            for d in range(m):
                y = y + pending[d][0][0] * ps[d]
            nxt = rs[-1] + beta * ps[-1]
            for l in range(1, n):
                for d in range(m):
                    if l in pending[d]:
                        y = y + pending[d][l][0] * P[l]
                        P[l] = rs[d] + pending[d][l][1] * P[l]
            p0[(k + 1) % ring] = nxt
            pending = []
        else:
            p0[(k + 1) % ring] = r[(k + 1) % ring] + beta * p
        if done:
            break
    return y


@pytest.mark.parametrize("drop", [False, True])
@pytest.mark.parametrize("ring", [1, 2, 4])
@pytest.mark.parametrize("chunk", [1, 2, 3, 5, 8, 64])
def test_ring_schedule_is_the_same_sum(ring, chunk, drop):
    A, b, sigma, w, crit = _problem()
    iters = 400 if drop else 150
    plain = _three_kernel(A, b, sigma, w, crit, 1e-10, iters, drop)
    y = _ring(A, b, sigma, w, crit, 1e-10, iters, drop, ring, chunk)
    assert np.linalg.norm(y - plain) < 1e-12 * np.linalg.norm(plain)
