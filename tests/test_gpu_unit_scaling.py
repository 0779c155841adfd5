"""Complete active sets in units far from one: lengths times L, velocities times V and masses times L V^2 (G = 1) scale
acceleration by V^2 / L, jerk by V^3 / L^2 and snap by V^4 / L^3.  L and V are powers of two that keep every operand of
the ordinary pair term (m q) q^2 and its sums within FP32's normal range, so the parity bounds of the precisions
(mixed 1e-6, EX 1e-12, of sum_j |T_ij|) hold as they do for L = V = 1.  The cube of 1 / r alone leaves that range:
2^-150 at unit distance for L = 2^50, and its low word below 2^-144 for L = 2^40."""
import numpy as np
import pytest

import nb_inputs as ni
import oracle as O
from nbhelp import check_parity, nb_gpu

pytestmark = pytest.mark.gpu


def dw(q):
    hi = q.astype(np.float32).astype(np.float64)
    return hi + (q - hi).astype(np.float32).astype(np.float64)


# sizes that take the ordinary kernel and sizes that take unordered pairs, tile edges among them
@pytest.mark.parametrize("prec,L,V", [(1, 50, 37), (1, 40, 30), (1, -24, -18), (2, 50, 37), (3, 40, 30), (3, -24, -18)])
@pytest.mark.parametrize("n", [600, 4097, 8192])
def test_scaled_units_keep_the_bounds(prec, L, V, n):
    nb = nb_gpu()
    lu, vu = 2.0 ** L, 2.0 ** V
    m, x, v = ni.plummer(n, 40 + n, imf="salpeter")
    a = ni.random_state(n, 41, scale=2.0)
    if prec == 2:  # single-precision positions
        x = x.astype(np.float32).astype(np.float64)
    if prec == 3:
        m, x, v, a = (dw(q) for q in (m, x, v, a))
    eps = 2.0 ** -10
    m, x, v, a, eps = m * (lu * vu * vu), x * lu, v * vu, a * (vu * vu / lu), eps * lu
    g = nb.NBody(m, x, v, eps, precision=prec, start_forces=False)
    g.set_state({"a": a})
    g.predict(0.0)
    got = g.evaluate(None)
    g.close()
    pick = np.unique(np.concatenate([np.arange(0, n, n // 61), [n - 1]])).astype(np.int32)
    ref = O.evaluate(m, x, v, a, eps, pick)
    kap = O.evaluate_kappa(m, x, v, a, eps, pick)
    for gq, rq, kq in zip(got, ref, kap):
        assert check_parity(1, gq[pick], rq, kq, tol_mixed=1e-12 if prec == 3 else 1e-6) <= 1.0


# near and far tiles in one launch: the outer half a system of its own scale, its masses as large as its distances ask
@pytest.mark.parametrize("prec,far,heavy", [(1, 45, 60), (3, 30, 50)])
@pytest.mark.parametrize("n", [4500, 8192])
def test_two_scales_keep_the_bounds(prec, far, heavy, n):
    nb = nb_gpu()
    m, x, v = ni.plummer(n, 43 + n, imf="salpeter")
    a = ni.random_state(n, 44, scale=2.0)
    out = np.arange(n) >= n // 2
    x[out] *= 2.0 ** far
    m[out] *= 2.0 ** heavy
    if prec == 3:
        m, x, v, a = (dw(q) for q in (m, x, v, a))
    g = nb.NBody(m, x, v, 2.0 ** -10, precision=prec, start_forces=False)
    g.set_state({"a": a})
    g.predict(0.0)
    got = g.evaluate(None)
    g.close()
    pick = np.unique(np.concatenate([np.arange(0, n, n // 61), [n // 2 - 1, n // 2, n - 1]])).astype(np.int32)
    ref = O.evaluate(m, x, v, a, 2.0 ** -10, pick)
    kap = O.evaluate_kappa(m, x, v, a, 2.0 ** -10, pick)
    for gq, rq, kq in zip(got, ref, kap):
        assert check_parity(1, gq[pick], rq, kq, tol_mixed=1e-12 if prec == 3 else 1e-6) <= 1.0
