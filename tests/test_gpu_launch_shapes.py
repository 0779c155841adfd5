"""The automatic evaluation launch shape against the FP64 CPU oracle where it can go wrong: one particle, fewer
particles than lanes, ragged i-tiles and j-chunks, one active particle.  Tolerances are the parity bounds of the
precisions (FP64 1e-12 of |ref|, mixed 1e-6 and EX 1e-12 of sum_j |T_ij|, EX on the double words it holds)."""
import numpy as np
import pytest

import nb_inputs as ni
import oracle as O
from nbhelp import check_parity, nb_gpu

pytestmark = pytest.mark.gpu


def dw(q):
    q = np.asarray(q, dtype=np.float64)
    hi = q.astype(np.float32).astype(np.float64)
    return hi + (q - hi).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("prec", [0, 1, 3])
@pytest.mark.parametrize("n,n_act", [(1, 1), (5, 5), (33, 33), (257, 256), (1025, 129), (4099, 1), (4099, 2049)])
def test_automatic_shape_matches_oracle(prec, n, n_act):
    nb = nb_gpu()
    eps = 1e-3
    m, x, v = ni.plummer(n, 70 + n, imf="salpeter")
    a = ni.random_state(n, 71, scale=2.0)
    if prec == 3:
        m, x, v, a = (dw(q) for q in (m, x, v, a))
    act = ni.active_subset(n, n_act, 72)
    g = nb.NBody(m, x, v, eps, precision=prec, start_forces=False)
    g.set_state({"a": a})
    g.predict(0.0)
    got = g.evaluate(act)
    g.close()
    ref = O.evaluate(m, x, v, a, eps, act)
    kap = O.evaluate_kappa(m, x, v, a, eps, act) if prec else (None,) * 3
    for gq, rq, kq in zip(got, ref, kap):
        assert check_parity(min(prec, 1), gq, rq, kq, tol_mixed=1e-6 if prec == 1 else 1e-12) <= 1.0
