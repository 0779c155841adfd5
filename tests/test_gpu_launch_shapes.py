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


# sizes at the edges of the tiles (mixed 256, 512, 768 particles, EX 64 to 256, FP64 32 to 128), even and odd
# tile counts, a last tile of one particle, several parts of a j-tile and several offsets per block
@pytest.mark.parametrize("prec,n", [(1, 4096), (1, 5121), (1, 7000), (1, 8192), (1, 16129), (1, 70000),
                                    (0, 1000), (0, 1025), (0, 2049), (0, 4096), (0, 8193),
                                    (3, 2000), (3, 3001), (3, 4096), (3, 8193), (3, 16641)])
def test_all_particles_matches_listed_particles(prec, n):
    """evaluate(None) may take each unordered pair once; the same particles given as a device list do not.  Both
    against the FP64 sums: the parity bound in units of sum_j |T_ij| on a sample, and the whole set to twice it."""
    nb = nb_gpu()
    import torch
    eps = 1e-4
    m, x, v = ni.plummer(n, 80, imf="salpeter")
    a = ni.random_state(n, 81, scale=2.0)
    if prec == 3:
        m, x, v, a = (dw(q) for q in (m, x, v, a))
    g = nb.NBody(m, x, v, eps, precision=prec, start_forces=False)
    g.set_state({"a": a})
    g.predict(0.0)
    got = g.evaluate(None)
    again = g.evaluate(np.arange(n, dtype=np.int32))
    listed = [q.cpu().numpy() for q in g.evaluate(torch.arange(n, dtype=torch.int32, device="cuda"), out="device")]
    kap = g.evaluate_kappa()
    g.close()
    tol = {0: 1e-13, 1: 1e-6, 3: 1e-12}[prec]
    pick = np.unique(np.concatenate([np.arange(0, n, n // 61), [n - 1]])).astype(np.int32)
    ref = O.evaluate(m, x, v, a, eps, pick)
    okap = O.evaluate_kappa(m, x, v, a, eps, pick)
    for gq, aq, lq, kq, rq, oq in zip(got, again, listed, kap, ref, okap):
        np.testing.assert_array_equal(gq, aq)       # the same list: the same evaluation, deterministic
        assert check_parity(1, gq[pick], rq, oq, tol_mixed=tol) <= 1.0
        assert (np.abs(gq - lq).max(axis=1) / kq).max() <= 2 * tol
