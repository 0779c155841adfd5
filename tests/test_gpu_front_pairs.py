"""Block steps with large active sets: the active particles among themselves by unordered pairs, against the others
by ordered ones (`nb_step`), against the evaluation of the same list after an ordinary prediction.  Both lie within
the parity bounds of the FP64 sums (FP64 1e-12, mixed 1e-6, EX 1e-12, in units of sum_j |T_ij|), so they differ by at
most twice those."""
import numpy as np
import pytest

import nb_inputs as ni
from nbhelp import nb_gpu

pytestmark = pytest.mark.gpu


# the others: none but a part of a 16-byte row, one row, some, most; odd counts; tiles' edges
@pytest.mark.parametrize("prec,n,n_act", [(0, 1201, 1200), (0, 2501, 2498), (0, 4097, 4093), (0, 4097, 2305), (0, 9000, 4097),
                                          (1, 12001, 11998), (1, 12001, 11993), (1, 20002, 17409), (1, 40000, 20481),
                                          (3, 5001, 4999), (3, 8193, 8188), (3, 8193, 7777), (3, 16400, 8001)])
def test_step_matches_listed_evaluation(prec, n, n_act):
    nb = nb_gpu()
    m, x, v = ni.plummer(n, 90, imf="salpeter")
    act = ni.active_subset(n, n_act, 91)
    rest = np.setdiff1d(np.arange(n), act)
    late = np.arange(n) >= n // 2  # the particles' own times differ
    t, dt = np.where(late, 2.0 ** -9, 0.0), np.where(late, 2.0 ** -9, 2.0 ** -8)
    t[rest] *= 2.0
    dt[rest] = np.where(late[rest], 2.0 ** -8, 2.0 ** -7)
    st = {"a": ni.random_state(n, 92, scale=2.0), "j": ni.random_state(n, 93, scale=1.0),
          "s": ni.random_state(n, 94, scale=1.0), "c": np.zeros((n, 3)), "t": t, "dt": dt}
    g = nb.NBody(m, x, v, 1e-4, precision=prec, start_forces=False)
    g.set_state(st)
    g.predict(2.0 ** -8)
    ref = g.evaluate(act)
    kap = g.evaluate_kappa(act)
    l0 = g.counters()
    tn, na = g.step()
    l1 = g.counters()
    assert (tn, na) == (2.0 ** -8, n_act)
    np.testing.assert_array_equal(g.active(), act)
    assert l1[1] - l0[1] == float(n) * n_act
    got = g.state()
    # one active: the ordered kernel alone
    g.set_state({**st, "t": np.zeros(n), "dt": np.where(np.arange(n) == 3, 2.0 ** -8, 2.0 ** -7)})
    l2 = g.counters()
    g.step()
    assert l1[0] - l0[0] > g.counters()[0] - l2[0]  # took the pairs
    g.close()
    tol = 2.0 * (1e-6 if prec == 1 else 1e-12)
    for key, r, k in zip("ajs", ref, kap):
        assert np.all(np.abs(got[key][act] - r) <= tol * k[:, None]), key
    for key in "ajs":
        np.testing.assert_array_equal(got[key][rest], st[key][rest])
