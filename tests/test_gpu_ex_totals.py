"""EX totals are FP64: double words (48 bits) hold the terms and sums of at most 512 of them, not the totals over those.

All mass is in two particles, A of mass 1 and B of 2^-49, whose terms meet only in totals.  The sums with and without B
then differ by B's term to one rounding of the total, 2^-53 of it, and B's own error (below 2^-40): the bound below
doubles the rounding.  A total in double words would round at 2^-49 or coarser, as much as B's term itself."""
import numpy as np
import pytest

import nb_inputs as ni
import oracle as O
from nbhelp import nb_gpu

pytestmark = pytest.mark.gpu

TINY = 2.0 ** -49


def check(with_b, without_b, term):
    for s1, s0, t in zip(with_b, without_b, term):
        assert np.abs(s0).min() > 0.0
        bound = 2.0 ** -52 * np.abs(s0) + 2.0 ** -40 * np.linalg.norm(t, axis=1, keepdims=True)
        assert np.all(np.abs((s1 - s0) - t) <= bound)


def masses(n, a, b):
    m = np.zeros((2, n))
    m[:, a] = 1.0
    m[1, b] = TINY
    mb = np.zeros(n)
    mb[b] = TINY
    return m[0], m[1], mb


# all particles active by unordered pairs, A and B 512 particles apart; jobs of one offset and of several (the larger
# sizes: four offsets of 256 particles), a ragged last tile
@pytest.mark.parametrize("n", [4096, 8193, 49179, 50052])
@pytest.mark.parametrize("a", [0, 1000])
def test_pair_totals(n, a):
    nb = nb_gpu()
    _, x, v = ni.plummer(n, 50)
    acc = ni.random_state(n, 51)
    b = a + 512
    m0, m1, mb = masses(n, a, b)
    sums = []
    for m in (m0, m1):
        g = nb.NBody(m, x, v, 1e-2, precision=3, start_forces=False)
        g.set_state({"a": acc})
        g.predict(0.0)
        sums.append(g.evaluate(None))
        g.close()
    others = np.setdiff1d(np.arange(0, n, max(1, n // 400)), [a, b]).astype(np.int32)
    check([q[others] for q in sums[1]], [q[others] for q in sums[0]], O.evaluate(mb, x, v, acc, 1e-2, others))


# the resident stepper: A and B are the two halves of one lane's packed sums
@pytest.mark.parametrize("seed", range(8))
def test_stepper_lanes(seed):
    nb = nb_gpu()
    n, h = 4, 2.0 ** -7
    x, v, acc = (ni.random_state(n, 3 * seed + q + 100) for q in range(3))
    m0, m1, mb = masses(n, 2, 3)
    sums = []
    for m in (m0, m1):
        g = nb.NBody(m, x, v, 1e-2, precision=3, start_forces=False, dt_max=h)
        g.set_state({"a": acc, "dt": np.full(n, h)})
        assert g.run_until(h)[0] == 1
        st = g.state()
        sums.append([st[k][:2] for k in "ajs"])
        g.close()
    xp, vp = x + h * (v + h / 2 * acc), v + h * acc
    check(sums[1], sums[0], O.evaluate(mb, xp, vp, acc, 1e-2, np.arange(2, dtype=np.int32)))
