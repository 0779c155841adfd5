"""FP64 sums beyond the largest double: infinite, not NaN, by unordered pairs as in the ordinary kernel.

Heavy particles on the right, massless ones at the origin: each term is finite (at most 1e308 x 2 / 5^(3/2)) and 32 of
them add up to more than the largest double along x only.  The other components stay far below it, so they agree
with the listed evaluation to the parity bound."""
import numpy as np
import pytest

from nbhelp import nb_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1000, 2049, 4096])
def test_overflowing_sum_is_infinite(n):
    nb = nb_gpu()
    import torch
    rng = np.random.default_rng(7 + n)
    heavy = np.sort(rng.choice(n, 32, replace=False))
    light = np.setdiff1d(np.arange(n), heavy)
    x = 0.05 * rng.uniform(-1.0, 1.0, (n, 3))
    x[heavy, 0] += 2.0
    m = np.zeros(n)
    m[heavy] = 1e308
    g = nb.NBody(m, x, np.zeros((n, 3)), 1.0, start_forces=False)
    g.predict(0.0)
    got = g.evaluate(None)
    listed = [q.cpu().numpy() for q in g.evaluate(torch.arange(n, dtype=torch.int32, device="cuda"), out="device")]
    g.close()
    for gq, lq in zip(got[1:], listed[1:]):
        np.testing.assert_array_equal(gq[light], 0.0 * lq[light])
    assert np.all(np.isposinf(listed[0][light, 0]))
    assert np.all(np.isposinf(got[0][light, 0]))
    np.testing.assert_allclose(got[0][light, 1:], listed[0][light, 1:], rtol=0.0, atol=1e-12 * 32 * (0.1 * 1e308 / 5.0 ** 1.5))
