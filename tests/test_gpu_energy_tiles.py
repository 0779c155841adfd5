"""nb_energy against the oracle at the edges of its tiles (32 particles below 6144, 128 from there, odd and even
tile counts) and beyond the FP32 range of the reciprocal square root's estimate.  Tolerance: the sums add terms of
one sign, a chain of at most 128 within a tile, at most T/2 tiles and a tree, each rounding 2^-53, and the
terms carry a few roundings: (128 + T/2 + 32) 2^-53 < 5e-14 relative at these sizes."""
import math

import numpy as np
import pytest

import nb_inputs as ni
import oracle as O
from nbhelp import nb_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 65, 1000, 6143, 6144, 6273])
def test_energy_matches_oracle_at_tile_edges(n):
    nb = nb_gpu()
    m, x, v = ni.plummer(n, 90 + n, imf="salpeter")
    g = nb.NBody(m, x, v, 1e-3, start_forces=False)
    ek, ep = g.energy()
    again = g.energy()
    g.close()
    ekr, epr = O.energy(m, x, v, 1e-3)
    assert (ek, ep) == again
    assert abs(ek - ekr) <= 5e-14 * abs(ekr) and abs(ep - epr) <= 5e-14 * abs(epr)


@pytest.mark.parametrize("far", [1e18, 1e19, 1e25, 1e150])
def test_energy_of_distant_particles(far):
    nb = nb_gpu()
    m = np.array([0.5, 0.25, 0.25])
    x = np.array([[0.0, 0.0, 0.0], [0.0, far, 0.0], [3e-3, 0.0, 4e-3]])
    g = nb.NBody(m, x, np.zeros((3, 3)), 1e-6, start_forces=False)
    _, ep = g.energy()
    g.close()
    assert ep == pytest.approx(-0.125 / math.sqrt(25e-6 + 1e-12), rel=1e-14)
    m = np.array([0.5, 0.25])
    g = nb.NBody(m, x[:2], np.zeros((2, 3)), 1e-6, start_forces=False)
    _, ep = g.energy()
    g.close()
    assert ep == pytest.approx(-0.125 / far, rel=1e-14)
