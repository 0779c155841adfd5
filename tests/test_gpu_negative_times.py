"""Block steps of a state whose times are negative or pass through zero.

Every time is a dyadic rational and the step criterion looks at a time only through its multiples of the steps, so a
run shifted by a multiple of dt_max takes the same steps with the same arithmetic: log and state agree to the bit with
the unshifted run, device-resident and host-driven."""
import numpy as np
import pytest

import nb_inputs as ni
from nbhelp import nb_gpu

pytestmark = pytest.mark.gpu

DT_MAX = 2.0 ** -5


# 64: every step within the resident stepper; 1000: steps on both sides of its limit
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("device_steps", [True, False])
@pytest.mark.parametrize("n", [64, 1000])
@pytest.mark.parametrize("shift,t_end", [(2 * DT_MAX, 4 * DT_MAX), (32.0, DT_MAX), (4 * DT_MAX, 4 * DT_MAX)])
def test_shifted_run_takes_the_same_steps(prec, device_steps, n, shift, t_end):
    nb = nb_gpu()
    m, x, v = ni.plummer(n, 60 + n)
    runs = []
    for s in (0.0, shift):
        g = nb.NBody(m, x, v, 1e-3, precision=prec, dt_max=DT_MAX, device_steps=device_steps)
        st = g.state()
        g.set_state(dict(st, t=st["t"] - s))
        steps, (lt, ln) = g.run_until(t_end - s, log_cap=8192)
        runs.append((steps, lt + s, ln, g.state()))
        g.close()
    (k0, t0, n0, s0), (k1, t1, n1, s1) = runs
    assert k0 == k1 > 0
    np.testing.assert_array_equal(t1, t0)
    np.testing.assert_array_equal(n1, n0)
    np.testing.assert_array_equal(s1["t"] + shift, s0["t"])
    for key in ("x", "v", "a", "j", "s", "c", "dt"):
        np.testing.assert_array_equal(s1[key], s0[key])


@pytest.mark.parametrize("n", [5, 1000])
def test_schedule_takes_the_earliest_of_mixed_signs(n):
    nb = nb_gpu()
    m, x, v = ni.plummer(n, 61)
    t = np.where(np.arange(n) % 3 == 0, 0.0, -0.25)
    t[1] = -0.5
    t[n - 1] = -0.5
    dt = np.full(n, 2.0 ** -4)
    g = nb.NBody(m, x, v, 1e-3, start_forces=False)
    g.set_state({"t": t, "dt": dt})
    tn, na = g.schedule()
    assert (tn, na) == (-0.5 + 2.0 ** -4, 2)
    np.testing.assert_array_equal(g.active(), [1, n - 1])
    g.close()
