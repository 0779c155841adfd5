"""The stages of a block step where their arithmetic leaves the FP64 pipe, or is spread over threads.

Conversions of the prediction are exact operations: a prediction to the particles' own time returns the state
rounded as the layout says, to the bit.  The step decision comes from FP32 logarithms unless they are in doubt:
the step must equal that of the FP64 criterion (the oracle's) over a wide range of magnitudes, at exact powers
of two of the criterion and for zero and non-finite derivatives.  Runs of block steps on the device are
compared with host-driven ones at the slice sizes where the launch changes."""
import numpy as np
import pytest

import nb_inputs as ni
import oracle as O
from nbhelp import nb_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [1, 3])
def test_prediction_to_own_time_rounds_exactly(prec):
    nb = nb_gpu()
    n = 4099
    vals = np.concatenate([ni.random_state(n, 5) * 2.0 ** (np.arange(n)[:, None] % 80 - 40.0),
                           [[0.0, -0.0, 1.0], [1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24, 1.0 - 2.0 ** -25],
                            [2.0 ** -126, 1.5 * 2.0 ** -127, 2.0 ** -150], [3e38, -3e38, 1e30],
                            [2.0 - 2.0 ** -24, 2.0 - 2.0 ** -25, 2.0 - 2.0 ** -52]]])
    k = len(vals)
    x, v, a = vals, np.roll(vals, 1, axis=1), np.roll(vals, 2, axis=1)
    g = nb.NBody(np.ones(k), x, v, 1e-3, precision=prec, start_forces=False)
    g.set_state({"a": a})
    g.predict(0.0)
    got = g.predicted()
    g.close()
    hi = lambda q: q.astype(np.float32).astype(np.float64)  # noqa: E731
    dw = lambda q: hi(q) + hi(q - hi(q))  # noqa: E731
    want = (dw(x), dw(v), dw(a)) if prec == 3 else (dw(x), hi(v), hi(a))
    for w, q in zip(want, got):
        np.testing.assert_array_equal(q, w)


def _steps(nb, a1, j1, s1, c0, h, t1):
    """New steps of particles whose old derivatives are a0 = j0 = s0 = c0-scaled, from one corrector call."""
    n = len(a1)
    z = np.zeros((n, 3))
    g = nb.NBody(np.ones(n), z, z, 1e-3, start_forces=False, dt_max=2.0 ** -3)
    g.set_state({"a": c0[0], "j": c0[1], "s": c0[2], "t": np.full(n, t1 - h), "dt": np.full(n, h)})
    act = np.arange(n, dtype=np.int32)
    g.predict(t1)
    g.set_forces(act, np.concatenate([a1.T, j1.T, s1.T]))
    g.correct(t1)
    dt = g.state()["dt"]
    g.close()
    return dt


def _oracle_steps(a1, j1, s1, c0, h, t1):
    out = np.empty(len(a1))
    for i in range(len(a1)):
        c, d, e = O.interpolate(h, c0[0][i], c0[1][i], c0[2][i], a1[i], j1[i], s1[i])
        out[i], _ = O.dt_quantise(O.dt_crit(0.4, a1[i], j1[i], s1[i], c, d, e), h, t1)
    return out


def test_step_decision_equals_the_fp64_criterion():
    nb = nb_gpu()
    n, h, t1 = 2500, 2.0 ** -9, 0.25
    rng = [ni.random_state(n, 20 + k) for k in range(6)]
    scale = 2.0 ** (np.arange(n)[:, None] % 121 - 60.0)
    omega = 2.0 ** (np.arange(n)[:, None] % 13 - 4.0)  # ratio of successive derivatives
    a0, j0, s0 = (r * scale * omega ** k for k, r in enumerate(rng[:3]))
    a1, j1, s1 = (r * scale * omega ** k for k, r in enumerate(rng[3:]))
    smooth = slice(0, n, 2)  # half of them: a smooth motion, whose criterion varies over several powers of two
    a1[smooth] = (a0 + j0 * h + s0 * h * h / 2)[smooth] * (1 + 1e-9 * rng[3][smooth])
    j1[smooth] = (j0 + s0 * h)[smooth] * (1 + 1e-7 * rng[4][smooth])
    s1[smooth] = s0[smooth] * (1 + 1e-4 * rng[5][smooth])
    got = _steps(nb, a1, j1, s1, (a0, j0, s0), h, t1)
    np.testing.assert_array_equal(got, _oracle_steps(a1, j1, s1, (a0, j0, s0), h, t1))
    assert len(np.unique(got)) >= 4


def test_step_decision_at_exact_powers_and_zero_derivatives():
    """Motions with one non-zero derivative at the end of the step (the criterion's ratio in closed form up to a
    scale) and scaled copies whose criterion crosses a power of two within a few 1e-6."""
    nb = nb_gpu()
    h, t1 = 2.0 ** -6, 0.5
    z = np.zeros(3)
    base = [([1.0, 0, 0], z, z), (z, [0, 1.0, 0], z), (z, z, [0, 0, 1.0]), (z, z, z), ([1.0, 0, 0], [0, 1.0, 0], z)]
    rows = [tuple(np.asarray(q, float) * f for q, f in zip(b, (1.0, s, s * s))) for b in base
            for s in np.concatenate([[1.0, 2.0 ** 10, 2.0 ** -10], 1.0 + 1e-6 * np.arange(-4, 5)])]
    a1, j1, s1 = (np.array([r[k] for r in rows]) for k in range(3))
    zero = np.zeros_like(a1)
    got = _steps(nb, a1, j1, s1, (zero, zero, zero), h, t1)
    np.testing.assert_array_equal(got, _oracle_steps(a1, j1, s1, (zero, zero, zero), h, t1))


@pytest.mark.parametrize("prec,n", [(0, 5), (0, 9), (0, 1216), (0, 1217), (3, 17), (3, 2433), (3, 14591), (3, 14593),
                                    (1, 14593)])
def test_device_steps_match_host_steps_at_launch_edges(prec, n):
    """FP64 and EX take the same decisions either way; states agree to the rounding of another summation order over
    a few block steps (1e-12 of the largest entry; mixed: 1e-6, positions 1e-9)."""
    nb = nb_gpu()
    m, x, v = ni.plummer(n, 33)
    out = []
    for device in (True, False):
        g = nb.NBody(m, x, v, 1e-2, precision=prec, device_steps=device, dt_max=2.0 ** -7,
                     step_noise=4e-7 if prec == 1 else 0.0)
        steps, log = g.run_until(2.0 ** -7, log_cap=4096)
        out.append((steps, log, g.state()))
        g.close()
    (sa, (ta, na), a), (sb, (tb, nb_), b) = out
    if prec != 1:
        assert sa == sb
        np.testing.assert_array_equal(ta, tb)
        np.testing.assert_array_equal(na, nb_)
    for k, tol in (("x", 1e-12), ("v", 1e-12), ("a", 1e-11), ("j", 1e-10)):
        tol = tol if prec != 1 else (1e-9 if k in "xv" else 1e-5)
        assert np.abs(a[k] - b[k]).max() <= tol * np.abs(b[k]).max(), k


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("shape", [(4, 64, 16), (8, 96, 64), (4, 160, 128), (16, 256, 256), (3, 128, 8)])
def test_ensemble_shapes_take_the_same_steps(prec, shape):
    """Block and lane counts that are no power of two, j-tiles smaller than the scratch that shares their memory:
    the decisions of the default shape, and its state to the rounding of another summation order."""
    nb = nb_gpu()
    sizes = np.array([5, 130, 301, 64])
    m, x, v = (np.concatenate([ni.plummer(int(k), 40 + q)[f] for q, k in enumerate(sizes)]) for f in range(3))
    out = []
    for sh in (None, shape):
        e = nb.Ensemble(sizes, m, x, v, 1e-2, precision=prec, dt_max=2.0 ** -6)
        if sh:
            e.set_shape(*sh)
        e.run(2.0 ** -6)
        out.append((e.stats()[0], e.state()))
        e.close()
    (sa, a), (sb, b) = out
    np.testing.assert_array_equal(sa, sb)
    np.testing.assert_array_equal(a["t"], b["t"])
    np.testing.assert_array_equal(a["dt"], b["dt"])
    for k, tol in (("x", 1e-12), ("v", 1e-12), ("a", 1e-11), ("j", 1e-10)):
        assert np.abs(a[k] - b[k]).max() <= tol * np.abs(b[k]).max(), k
