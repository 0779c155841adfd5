"""Gradients of the pair sums with a softening far below the distances, by ordered pairs (up to 699 particles) and by
unordered ones, against autograd of the plain formula on the CPU.  A term has some 200 roundings and a sum fewer than
800 terms, so (200 + 800) 2^-53 = 1.1e-13 of the terms' magnitudes; the bound is 1e-10 of the largest entry, for
the cancellation among them.  The term of a particle with itself is exactly zero: 1 / eps^3 is 2^60 here."""
import numpy as np
import pytest

import nb_inputs as ni
from nbhelp import nb_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 5, 64, 333, 699, 768])
def test_gradients_with_small_softening(n):
    nb_gpu()
    import torch
    from oracle import adjoint_ref as R
    from paper_1901_08532_gb300 import adjoint as A
    eps = 2.0 ** -20
    m, x, v = ni.plummer(n, 38, imf="salpeter")
    host = [torch.tensor(q, dtype=torch.float64, requires_grad=True) for q in (m, x, v, ni.random_state(n, 39))]
    cot = [torch.tensor(ni.random_state(n, k)) for k in (40, 41, 42)]
    dev = [t.detach().cuda().requires_grad_(True) for t in host]
    ref = torch.autograd.grad(sum((o * g).sum() for o, g in zip(R.pair_sums(*host, eps), cot)), host)
    got = torch.autograd.grad(sum((o * g.cuda()).sum() for o, g in zip(A.PairSums.apply(*dev, eps), cot)), dev)
    for name, g, r in zip(("m", "x", "v", "a"), got, ref):
        g, r = g.cpu().numpy(), r.numpy()
        assert np.abs(g - r).max() <= 1e-10 * np.abs(r).max(), name
