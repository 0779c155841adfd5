"""Device memory that a context holds after evaluating all of its particles: the state and buffers (under 400 bytes a
particle), the partial sums of the pairs (two slots of 72 bytes a particle at least, else within 256 MB up to some
150000 particles), and the allocator's granularity (2 MB for each of some 20 allocations)."""
import pytest

import nb_inputs as ni
from nbhelp import nb_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [(1, 65536), (3, 65536), (0, 32768)])
def test_context_memory(prec, n):
    nb = nb_gpu()
    import torch
    for k in (5000, n):  # the first loads the kernels
        m, x, v = ni.plummer(k, 30)
        torch.cuda.synchronize()
        free0, _ = torch.cuda.mem_get_info()
        g = nb.NBody(m, x, v, 1e-3, precision=prec, start_forces=False)
        g.predict(0.0)
        g.evaluate(None, out=False)
        torch.cuda.synchronize()
        free1, _ = torch.cuda.mem_get_info()
        g.close()
    assert free0 - free1 <= 400 * n + 256e6 + 40e6
