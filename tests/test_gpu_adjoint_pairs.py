"""The pair adjoint by unordered pairs (with workspace) against the one by ordered pairs (without) at tile edges:
tiles of 32, 64 and 128 particles, odd and even tile counts, a last tile of one particle, and a size that stays
on the ordered kernel.  Tolerance: both are FP64 sums of the same terms; 1e-12 of the largest entry, the FP64
parity bound (a chain of n terms rounds by at most n 2^-53 < 1e-12 of the sum of their magnitudes)."""
import ctypes as C

import pytest

import nb_inputs as ni
from nbhelp import nb_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 700, 769, 1024, 1089, 2048, 4097])
def test_adjoint_by_unordered_pairs_matches_ordered(n):
    nb = nb_gpu()
    import torch
    lib = nb.lib()
    cuda = lambda q: torch.from_numpy(q).cuda()  # noqa: E731
    m, x, v = (cuda(q) for q in ni.plummer(n, 60, imf="salpeter"))
    rows = [x, v] + [cuda(ni.random_state(n, 61 + k)) for k in range(4)]  # x, v, a, cotangents
    stream = torch.cuda.current_stream().cuda_stream
    p = lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
    args = [p(t) for t in (m, *rows[:3])]
    cot = [p(t) for t in rows[3:]]
    outs = [[torch.full((n, 3), float("nan"), dtype=torch.float64, device="cuda") for _ in range(3)]
            + [torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")] for _ in range(3)]
    assert lib.nb_pairs_fp64_adjoint(n, *args, 1e-2, *cot, *[p(t) for t in outs[0]], C.c_void_p(stream)) == 0
    nbytes = lib.nb_pairs_adjoint_workspace_bytes(n)
    assert (nbytes > 0) == (n >= 700)
    for o in outs[1:]:
        work = torch.full((max(1, nbytes),), 255, dtype=torch.uint8, device="cuda")
        assert lib.nb_pairs_fp64_adjoint_work(n, *args, 1e-2, *cot, *[p(t) for t in o],
                                              p(work) if nbytes else None, C.c_void_p(stream)) == 0
    for ref, got, again in zip(*outs):
        assert torch.equal(got, again)
        assert float((got - ref).abs().max()) <= 1e-12 * float(ref.abs().max())
