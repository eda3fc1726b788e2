"""One handle gives a cell the same bits whether a call carries that cell alone or every cell: C[W], the
product with its transposed derivative, and the allocation-free entry (whose static array takes its cells in
batches).  The cell counts lie above the line at which the partials' sums are taken by one thread each, so
that a rule by the cells of the call would sum the single cell in another order."""
import numpy as np
import pytest

from paper_1408_1782_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qbe():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()
    from paper_1408_1782_gb300 import qbe as q

    return q


def _state(N, ncells):
    import torch

    w = inputs.synthetic_w(N, 5, seed=N, perturb=0.05)
    return torch.from_numpy(np.tile(w, ((ncells + 4) // 5, 1, 1, 1))[:ncells].copy()).cuda()


# 152 x 1024 threads over the 16-byte words of a cell's sums: 62 cells (FP64) and 124 (FP32) at N = 16,
# 3.8 and 7.6 at N = 64, 6.8 (FP64) at N = 48
@pytest.mark.parametrize("prec,N,ncells", [(0, 16, 70), (1, 16, 140), (0, 64, 5), (1, 64, 9), (0, 48, 8)])
def test_one_cell_of_many(qbe, prec, N, ncells):
    import torch

    s = qbe.Solver(N, ncells, J=16, M=2, stream=torch.cuda.current_stream(), precision=prec)
    w = _state(N, ncells)
    lam = torch.from_numpy(inputs.random_field((1, 4, N, N), seed=3)).cuda().repeat(ncells, 1, 1, 1)
    c, g = s.collide(w), s.collide_vjp(w, lam)
    for i in (0, ncells - 1):
        assert torch.equal(s.collide(w[i:i + 1].contiguous())[0], c[i])
        assert torch.equal(s.collide_vjp(w[i:i + 1].contiguous(), lam[:1])[0], g[i])
    s.close()


# 304 and 76 cells without the Fourier-space partials
@pytest.mark.parametrize("N,ncells", [(8, 320), (16, 80)])
def test_one_cell_of_many_without_allocation(qbe, N, ncells):
    import torch

    w = _state(N, ncells)
    out, one = torch.empty_like(w), torch.empty_like(w[:1])
    qbe.collide_noalloc(w, out, J=16, M=2, stream=torch.cuda.current_stream())
    for i in (0, ncells - 1):
        qbe.collide_noalloc(w[i:i + 1].contiguous(), one, J=16, M=2, stream=torch.cuda.current_stream())
        assert torch.equal(one[0], out[i])
