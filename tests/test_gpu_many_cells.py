"""A call of more cells than fit 32-bit element counts: 1.7 million cells of N = 8 (5 x 256 values each in the
sums of the angle chunks), against the same five states in a call of their own.

Tolerance: the FP32-split form's stated 5e-6 of max |C|."""
import pytest

from paper_1408_1782_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_more_cells_than_32_bit_counts():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 160 << 30:
        pytest.skip("needs 130 GB of device memory")
    import __graft_entry__ as g

    g.build()
    from paper_1408_1782_gb300 import qbe

    N, ncells = 8, 1_700_000
    w = torch.from_numpy(inputs.synthetic_w(N, 5, seed=4, perturb=0.05)).cuda()
    few = qbe.Solver(N, 5, J=2, M=1, stream=torch.cuda.current_stream(), precision=1)
    ref = few.collide(w)
    few.close()
    many = qbe.Solver(N, ncells, J=2, M=1, stream=torch.cuda.current_stream(), precision=1)
    w = w.repeat(ncells // 5, 1, 1, 1)
    got = many.collide(w).view(-1, 5, 4, N, N)
    many.close()
    err = max(float((g - ref).abs().max()) for g in got.split(100_000))
    del w, got
    torch.cuda.empty_cache()
    assert err < 5e-6 * float(ref.abs().max())
