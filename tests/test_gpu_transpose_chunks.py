"""The transposed product of the FP32-split form where a work unit holds several groups of radial nodes (the other
tests' few cells leave one group a unit): sums carried from group to group, and teams of a block whose units hold
unequal numbers of them.  Against the FP64 product, every variant.

Tolerance: the FP32-split form's stated 5e-6 of the maximum."""
import numpy as np
import pytest

from paper_1408_1782_gb300 import inputs

pytestmark = pytest.mark.gpu


# chunks of M nodes on 152 SMs, and the groups (pairs, and the middle node of an odd M) in them
@pytest.mark.parametrize("N,ncells,J,M", [
    (16, 152, 64, 6),    # 1: three pairs
    (16, 152, 64, 5),    # 1: two pairs and the middle node
    (16, 304, 16, 7),    # 2: two pairs; a pair and the middle node
    (32, 16, 32, 32),    # 7: two or three pairs
    (32, 76, 16, 7),     # 2, as above
    (48, 19, 16, 7),     # 2
    (64, 19, 16, 7),     # 2, both variants
])
def test_several_groups_of_nodes_in_a_unit(N, ncells, J, M):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()
    from paper_1408_1782_gb300 import qbe

    few = 4
    tile = (ncells + few - 1) // few
    w = torch.from_numpy(inputs.synthetic_w(N, few, seed=50 + N, perturb=0.05)).cuda()
    lam = torch.from_numpy(inputs.random_field(w.shape, seed=51)).cuda()
    s = qbe.Solver(N, few, J=J, M=M, stream=torch.cuda.current_stream())
    ref = s.collide_vjp(w, lam)
    s.close()
    w, lam = (x.repeat(tile, 1, 1, 1)[:ncells].contiguous() for x in (w, lam))
    s = qbe.Solver(N, ncells, J=J, M=M, stream=torch.cuda.current_stream(), precision=1)
    for v in range(s.vjp_i3_variant()[1]):
        s.set_vjp_i3_variant(v)
        got = s.collide_vjp(w, lam)
        for i in range(0, ncells, few):
            part = got[i:i + few]
            assert float((part - ref[:len(part)]).abs().max()) < 5e-6 * float(ref.abs().max()), (v, i)
    s.close()
