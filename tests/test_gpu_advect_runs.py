"""The transport kernel walks runs of 8, 4, 2 or 1 cells per thread, by the size of the state: against the
oracle at cell counts that leave a partial last run, for every boundary (ghost cells at both run ends).

Tolerance: a substep adds about six roundings of values at most max |W|; three substeps stay below
1e-14 max |W|."""
import numpy as np
import pytest

from oracle import qbe_oracle as O
from paper_1408_1782_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", ["periodic", "dirichlet", "maxwell"])
@pytest.mark.parametrize("N,Nx", [(64, 41), (32, 79), (32, 39), (16, 5), (8, 2), (8, 1)])
def test_runs_match_oracle(bc, N, Nx):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()
    from paper_1408_1782_gb300 import qbe

    w = inputs.synthetic_w(N, Nx, seed=5, perturb=0.05)
    s = qbe.Solver(N, Nx, J=2, M=1)
    if bc != "periodic":
        fd = qbe.fd_state(1.0, 0.3, -0.2)
        s.set_boundary(bc, fd, fd, alpha=0.5)
    s.set_state(w)
    tau = 2.7 / (12.0 * Nx)                       # three substeps
    s.advect(tau)
    wall = (1.0, 0.3, -0.2, np.eye(2))
    ref = O.advect(w, tau, O.Params(N=N, J=2, M=1), O.Boundary(bc, wall, wall, alpha=0.5))
    assert np.abs(s.get_state() - ref).max() <= 1e-14 * np.abs(w).max()
    s.close()
