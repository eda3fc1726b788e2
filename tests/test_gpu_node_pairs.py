"""The radial nodes of the Hu-Ying term taken in pairs +-rho_m (eq. approxH-JM): C[W] against the oracle
over node counts and m-chunkings at which the pairing changes form -- a lone middle node (M = 1), odd M,
one pair, chunks that hold several pairs, one pair and half a pair -- for every launch variant; and a
batch whose members ask for different variants.

Tolerances: the FP64 form's parity bound 1e-11 of max |C| and the FP32-split form's stated 5e-6."""
import numpy as np
import pytest

from oracle import qbe_oracle as O
from paper_1408_1782_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = {0: 1e-11, 1: 5e-6}


@pytest.fixture(scope="module")
def qbe():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()
    from paper_1408_1782_gb300 import qbe as q

    return q


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N,J,M,ncells", [(8, 4, 1, 2), (8, 4, 2, 3), (16, 4, 5, 2), (16, 2, 8, 1), (32, 2, 3, 2),
                                          (48, 2, 4, 1), (64, 2, 5, 2), (96, 2, 3, 1), (128, 2, 2, 1)])
def test_every_chunking_of_every_variant(qbe, N, J, M, ncells, prec):
    import torch

    w = inputs.synthetic_w(N, ncells, seed=90 + N + M, perturb=0.05)
    ref = O.collision(w, O.Params(N=N, J=J, M=M))
    s = qbe.Solver(N, ncells, J=J, M=M, stream=torch.cuda.current_stream(), precision=prec)
    wd = torch.from_numpy(np.ascontiguousarray(w)).cuda()
    top = s.i3_shape()["m_chunks"]
    assert top == M                       # few units: one item per chunk to begin with
    for v in range(s.i3_shape()["nvariants"]):
        for chunks in range(1, top + 1):
            s.set_i3_shape(variant=v, m_chunks=chunks)
            got = s.collide(wd).cpu().numpy()
            assert np.abs(got - ref).max() < TOL[prec] * np.abs(ref).max(), (v, chunks)
    s.close()


@pytest.mark.parametrize("first,second", [(0, 2), (2, 0)])
def test_batch_of_members_with_different_variants(qbe, first, second):
    """The group's launch takes the first member's variant for all: each member's post-processing must
    read what that launch wrote."""
    dt, shapes = 0.002, [(16, 3), (16, 2)]

    def make():
        out = []
        for k, (N, Nx) in enumerate(shapes):
            s = qbe.Solver(N, Nx, J=4, M=3)
            s.set_state(inputs.synthetic_w(N, Nx, seed=70 + k, perturb=0.05))
            out.append(s)
        return out

    solo, together = make(), make()
    for s, v in zip(together, (first, second)):
        s.set_i3_shape(variant=v)
    b = qbe.Batch(together)
    b.step(dt, 2)
    for s, s1 in zip(together, solo):
        s1.step(dt, 2)
        ref = s1.get_state()
        assert np.abs(s.get_state() - ref).max() <= 1e-12 * np.abs(ref).max()
    # and alone again, each with its own variant
    for s, s1 in zip(together, solo):
        s.step(dt, 1)
        s1.step(dt, 1)
        ref = s1.get_state()
        assert np.abs(s.get_state() - ref).max() <= 1e-12 * np.abs(ref).max()
    b.close()


@pytest.mark.parametrize("N,J,M,ncells", [(16, 32, 8, 24), (32, 32, 8, 8), (64, 16, 3, 12)])
def test_fp32_with_every_team_busy(qbe, N, J, M, ncells):
    """More units than the launch works on at a time (16, 4 and 1 per block for N = 16, 32, 64), so that
    every team of every block has several: against the FP64 form."""
    import torch

    w = torch.from_numpy(inputs.synthetic_w(N, ncells, seed=120 + N, perturb=0.05)).cuda()
    out = []
    for prec in (0, 1):
        s = qbe.Solver(N, ncells, J=J, M=M, stream=torch.cuda.current_stream(), precision=prec)
        out.append(s.collide(w).cpu().numpy())
        s.close()
    assert np.abs(out[1] - out[0]).max() < TOL[1] * np.abs(out[0]).max()


@pytest.mark.parametrize("N,J,M,ncells", [(48, 32, 8, 8), (48, 2, 9, 40), (96, 4, 3, 4)])
def test_fp32_grids_with_a_factor_of_three_every_team_busy(qbe, N, J, M, ncells):
    """The same for the two teams per block of N = 48 and the clusters of N = 96 (odd M: a middle node)."""
    test_fp32_with_every_team_busy(qbe, N, J, M, ncells)


def _derivative(s, w, dw):
    """C'(w) dw: C is cubic in w, so the five-point difference is exact for every step."""
    f = [s.collide(np.ascontiguousarray(w + h * dw)) for h in (1.0, -1.0, 2.0, -2.0)]
    return (8.0 * (f[0] - f[1]) - (f[2] - f[3])) / 12.0


@pytest.mark.parametrize("N,J,M,ncells", [(8, 4, 1, 2), (8, 4, 2, 3), (16, 4, 5, 2), (16, 16, 6, 24), (32, 2, 3, 2),
                                          (48, 2, 2, 1), (64, 2, 3, 2), (96, 2, 1, 1), (128, 2, 2, 1)])
def test_transpose_with_node_pairs(qbe, N, J, M, ncells):
    """(dC/dW)^T over a lone middle node, odd M, half pairs (few units) and whole pairs: the FP64 product
    against the forward's own derivative (1e-11 of the sum of absolute products, the adjoint tests'
    bound), the FP32-split product against the FP64 one."""
    w = inputs.synthetic_w(N, ncells, seed=30 + N, perturb=0.05)
    dw = 0.1 * w * inputs.random_field(w.shape, seed=31)
    lam = inputs.random_field(w.shape, seed=32)
    s = qbe.Solver(N, ncells, J=J, M=M)
    g = s.collide_vjp(w, lam)
    jv = _derivative(s, w, dw)
    gap = abs(np.sum(lam * jv) - np.sum(g * dw)) / max(np.sum(np.abs(lam * jv)), np.sum(np.abs(g * dw)))
    assert gap < 1e-11
    s.close()
    s = qbe.Solver(N, ncells, J=J, M=M, precision=1)
    for v in range(s.vjp_i3_variant()[1]):
        s.set_vjp_i3_variant(v)
        assert np.abs(s.collide_vjp(w, lam) - g).max() < TOL[1] * np.abs(g).max(), v
    s.close()
