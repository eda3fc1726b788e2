"""A handle and its workspace of transposed products made where the device's free memory holds a part of what
they take otherwise: the calls work on parts of the cells and agree with those of a handle that has it all, also
in a batch.

Tolerance: the sums' order changes with the chunks, 1e-12 of the maximum (FP64)."""
import numpy as np
import pytest

from paper_1408_1782_gb300 import inputs

pytestmark = pytest.mark.gpu

N, NX, J, M = 32, 800, 4, 1     # about 2 MB a cell, twenty times the part that does not depend on the cells


def _free():
    import torch

    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _leave(nbytes):
    import torch

    return torch.empty(_free() - nbytes, dtype=torch.uint8, device="cuda")


def _close(a, b):
    assert float((a - b).abs().max()) <= 1e-12 * float(b.abs().max())


def test_calls_in_parts_where_memory_is_short():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()
    from paper_1408_1782_gb300 import qbe

    stream = torch.cuda.current_stream()
    w = torch.from_numpy(np.tile(inputs.synthetic_w(N, 5, seed=8, perturb=0.05), (NX // 5, 1, 1, 1))).cuda()
    lam = w.flip(0).contiguous()
    qbe.Solver(N, 2, J=J, M=M, stream=stream).close()      # the library's own context memory
    before = _free()
    full = qbe.Solver(N, NX, J=J, M=M, stream=stream)
    need = before - _free()
    c = full.collide(w)
    before = _free()
    grad = full.collide_vjp(w, lam)
    need_vjp = before - _free() - grad.nbytes
    full.set_state(w)
    full.step(0.002, 1)
    stepped = torch.empty_like(w)
    full.get_state(stepped)
    full.close()

    out, out_vjp = torch.empty_like(w), torch.empty_like(w)
    filler = _leave(int(0.6 * need))
    short = qbe.Solver(N, NX, J=J, M=M, stream=stream)
    del filler
    filler = _leave(int(0.6 * need_vjp))
    short.collide(w, out)
    short.collide_vjp(w, lam, out_vjp)
    del filler
    torch.cuda.empty_cache()
    _close(out, c)
    _close(out_vjp, grad)
    host = short.collide_vjp(w.cpu().numpy(), lam.cpu().numpy())
    assert np.array_equal(host, out_vjp.cpu().numpy())
    short.set_state(w)
    short.step(0.002, 1)
    short.get_state(out)
    _close(out, stepped)

    other = qbe.Solver(N, 5, J=J, M=M, stream=stream)
    for s, x in ((short, w), (other, w[:5].contiguous())):
        s.set_state(x)
    b = qbe.Batch([short, other], stream=stream)
    b.autotune()
    b.step(0.002, 1)
    short.get_state(out)
    _close(out, stepped)
    b.close()
    short.close()
    other.close()
