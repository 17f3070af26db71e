"""The refinement update that stages its planes by single copies (odd rows,
offsets off 16 bytes, periodic directions): grids smaller than its 32 x 16
tiles, one point past them, a last tile of few planes, rows that start on odd
elements, the shortest periodic side, several orbitals.

Tolerance: as for the other Kronecker solves, ||b - A V|| <= 1e-11 ||b|| leaves
V within 1e-9 max |V| of the discrete solution."""
import numpy as np
import pytest

from test_gpu_mg_coarse import _orbitals

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,bc", [
    ((5, 7, 9), "isolated"), ((31, 15, 33), "isolated"), ((33, 17, 65), "isolated"), ((65, 33, 8), "isolated"),
    ((37, 50, 49), "isolated"), ((21, 14, 13), "periodic"), ((33, 34, 32), "periodic"), ((40, 17, 33), "slab")])
def test_odd_blocks_match_the_oracle(dims, bc):
    import torch
    import oracle
    from paper_2108_01186_gb300 import flosic as F
    h = 0.4
    phi, o = _orbitals(dims, h, 3, seed=sum(dims))
    ref, _ = oracle.poisson(phi ** 2, (*dims, h, o), tol=1e-13, bc=bc)
    ctx = F.Context([dict(nx=dims[0], ny=dims[1], nz=dims[2], h=h, origin=list(o), norb=[3])], precision=F.MIXED,
                    cg_tol=1e-11, solver=F.SOLVER_KRON,
                    boundary={"isolated": F.BC_ISOLATED, "periodic": F.BC_PERIODIC, "slab": F.BC_SLAB}[bc])
    p = torch.tensor(phi.ravel(), device="cuda")
    V, _, conv = ctx.orbital_poisson(p)
    assert torch.all(conv == 1)
    assert np.max(np.abs(V.cpu().numpy().reshape(3, -1) - ref)) < 1e-9 * np.max(np.abs(ref))
    W, _, conv = ctx.orbital_poisson(p, V=1.01 * V)   # warm start: x is read from the first round on
    assert torch.all(conv == 1)
    assert np.max(np.abs(W.cpu().numpy().reshape(3, -1) - ref)) < 1e-9 * np.max(np.abs(ref))
