"""A system's results alone and in a batch: the tiles' depth and the number of
partial sums follow the whole batch, so the last bits may differ, no more.

Tolerance: either solve leaves V within 1e-9 max |V| of the discrete solution
(||b - A V|| <= 1e-11 ||b||), as in the other solver tests."""
import numpy as np
import pytest

from test_gpu_mg_coarse import _orbitals

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,solver", [("FP64", "PCG"), ("MIXED", "PCG"), ("MIXED", "KRON")])
def test_alone_and_among_others(prec, solver):
    import torch
    from paper_2108_01186_gb300 import flosic as F
    h, batch = 0.4, [((24, 24, 40), 2), ((64, 48, 40), 12), ((33, 20, 17), 3)]
    sys, phis = [], []
    for k, (d, N) in enumerate(batch):
        phi, o = _orbitals(d, h, N, seed=k)
        sys.append(dict(nx=d[0], ny=d[1], nz=d[2], h=h, origin=list(o), norb=[N]))
        phis.append(torch.tensor(phi.ravel(), device="cuda"))
    opt = dict(precision=getattr(F, prec), solver=getattr(F, "SOLVER_" + solver), cg_tol=1e-11)
    V, _, _ = F.Context(sys, **opt).orbital_poisson(torch.cat(phis))
    for s, p, v in zip(sys, phis, torch.split(V, [p.numel() for p in phis])):
        W, _, _ = F.Context([s], **opt).orbital_poisson(p)
        assert torch.max(torch.abs(W - v)) < 2e-9 * torch.max(torch.abs(W))
