"""Multigrid PCG in mixed precision on boxes whose tiles start on odd planes (an even
split of the planes may have any depth): the V-cycle's strength does not depend on
where the tiles lie.

Bounds: the cycle's convergence does not depend on the grid, 26 to 28 iterations to
1e-10 on 64^3 and 128^3 points; 40 leaves room for the shapes here.  V as for the
other multigrid solves: ||b - A V|| <= 1e-11 ||b|| leaves it within 1e-9 max |V|."""
import numpy as np
import pytest

from test_gpu_mg_coarse import _orbitals

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,N", [((32, 32, 9), 10), ((32, 48, 70), 12), ((64, 33, 21), 6)])
def test_thin_boxes_match_the_oracle(dims, N):
    import torch
    import oracle
    from paper_2108_01186_gb300 import flosic as F
    h = 0.4
    phi, o = _orbitals(dims, h, 2, seed=sum(dims))
    ref, _ = oracle.poisson(phi ** 2, (*dims, h, o), tol=1e-13)
    ctx = F.Context([dict(nx=dims[0], ny=dims[1], nz=dims[2], h=h, origin=list(o), norb=[N])], precision=F.MIXED,
                    cg_tol=1e-11, solver=F.SOLVER_PCG, preconditioner=1)
    V, iters, conv = ctx.orbital_poisson(torch.tensor(np.tile(phi.ravel(), N // 2), device="cuda"))
    assert torch.all(conv == 1) and int(iters.max()) <= 40
    err = np.abs(V.cpu().numpy().reshape(N // 2, 2, -1) - ref[None])
    assert np.max(err) < 1e-9 * np.max(np.abs(ref))


def test_a_hundred_cubed_converges():
    """20 orbitals of 100^3: four tiles of 25 planes."""
    import torch
    from paper_2108_01186_gb300 import flosic as F
    n, N, h = 100, 20, 0.3
    x = torch.arange(n, dtype=torch.float64, device="cuda") * h - 0.5 * h * (n - 1)
    r2 = x[:, None, None] ** 2 + x[None, :, None] ** 2 + x[None, None, :] ** 2
    phi = torch.cat([torch.exp(-(0.4 + 0.02 * k) * r2).reshape(-1) for k in range(N)])
    ctx = F.Context([dict(nx=n, ny=n, nz=n, h=h, origin=[float(x[0])] * 3, norb=[N])], precision=F.MIXED, cg_tol=1e-10,
                    solver=F.SOLVER_PCG, preconditioner=1, max_iter=200)
    _, iters, conv = ctx.orbital_poisson(phi, check=False)
    assert torch.all(conv == 1) and int(iters.max()) <= 40
