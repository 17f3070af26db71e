"""The tensor-core Kronecker transforms on sides that are padded (not multiples
of 8, or above 128): every remainder modulo 4, the edges of the 32-point boxes
and 16-point K steps, both size classes, against the oracle's Poisson solve.

Tolerance: the solves stop at ||b - A V|| <= 1e-11 ||b||; on these grids
max |V| exceeds 1e-3 ||b|| / lambda_min(A), so V is within 1e-9 max |V| of the
exact discrete solution (the bar of the unpadded transforms' tests)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _orbitals(nx, ny, nz, h, N, seed):
    rng = np.random.default_rng(seed)
    o = -0.5 * h * (np.array([nx, ny, nz]) - 1)
    x, y, z = (o[d] + h * np.arange(n) for d, n in enumerate((nx, ny, nz)))
    out = []
    for _ in range(N):
        c = rng.uniform(-0.15, 0.15, 3) * h * np.array([nx, ny, nz])
        s = rng.uniform(0.6, 1.2)
        f = (np.exp(-(z - c[2]) ** 2 / (2 * s * s))[:, None, None] * np.exp(-(y - c[1]) ** 2 / (2 * s * s))[None, :, None]
             * np.exp(-(x - c[0]) ** 2 / (2 * s * s))[None, None, :]).ravel()
        out.append(f / np.sqrt(np.sum(f * f) * h ** 3))
    return np.array(out), o


@pytest.mark.parametrize("dims,bc", [
    ((33, 34, 35), "isolated"), ((32, 47, 50), "isolated"), ((63, 65, 66), "isolated"), ((62, 97, 95), "isolated"),
    ((127, 36, 126), "isolated"), ((129, 33, 130), "isolated"), ((192, 35, 34), "isolated"), ((34, 191, 161), "isolated"),
    ((33, 34, 35), "periodic"), ((45, 38, 41), "slab")])
def test_padded_transforms_match_the_oracle(dims, bc):
    import torch
    import oracle
    from paper_2108_01186_gb300 import flosic as F
    nx, ny, nz = dims
    h = 0.3
    phi, o = _orbitals(nx, ny, nz, h, 2, seed=sum(dims))
    grid = (nx, ny, nz, h, o)
    Vref, _ = oracle.poisson(phi ** 2, grid, tol=1e-13, bc=bc)
    per = {"isolated": F.BC_ISOLATED, "periodic": F.BC_PERIODIC, "slab": F.BC_SLAB}[bc]
    ctx = F.Context([dict(nx=nx, ny=ny, nz=nz, h=h, origin=list(o), norb=[2])], precision=F.MIXED, cg_tol=1e-11,
                    solver=F.SOLVER_KRON, boundary=per)
    assert ctx.block_paths()[0]["tensor_core_transforms"]
    p = torch.tensor(phi.ravel(), device="cuda")
    for _ in range(2):   # the padding of the second solve's arrays holds the first one's values
        V, iters, conv = ctx.orbital_poisson(p)
        assert torch.all(conv == 1)
        assert np.max(np.abs(V.cpu().numpy().reshape(2, -1) - Vref)) < 1e-9 * np.max(np.abs(Vref))
    V2, _, _ = ctx.orbital_poisson(p, V=V.clone())   # warm start
    assert np.max(np.abs(V2.cpu().numpy().reshape(2, -1) - Vref)) < 1e-9 * np.max(np.abs(Vref))


def test_batch_of_both_size_classes_and_the_cuda_cores():
    import torch
    import oracle
    from paper_2108_01186_gb300 import flosic as F
    specs = [(129, 40, 33, 2), (21, 22, 23, 3), (64, 64, 40, 2), (35, 35, 35, 1)]
    sysd, phis, refs = [], [], []
    for nx, ny, nz, N in specs:
        phi, o = _orbitals(nx, ny, nz, 0.3, N, seed=nx)
        sysd.append(dict(nx=nx, ny=ny, nz=nz, h=0.3, origin=list(o), norb=[N]))
        phis.append(phi)
        refs.append(oracle.poisson(phi ** 2, (nx, ny, nz, 0.3, o), tol=1e-13)[0])
    ctx = F.Context(sysd, precision=F.MIXED, cg_tol=1e-11, solver=F.SOLVER_KRON, autotune=0)
    assert [b["tensor_core_transforms"] for b in ctx.block_paths()] == [True, False, True, True]
    V, _, conv = ctx.orbital_poisson(torch.tensor(np.concatenate([p.ravel() for p in phis]), device="cuda"))
    assert torch.all(conv == 1)
    V, off = V.cpu().numpy(), 0
    for ref in refs:
        got = V[off:off + ref.size].reshape(ref.shape)
        assert np.max(np.abs(got - ref)) < 1e-9 * np.max(np.abs(ref))
        off += ref.size
