"""The mixed-precision Hamiltonian apply (exact integer sums of psi in two
digits scaled by the tiles' largest exponents): sides around the 32 x 16 tiles
and the z-depths, odd rows, periodic wraps, values that span many decades from
tile to tile, and values that are not finite.

Tolerance per point: psi is held to 2^-57 of the largest value m the tile's
taps reach, the oracle rounds its 37 products and sums in float64 (at most 40
2^-53 of the terms' magnitudes), and the result leaves a float-float pair
(2^-45).  The weights' magnitudes sum to 21.2 / (2 h^2), so
|error| <= 21.2 / (2 h^2) (2^-57 + 40 2^-53) m + 2^-45 (|H psi| + |v psi|)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TILE = (32, 16, 32)


def _near_max(psi, dims, per):
    """Per point the largest |psi| of its tile and the neighbouring tiles (all
    tiles in a periodic cell)."""
    nx, ny, nz = dims
    a = np.abs(psi.reshape(-1, nz, ny, nx))
    out = np.empty_like(a)
    for f, o in zip(a, out):
        for z in range(0, nz, TILE[2]):
            for y in range(0, ny, TILE[1]):
                for x in range(0, nx, TILE[0]):
                    box = f if per else f[max(z - TILE[2], 0):z + 2 * TILE[2], max(y - TILE[1], 0):y + 2 * TILE[1],
                                          max(x - TILE[0], 0):x + 2 * TILE[0]]
                    o[z:z + TILE[2], y:y + TILE[1], x:x + TILE[0]] = box.max()
    return out.reshape(psi.shape)


def _run(F, dims, h, psi, vloc, vavg, bc):
    import torch
    nx, ny, nz = dims
    ctx = F.Context([dict(nx=nx, ny=ny, nz=nz, h=h, origin=[0.0, 0.0, 0.0], norb=[psi.shape[0]])], precision=F.MIXED,
                    solver=F.SOLVER_KRON, boundary={"isolated": F.BC_ISOLATED, "periodic": F.BC_PERIODIC, "slab": F.BC_SLAB}[bc])
    d = [None if v is None else torch.tensor(v, device="cuda") for v in (psi.ravel(), vloc, vavg)]
    return ctx.hamiltonian_apply(*d).cpu().numpy().reshape(psi.shape)


@pytest.mark.parametrize("dims,bc,N", [
    ((12, 13, 14), "isolated", 2), ((32, 16, 32), "isolated", 1), ((33, 17, 31), "isolated", 2), ((31, 15, 5), "isolated", 3),
    ((65, 49, 37), "isolated", 1), ((38, 22, 96), "isolated", 12), ((128, 16, 64), "isolated", 7),
    ((33, 34, 35), "periodic", 2), ((32, 16, 32), "periodic", 1), ((45, 18, 41), "slab", 2)])
def test_digits_match_the_oracle(dims, bc, N):
    import oracle
    from paper_2108_01186_gb300 import flosic as F
    rng = np.random.default_rng(sum(dims))
    G, h = dims[0] * dims[1] * dims[2], 0.3
    grid = (*dims, h, np.zeros(3))
    vloc, vavg = rng.normal(size=G) - 1.0, 0.1 * rng.normal(size=G)
    # noise, and values falling by 60 decades along one direction
    decay = np.exp(-np.linspace(0.0, 138.0, dims[0]))[None, None, :] * np.ones((dims[2], dims[1], 1))
    for psi in (rng.normal(size=(N, G)), rng.normal(size=(N, G)) * decay.ravel(), 1e-25 * rng.normal(size=(N, G))):
        near = _near_max(psi, dims, bc != "isolated")
        for v, w in ((None, None), (vloc, None), (vloc, vavg)):
            got = _run(F, dims, h, psi, v, w, bc)
            ref = oracle.hamiltonian_apply(psi, grid, v, w, bc=bc)
            vp = np.abs(((0 if v is None else v) + (0 if w is None else w)) * psi)
            tol = 21.2 / (2 * h * h) * (2.0 ** -57 + 40 * 2.0 ** -53) * near + 2.0 ** -45 * (np.abs(ref) + vp)
            assert np.all(np.abs(got - ref) <= tol), float(np.max(np.abs(got - ref) / tol))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("at", [(0, 0, 0), (31, 15, 3), (32, 16, 20), (40, 33, 39)])
def test_values_that_are_not_finite(bad, at):
    import oracle
    from paper_2108_01186_gb300 import flosic as F
    dims, h = (41, 34, 40), 0.3
    rng = np.random.default_rng(3)
    G = dims[0] * dims[1] * dims[2]
    psi = rng.normal(size=(2, G))
    clean = oracle.hamiltonian_apply(psi, (*dims, h, np.zeros(3)))
    x, y, z = at
    psi.reshape(2, dims[2], dims[1], dims[0])[1, z, y, x] = bad
    got = _run(F, dims, h, psi, None, None, "isolated").reshape(2, dims[2], dims[1], dims[0])
    hit = np.zeros(got.shape, bool)
    hit[1, max(z - 6, 0):z + 7, y, x] = hit[1, z, max(y - 6, 0):y + 7, x] = hit[1, z, y, max(x - 6, 0):x + 7] = True
    assert np.all(np.isnan(got[hit]))
    near = np.max(np.abs(psi[np.isfinite(psi)]))
    tol = 21.2 / (2 * h * h) * (2.0 ** -57 + 40 * 2.0 ** -53) * near + 2.0 ** -45 * np.abs(clean.reshape(got.shape)[~hit])
    assert np.all(np.abs(got[~hit] - clean.reshape(got.shape)[~hit]) <= tol)
