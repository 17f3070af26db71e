"""SC_AvgSIC Hamiltonian apply in mixed precision on fields whose values differ
widely from place to place: points that no tap connects to a value out of range
keep their result."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(dims, h, psi, bc, vloc=None, vavg=None):
    import torch
    from paper_2108_01186_gb300 import flosic as F
    nx, ny, nz = dims
    ctx = F.Context([dict(nx=nx, ny=ny, nz=nz, h=h, origin=[0.0, 0.0, 0.0], norb=[psi.shape[0]])], precision=F.MIXED,
                    solver=F.SOLVER_KRON, boundary={"isolated": F.BC_ISOLATED, "periodic": F.BC_PERIODIC, "slab": F.BC_SLAB}[bc])
    d = [None if v is None else torch.tensor(v, device="cuda") for v in (psi.ravel(), vloc, vavg)]
    return ctx.hamiltonian_apply(*d).cpu().numpy().reshape(psi.shape[0], nz, ny, nx)


@pytest.mark.parametrize("bc", ["periodic", "slab"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -1e300])
@pytest.mark.parametrize("peak_at", [(5, 3, 130), (40, 60, 70)])
def test_a_bad_value_in_a_periodic_orbital_of_many_tiles(bad, peak_at, bc):
    """264 tiles of 32 x 16 x 4 points.  The value out of range sits in the first tile,
    the orbital's largest finite value in the 257th, or in another.  Every point off the
    bad value's three lines agrees with the oracle on the field without it: the oracle's
    37 float64 products and sums and the kernel's fixed point leave
    21.2 / (2 h^2) (2^-57 + 40 2^-53) of the largest value and 2^-45 of the result."""
    import oracle
    dims, h = (64, 64, 132), 0.3
    nx, ny, nz = dims
    rng = np.random.default_rng(5)
    psi = 1e-6 * rng.normal(size=(1, nz, ny, nx))
    psi[0, peak_at[2], peak_at[1], peak_at[0]] = 1.0
    bx, by, bz = 16, 8, 1
    ref = oracle.hamiltonian_apply(psi.reshape(1, -1), (*dims, h, np.zeros(3)), None, None, bc=bc).reshape(psi.shape)
    psi[0, bz, by, bx] = bad
    got = _run(dims, h, psi.reshape(1, -1), bc)
    hit = np.zeros(got.shape, bool)
    hit[0, np.arange(bz - 6, bz + 7) % nz if bc == "periodic" else slice(0, bz + 7), by, bx] = True
    hit[0, bz, by, bx - 6:bx + 7] = hit[0, bz, by - 6:by + 7, bx] = True
    assert np.all(np.isnan(got[hit]))
    tol = 21.2 / (2 * h * h) * (2.0 ** -57 + 40 * 2.0 ** -53) + 2.0 ** -45 * np.abs(ref[~hit])
    assert np.all(np.abs(got[~hit] - ref[~hit]) <= tol)
