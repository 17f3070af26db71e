"""The mixed-precision Hamiltonian apply where psi is far below its tile's largest
value: an orbital's tail is held as exactly, in its own magnitude, as its bulk.

Tolerance per point, from the taps that it reads, with A = sum |w| |psi| / (2 h^2)
over its 37 taps: every value is held to 2^-48 of itself; the low parts of one
distance (six values' and five sums' errors, each at most 2^-24 of the values) are
added in float32, at most 60 roundings of 2^-24 of them; the oracle's own float64
products and sums round 40 times.  |error| <= (64 2^-48 + 40 2^-53) A + 4 2^-53 (|H psi| + |v psi|)."""
import numpy as np
import pytest

from test_gpu_hamiltonian_values import _run

pytestmark = pytest.mark.gpu
W = [0.0] + [2.0 * (-1) ** (m + 1) * 518400.0 / (m * m * f) for m, f in
             ((1, 604800.0), (2, 967680.0), (3, 2177280.0), (4, 7257600.0), (5, 39916800.0), (6, 479001600.0))]
W[0] = -2.0 * sum(W[1:])


def _terms(psi, h, per):
    """sum |w| |psi| / (2 h^2) over the taps of every point, psi [N, nz, ny, nx]."""
    a = np.abs(psi)
    out = 3.0 * abs(W[0]) * a
    for d in range(3):                        # x, y, z
        ax = 3 - d
        for m in range(1, 7):
            for s in (m, -m):
                t = np.roll(a, s, axis=ax)
                if d not in per:
                    cut = [slice(None)] * 4
                    cut[ax] = slice(0, s) if s > 0 else slice(s, None)
                    t[tuple(cut)] = 0.0
                out = out + abs(W[m]) * t
    return out / (2.0 * h * h)


@pytest.mark.parametrize("bc", ["isolated", "periodic", "slab"])
@pytest.mark.parametrize("dims", [(40, 40, 40), (37, 18, 45), (96, 17, 14)])
def test_tails_keep_their_bits(dims, bc):
    import oracle
    nx, ny, nz = dims
    h = 0.25
    rng = np.random.default_rng(sum(dims))
    z, y, x = np.meshgrid(*[np.arange(n) / n - 0.3 for n in (nz, ny, nx)], indexing="ij")
    r2 = (x * x + y * y + z * z) / 1.47                      # 0 near a corner, up to 1 in the opposite one
    psi = np.stack([np.exp(-100.0 * r2),                     # 2^-144 at the far corner
                    (x - 0.05) * np.exp(-60.0 * r2),         # with a nodal plane
                    rng.normal(size=r2.shape) * np.exp2(-130.0 * r2)])
    vloc, vavg = rng.normal(size=psi[0].size) - 1.0, 0.1 * rng.normal(size=psi[0].size)
    A = _terms(psi, h, {"isolated": (), "periodic": (0, 1, 2), "slab": (0, 1)}[bc])
    for v, w in ((None, None), (vloc, vavg)):
        got = _run(dims, h, psi.reshape(3, -1), bc, v, w)
        ref = oracle.hamiltonian_apply(psi.reshape(3, -1), (*dims, h, np.zeros(3)), v, w, bc=bc).reshape(psi.shape)
        vp = 0.0 if v is None else np.abs((v + w).reshape(psi.shape[1:]) * psi)
        tol = (64 * 2.0 ** -48 + 40 * 2.0 ** -53) * A + 4 * 2.0 ** -53 * (np.abs(ref) + vp)
        assert np.all(np.abs(got - ref) <= tol), float(np.max(np.abs(got - ref) / tol))
