"""Multigrid PCG solves of batches on either side of the rule that gives a level
to the one-launch coarse part: 24^3 points, level 0 in its own launches for few
orbitals and for more than one wave of them, in the one launch for nearly a
wave.  The launches show which way was taken.

Tolerance: as for the other multigrid solves, ||b - A V|| <= 1e-11 ||b|| leaves V
within 1e-9 max |V| of the discrete solution."""
import numpy as np
import pytest

from test_gpu_mg_coarse import _orbitals

pytestmark = pytest.mark.gpu


def _solve(dims, h, o, phi, ref, count):
    import torch
    from paper_2108_01186_gb300 import flosic as F
    n = len(phi)
    ctx = F.Context([dict(nx=dims[0], ny=dims[1], nz=dims[2], h=h, origin=list(o), norb=[n])] * (count // n),
                    precision=F.MIXED, cg_tol=1e-11, solver=F.SOLVER_PCG, preconditioner=1)
    V, iters, conv = ctx.orbital_poisson(torch.tensor(np.tile(phi.ravel(), count // n), device="cuda"))
    assert torch.all(conv == 1)
    err = np.abs(V.cpu().numpy().reshape(count // n, n, -1) - ref[None])
    assert np.max(err) < 1e-9 * np.max(np.abs(ref))
    return ctx.profile_read()["launches"] / int(iters.max())


def test_level_zero_is_fused_for_nearly_a_wave_of_orbitals_only():
    import torch
    import oracle
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    dims, h = (24, 24, 24), 0.4
    phi, o = _orbitals(dims, h, 5, seed=9)
    ref, _ = oracle.poisson(phi ** 2, (*dims, h, o), tol=1e-13)
    few, wave, more = (_solve(dims, h, o, phi, ref, n) for n in (5, sms // 5 * 5, sms // 5 * 5 + 10))
    # a level in its own launches takes four per V-cycle, so more than two per iteration on average
    assert few > wave + 2 and more > wave + 2
