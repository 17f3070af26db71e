"""Caller arrays that start on an 8-byte boundary only (a contiguous view such as
buf[1:]): the calls promise no more than the alignment of their elements, so the
16-byte accesses of aligned arrays have to give way to single ones.

Tolerances: V as for the other solves (||b - A V|| <= 1e-11 ||b|| leaves V within
1e-9 max |V| of the discrete solution); S within 1e-6 of the overlap, as for aligned
psi; H psi and the energies come from the same operations in the same order."""
import numpy as np
import pytest

from test_gpu_mg_coarse import _orbitals

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _odd(a):
    """a's values in a contiguous tensor 8 bytes off a 16-byte boundary."""
    buf = torch.empty(a.numel() + 2, dtype=torch.float64, device="cuda")
    at = 1 if buf.data_ptr() % 16 == 0 else 2
    v = buf[at:at + a.numel()]
    v.copy_(a.reshape(-1))
    assert v.is_contiguous() and v.data_ptr() % 16 == 8
    return v


@pytest.mark.parametrize("prec,solver", [("FP64", "PCG"), ("MIXED", "PCG"), ("MIXED", "AAR"), ("MIXED", "KRON")])
@pytest.mark.parametrize("dims", [(40, 24, 32), (33, 16, 20)])
def test_poisson_into_an_unaligned_potential(dims, prec, solver):
    import oracle
    from paper_2108_01186_gb300 import flosic as F
    h = 0.4
    phi, o = _orbitals(dims, h, 2, seed=sum(dims))
    ref, _ = oracle.poisson(phi ** 2, (*dims, h, o), tol=1e-13)
    ctx = F.Context([dict(nx=dims[0], ny=dims[1], nz=dims[2], h=h, origin=list(o), norb=[2])], cg_tol=1e-11,
                    precision=getattr(F, prec), solver=getattr(F, "SOLVER_" + solver))
    p = _odd(torch.tensor(phi.ravel(), device="cuda"))
    Va, _, _ = ctx.orbital_poisson(p.clone())
    # a cold start through the C entry (the binding allocates V itself), then a warm one
    V = _odd(torch.full_like(Va, 7.0))
    L = F.load_library()
    assert L.flosic_orbital_poisson(ctx._h, F._ptr(p), F._ptr(V), 0, None, None, F._stream()) == F.FLOSIC_OK
    W = _odd(1.01 * Va)
    ctx.orbital_poisson(p, V=W)
    for v in (V, W):
        assert np.max(np.abs(v.cpu().numpy().reshape(2, -1) - ref)) < 1e-9 * np.max(np.abs(ref))


@pytest.mark.parametrize("prec", ["FP64", "MIXED"])
def test_the_other_calls_on_unaligned_arrays(prec):
    from paper_2108_01186_gb300 import flosic as F
    from paper_2108_01186_gb300 import synth
    s = synth.make_system(24, 0.5, 2, [4], seed=11)
    ctx = F.Context([s], precision=getattr(F, prec), cg_tol=1e-10, solver=F.SOLVER_KRON if prec == "MIXED" else F.SOLVER_PCG)
    psi, fods = (torch.tensor(np.ascontiguousarray(a).ravel(), device="cuda") for a in (s.psi[0], s.fods[0]))
    phi, S, _ = ctx.build_flos(psi, fods)
    V, _, _ = ctx.orbital_poisson(phi)
    E, Vavg, U, Exc = ctx.sic_energy_potential(psi, phi, V)
    H = ctx.hamiltonian_apply(psi, None, Vavg)
    _, S2, _ = ctx.build_flos(_odd(psi), _odd(fods))
    assert torch.max(torch.abs(S2 - S)) < 2e-6
    E2, Vavg2, U2, Exc2 = ctx.sic_energy_potential(_odd(psi), _odd(phi), _odd(V))
    for a, b in ((E, E2), (Vavg, Vavg2), (U, U2), (Exc, Exc2)):
        assert torch.equal(a, b)
    out = _odd(torch.zeros_like(H))
    assert torch.equal(ctx.hamiltonian_apply(_odd(psi), None, _odd(Vavg), out=out), H)
    gE = torch.ones(1, dtype=torch.float64, device="cuda")
    ctx.build_flos(psi, fods)
    ctx.sic_energy_potential(psi, phi, V)
    d = ctx.sic_backward(psi, fods, phi, V, gE)
    ctx.sic_energy_potential(psi, phi, V)
    d2 = ctx.sic_backward(_odd(psi), _odd(fods), _odd(phi), _odd(V), gE)
    assert torch.equal(d[0], d2[0]) and torch.equal(d[1], d2[1])
