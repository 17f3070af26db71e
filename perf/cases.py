"""Performance cases of the FLO-SIC step, through the public Python entry points.

Every case is one call (or one short sequence of calls) of
``paper_2108_01186_gb300.flosic`` on seeded synthetic systems: normalised s and
p Gaussians on randomly placed atoms, random orthonormal combinations of them
as Kohn-Sham orbitals, one Fermi-orbital descriptor (FOD) per orbital near an
atom.  Gaussians are separable, so the inputs (and, where a case starts from
them, the Fermi-Loewdin orbitals) are one small matrix times the basis, built
on the GPU.

Kinds:

* ``flos``         Context.build_flos: psi, FODs -> phi, S, S^{-1/2}
* ``poisson``      Context.orbital_poisson: phi -> V, convergence flags
* ``energy``       Context.sic_energy_potential: psi, phi, V -> E, V_avg, U, Exc
* ``backward``     Context.sic_backward: -> dE/dpsi, dE/dfod
* ``hamiltonian``  Context.hamiltonian_apply: H psi
* ``step``         FlosicStep forward and backward (the autograd function)
* ``fod_step``     one energy and force evaluation of an FOD relaxation

``exact`` evaluates the same quantities in float64 with torch and numpy: the
12th-order Laplacian, l <= 2 multipole (isolated), neutralised periodic or
dipole-corrected slab boundaries, tricubic interpolation at the FODs, Loewdin
orthogonalisation, fully polarised LSDA, and the reverse mode of E_SIC with the
potential reused.
"""
import math
import random

import numpy as np
import torch

from paper_2108_01186_gb300 import flosic as F

# 12th-order centred second-derivative weights on a unit grid
_M = 6
_W = [0.0] + [2.0 * (-1) ** (k + 1) * math.factorial(_M) ** 2
              / (k * k * math.factorial(_M - k) * math.factorial(_M + k)) for k in range(1, _M + 1)]
_W[0] = -2.0 * sum(1.0 / (k * k) for k in range(1, _M + 1))

_PERIODIC = {"isolated": (), "periodic": (0, 1, 2), "slab": (0, 1)}
_BC = {"isolated": F.BC_ISOLATED, "periodic": F.BC_PERIODIC, "slab": F.BC_SLAB}
_SOLVER = {"pcg": F.SOLVER_PCG, "kron": F.SOLVER_KRON}
_PREC = {"fp64": F.FP64, "mixed": F.MIXED}


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def _case(name, kind, n, h, norb, solver="kron", precision="mixed", boundary="isolated", scale=1.0):
    """n: side lengths "nx,ny,nz" (one system) or "n;n;..." (cubes of a batch);
    norb: orbitals per spin "N[,N]", one entry per system."""
    c = dict(kind=kind, n=n, h=h, norb=norb, solver=solver, precision=precision, boundary=boundary, scale=scale)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The plain float64 step on the smallest molecule (40^3, 5 orbitals, one
        # spin): energies, V_avg and both gradients; latency-bound.
        _case("step_fp64_40", "step", "40,40,40", 0.3, "5", solver="pcg", precision="fp64"),
        # One energy and force evaluation of an FOD relaxation on a mid-size
        # two-spin molecule with the scaled potential.
        _case("fod_step_96", "fod_step", "96,96,96", 0.2, "16,16", scale=0.5),
        # The Poisson solves of a small molecule: few points, launches count.
        _case("poisson_40", "poisson", "40,40,40", 0.3, "5"),
        # ... of the benchmark's molecule (both spins in one batch).
        _case("poisson_128", "poisson", "128,128,128", 0.2, "32,32"),
        # ... on a box whose odd sides fit no tile.
        _case("poisson_117", "poisson", "117,117,117", 0.2, "20"),
        # ... on the fine grid of the largest molecules (one spin's share).
        _case("poisson_192", "poisson", "192,192,192", 0.15, "24"),
        # ... with the library's default inner solver (multigrid PCG).
        _case("poisson_pcg_64", "poisson", "64,64,64", 0.25, "10", solver="pcg"),
        # ... of a batch of independent molecules of uneven grids and orbital counts.
        _case("poisson_batch", "poisson", "48;61;75;88;104;127", 0.2, "7;22;13;38;9;17"),
        # The four grid passes around the solves at the benchmark's size.
        _case("flos_128", "flos", "128,128,128", 0.2, "32,32"),
        _case("energy_128", "energy", "128,128,128", 0.2, "32,32", scale=0.5),
        _case("backward_128", "backward", "128,128,128", 0.2, "32,32"),
        # The averaged-SIC Hamiltonian of a self-consistency iteration.
        _case("hamiltonian_128", "hamiltonian", "128,128,128", 0.2, "32,32"),
    ]


def _max_norb(sides, h):
    """Orbitals that fit the box: two per atom, atoms 2 bohr apart."""
    half = [_half_width(s, h) for s in sides]
    cells = 1.0
    for w in half:
        cells *= w + 1.0
    return max(2, 2 * int(0.3 * cells))


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "fod_step", "poisson", "poisson", "poisson", "poisson", "pcg", "batch", "flos",
                       "energy", "backward", "hamiltonian"])
    h = round(rng.uniform(0.15, 0.3), 3)
    if kind == "batch":
        k = rng.randint(3, 8)
        sides, norbs, left = [], [], 82e6
        for _ in range(k):
            n = rng.randint(48, 128)
            N = min(rng.randint(2, 40), _max_norb((n, n, n), h), max(2, int(left / n ** 3 / 2)))
            if n ** 3 * N > left:
                break
            left -= n ** 3 * N
            sides.append(str(n))
            norbs.append(str(N))
        return _case(None, "poisson", ";".join(sides), h, ";".join(norbs))
    # (smallest side, largest side, most orbitals a spin, most orbital points)
    lo, hi, most, points = {
        "step": (20, 48, 8, 4e5), "fod_step": (32, 128, 40, 2.8e7), "poisson": (32, 192, 64, 1.3e8),
        "pcg": (32, 96, 16, 2.6e6), "flos": (32, 160, 64, 1.3e8), "energy": (32, 160, 64, 1.3e8),
        "backward": (32, 160, 64, 1.3e8), "hamiltonian": (32, 160, 64, 1.3e8)}[kind]
    n = _log_int(rng, lo, hi)
    if rng.random() < 0.4:
        n = max(lo, n // 8 * 8)          # boxes are often chosen for the tiles
    sides = [n, n, n]
    if rng.random() < 0.25:              # a box around a long or flat molecule
        sides = [max(lo, min(hi, int(n * rng.uniform(0.75, 1.2)))) for _ in range(3)]
    G = sides[0] * sides[1] * sides[2]
    nspin = rng.choice([1, 2])
    top = max(1, min(most, _max_norb(sides, h), int(points / G / nspin)))
    N = _log_int(rng, min(2, top), top)
    norb = [N] if nspin == 1 else [N, max(1, N - rng.choice([0, 0, 1, 2]))]
    boundary = "isolated"
    if kind == "poisson" and rng.random() < 0.2:
        boundary = rng.choice(["periodic", "slab"])
    c = _case(None, "poisson" if kind == "pcg" else kind, ",".join(map(str, sides)), h, ",".join(map(str, norb)),
              solver="pcg" if kind in ("step", "pcg") else "kron", precision="fp64" if kind == "step" else "mixed",
              boundary=boundary)
    if kind in ("energy", "fod_step"):
        c["scale"] = rng.choice([0.5, 1.0])
    return c


def _systems(case):
    """[(sides, norb per spin)] of the case's batch."""
    out = []
    for n, N in zip(case["n"].split(";"), case["norb"].split(";")):
        s = [int(x) for x in n.split(",")]
        out.append((tuple(s * 3 if len(s) == 1 else s), [int(x) for x in N.split(",")]))
    return out


def work(case):
    """Bytes: each input read once, each output written once.  Flops: the
    products with N x N matrices; one Kronecker inverse by half-size products
    per solve; about 60 per point for LSDA; the stencil's multiply-adds."""
    by = fl = 0.0
    for (nx, ny, nz), norb in _systems(case):
        G = nx * ny * nz
        side = 2.0 * (nx + ny + nz)
        for N in norb:
            P = float(N) * G
            b = {"flos": 16 * P, "poisson": 16 * P, "energy": 24 * P + 8 * G, "backward": 20 * P,
                 "hamiltonian": 16 * P + 16 * G, "step": 16 * P + 8 * G, "fod_step": 8 * P}[case["kind"]]
            f = {"flos": 4 * N * P, "poisson": side * P, "energy": 60 * P, "backward": 6 * N * P,
                 "hamiltonian": 58 * P, "step": (10 * N + 60 + side) * P,
                 "fod_step": (6 * N + 60 + side) * P}[case["kind"]]
            by += b
            fl += f
    return {"bytes": by, "flops": fl}


# --------------------------------------------------------------------------
# seeded systems
# --------------------------------------------------------------------------

def _half_width(n, h):
    L = n * h
    return L / 2.0 - min(6.0, 0.4 * L)


class _System:
    """Atoms, basis, orbital coefficients and FODs of one system."""

    def __init__(self, sides, h, norb, boundary, rng):
        self.sides, self.h, self.norb, self.boundary = sides, h, norb, boundary
        self.per = _PERIODIC[boundary]
        self.origin = [-0.5 * h * (n - 1) for n in sides]
        L = [n * h for n in sides]
        box = [l / 2.0 if d in self.per else _half_width(n, h) for d, (l, n) in enumerate(zip(L, sides))]
        sep, tries, atoms = 2.0, 0, []
        while len(atoms) < (max(norb) + 1) // 2:
            x = [rng.uniform(-w, w) for w in box]
            tries += 1
            if tries % 2000 == 0:
                sep *= 0.9                       # a crowded box
            if all(math.dist(x, a) >= sep for a in atoms):
                atoms.append(x)
        self.blocks = []
        for N in norb:
            fun = [(a, lm, rng.uniform(0.3, 3.0)) for a in atoms for lm in range(4)]
            g1 = [self._factors(d, fun) for d in range(3)]      # per direction [nb, n]
            over = h ** 3 * (g1[0] @ g1[0].T) * (g1[1] @ g1[1].T) * (g1[2] @ g1[2].T)
            C = np.array([[rng.gauss(0.0, 1.0) for _ in fun] for _ in range(N)])
            C = np.linalg.solve(np.linalg.cholesky(C @ over @ C.T), C)   # dV psi psi^T = 1
            fods = []
            while len(fods) < N:
                a = atoms[len(fods) % len(atoms)]
                v = [rng.gauss(0.0, 1.0) for _ in range(3)]
                r = 0.5 * rng.random() ** (1.0 / 3.0) / math.sqrt(sum(q * q for q in v))
                x = [p + r * q for p, q in zip(a, v)]
                if all(math.dist(x, f) >= 0.3 for f in fods):
                    fods.append(x)
            self.blocks.append(dict(fun=fun, g1=g1, C=C, fods=np.array(fods)))

    def _factors(self, d, fun):
        """1-D factors along direction d of every basis function, summed over
        periodic images two cells away."""
        x = self.origin[d] + self.h * np.arange(self.sides[d])
        L = self.h * self.sides[d]
        out = np.zeros((len(fun), x.size))
        for b, (a, lm, al) in enumerate(fun):
            for k in (range(-2, 3) if d in self.per else (0,)):
                u = x - a[d] - k * L
                g = (2.0 * al / math.pi) ** 0.25 * np.exp(-al * u * u)
                out[b] += 2.0 * math.sqrt(al) * u * g if lm == d + 1 else g
        return out

    def fields(self, blk, C):
        """[rows of C][G] on the GPU: C times the basis."""
        gx, gy, gz = (torch.tensor(g, device="cuda") for g in blk["g1"])
        C = torch.as_tensor(C, device="cuda")
        xy = (gy[:, :, None] * gx[:, None, :]).reshape(gx.shape[0], -1)            # [nb, ny nx]
        left = (C[:, None, :] * gz.T[None, :, :]).reshape(-1, gx.shape[0])         # [N nz, nb]
        return (left @ xy).reshape(C.shape[0], -1)

    def nodes(self, blk):
        """Tricubic Lagrange nodes and weights of every FOD along each
        direction: index [N, 4] (-1 outside), weights and derivatives [N, 4]."""
        out = []
        for d in range(3):
            n = self.sides[d]
            u = (blk["fods"][:, d] - self.origin[d]) / self.h
            if d in self.per:
                u = u - n * np.floor(u / n)
            i0 = np.floor(u).astype(int)
            t = u - i0
            L = np.stack([-t * (t - 1) * (t - 2) / 6, (t + 1) * (t - 1) * (t - 2) / 2,
                          -(t + 1) * t * (t - 2) / 2, (t + 1) * t * (t - 1) / 6], 1)
            dL = np.stack([-(3 * t * t - 6 * t + 2) / 6, (3 * t * t - 4 * t - 1) / 2,
                           -(3 * t * t - 2 * t - 2) / 2, (3 * t * t - 1) / 6], 1) / self.h
            q = i0[:, None] + np.arange(-1, 3)[None, :]
            q = q % n if d in self.per else np.where((q >= 0) & (q < n), q, -1)
            ok = q >= 0
            out.append((q, L * ok, dL * ok))
        return out

    def loewdin(self, blk):
        """psi and grad psi at the FODs, T, S, its eigenpairs and S^{-1/2}."""
        ev = []
        for d, (q, L, dL) in enumerate(self.nodes(blk)):
            g = blk["g1"][d][:, np.maximum(q, 0)]                                   # [nb, N, 4]
            ev.append(((g * L).sum(-1), (g * dL).sum(-1)))
        (x, dx), (y, dy), (z, dz) = ev
        vals = (blk["C"] @ (x * y * z)).T                                           # [FOD, orbital]
        grads = np.stack([(blk["C"] @ p).T for p in (dx * y * z, x * dy * z, x * y * dz)], -1)
        rho = (vals ** 2).sum(1)
        T = vals / np.sqrt(rho)[:, None]
        over = self.h ** 3
        for g in blk["g1"]:
            over = over * (g @ g.T)
        TC = T @ blk["C"]
        S = TC @ over @ TC.T
        lam, U = np.linalg.eigh(S)
        Q = (U / np.sqrt(lam)) @ U.T
        return dict(vals=vals, grads=grads, rho=rho, T=T, S=S, lam=lam, U=U, Q=Q)


def _make(case, seed):
    rng = random.Random("%d %s %s" % (seed, case["n"], case["norb"]))
    return [_System(s, case["h"], N, case["boundary"], rng) for s, N in _systems(case)]


def _cat(parts):
    return torch.cat([p.reshape(-1) for p in parts])


def _psi(systems):
    return _cat([s.fields(b, b["C"]) for s in systems for b in s.blocks])


def _phi(systems):
    out = []
    for s in systems:
        for b in s.blocks:
            lo = s.loewdin(b)
            out.append(s.fields(b, lo["Q"] @ lo["T"] @ b["C"]))
    return out


def _fods(systems):
    return torch.tensor(np.concatenate([b["fods"].reshape(-1) for s in systems for b in s.blocks]), device="cuda")


# --------------------------------------------------------------------------
# float64 reference
# --------------------------------------------------------------------------

def _operator(n, h, periodic):
    """-d^2/dx^2 on n points (zero outside, or wrapped): eigenpairs."""
    A = np.zeros((n, n))
    for k in range(-_M, _M + 1):
        w = -_W[abs(k)] / (h * h)
        for i in range(n):
            if 0 <= i + k < n:
                A[i, i + k] += w
            elif periodic:
                A[i, (i + k) % n] += w
    return np.linalg.eigh(A)


def _along(M, f, d):
    """M applied along direction d (x = 0) of f [..., nz, ny, nx]."""
    if d == 0:
        return f @ M.T
    if d == 1:
        return M @ f
    return (M @ f.reshape(f.shape[0], f.shape[1], -1)).reshape(f.shape)


def _moments(s, rho):
    dV = s.h ** 3
    c = [torch.arange(n, device="cuda", dtype=torch.float64) * s.h - 0.5 * s.h * (n - 1) for n in s.sides]
    X, Y, Z = c[0][None, None, :], c[1][None, :, None], c[2][:, None, None]
    r2 = X * X + Y * Y + Z * Z
    basis = [torch.ones_like(r2), X + 0 * r2, Y + 0 * r2, Z + 0 * r2, 3 * X * X - r2, 3 * Y * Y - r2, 3 * Z * Z - r2,
             3 * X * Y + 0 * r2, 3 * X * Z + 0 * r2, 3 * Y * Z + 0 * r2]
    return dV * rho.reshape(rho.shape[0], -1) @ torch.stack([b.reshape(-1) for b in basis], 1)


def _multipole(m, X, Y, Z):
    m = [m[:, k].reshape(-1, 1, 1, 1) for k in range(10)]
    r2 = X * X + Y * Y + Z * Z
    r = torch.sqrt(r2)
    quad = m[4] * X * X + m[5] * Y * Y + m[6] * Z * Z + 2 * (m[7] * X * Y + m[8] * X * Z + m[9] * Y * Z)
    return m[0] / r + (m[1] * X + m[2] * Y + m[3] * Z) / (r2 * r) + 0.5 * quad / (r2 * r2 * r)


def _add_ghosts(s, rho, b):
    """Adds the Dirichlet values on the ghost layers to the right-hand side b."""
    c = [torch.arange(n, device="cuda", dtype=torch.float64) * s.h - 0.5 * s.h * (n - 1) for n in s.sides]
    mom = None
    if s.boundary == "isolated":
        mom = _moments(s, rho)
    for d in range(3):
        if d in s.per:
            continue
        n = s.sides[d]
        for side in (0, 1):
            q = torch.arange(-_M, 0, device="cuda") if side == 0 else torch.arange(n, n + _M, device="cuda")
            u = q.to(torch.float64) * s.h - 0.5 * s.h * (n - 1)
            ax = list(c)
            ax[d] = u
            X, Y, Z = ax[0][None, None, None, :], ax[1][None, None, :, None], ax[2][None, :, None, None]
            if mom is not None:
                vb = _multipole(mom, X, Y, Z)
            else:
                dV = s.h ** 3
                planes = dV * rho.sum((2, 3))
                Q, pz = planes.sum(1), planes @ c[2]
                area = s.sides[0] * s.sides[1] * s.h ** 2
                vb = (-2 * math.pi / area) * (Q[:, None] * u.abs()[None, :] - torch.sign(u)[None, :] * pz[:, None])
                vb = vb.reshape(rho.shape[0], -1, 1, 1).expand(-1, -1, s.sides[1], s.sides[0])
            near = min(n, _M)
            p = torch.arange(near, device="cuda") + (0 if side == 0 else n - near)
            dist = (p[:, None] - q[None, :]).abs()
            W = torch.tensor(_W + [0.0] * (2 * _M), device="cuda", dtype=torch.float64)[dist.clamp(max=_M + 1)]
            W = W / (s.h * s.h)
            add = _along(W, vb.contiguous(), d) if d < 2 else (W @ vb.reshape(vb.shape[0], _M, -1)).reshape(
                vb.shape[0], near, s.sides[1], s.sides[0])
            at = [slice(None)] * 4
            at[3 - d] = slice(int(p[0]), int(p[-1]) + 1)
            b[tuple(at)] += add
    return b


def _solve(s, phi):
    """V of every row of phi [N, G]: -Delta_h V = 4 pi phi^2 with the system's boundary."""
    nx, ny, nz = s.sides
    eig = [_operator(n, s.h, d in s.per) for d, n in enumerate(s.sides)]
    lam = [torch.tensor(e[0], device="cuda") for e in eig]
    Q = [torch.tensor(e[1], device="cuda") for e in eig]
    den = lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
    zero = None
    if len(s.per) == 3:
        zero = den < 1e-9 * float(den.max())
        den = torch.where(zero, torch.ones_like(den), den)
    V = torch.empty_like(phi)
    rows = max(1, int(1.5e8 // phi.shape[1]))
    for i in range(0, phi.shape[0], rows):
        rho = (phi[i:i + rows] ** 2).reshape(-1, nz, ny, nx)
        b = 4 * math.pi * rho
        if len(s.per) == 3:
            b -= b.mean((1, 2, 3), keepdim=True)
        else:
            b = _add_ghosts(s, rho, b)
        for d in range(3):
            b = _along(Q[d].T.contiguous(), b, d)
        b /= den
        if zero is not None:
            b[:, zero] = 0.0
        for d in range(3):
            b = _along(Q[d], b, d)
        V[i:i + rows] = b.reshape(b.shape[0], -1)
    return V


def _lsda(n):
    """eps_xc and v_xc of the spin densities (n, 0): Slater exchange, PW92 correlation at zeta = 1."""
    A, a1, b1, b2, b3, b4 = 0.015545, 0.20548, 14.1189, 6.1977, 3.3662, 0.62517
    on = n > 1e-30
    n = torch.where(on, n, torch.ones_like(n))
    k = (6.0 * n / math.pi) ** (1.0 / 3.0)
    rs = (3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
    sr = torch.sqrt(rs)
    q0 = -2.0 * A * (1.0 + a1 * rs)
    q1 = 2.0 * A * (b1 * sr + b2 * rs + b3 * rs * sr + b4 * rs * rs)
    dq1 = A * (b1 / sr + 2.0 * b2 + 3.0 * b3 * sr + 4.0 * b4 * rs)
    lg = torch.log1p(1.0 / q1)
    ec = q0 * lg
    dec = -2.0 * A * a1 * lg - q0 * dq1 / (q1 * q1 + q1)
    zero = torch.zeros_like(n)
    return torch.where(on, ec - 0.75 * k, zero), torch.where(on, ec - rs / 3.0 * dec - k, zero)


def _energy(s, psi, phi, V, scale):
    """(U, Exc, V_avg, V^SIC) of one spin block, orbital by orbital."""
    dV = s.h ** 3
    U, X = [], []
    num = torch.zeros_like(psi[0])
    vs = torch.empty_like(phi)
    for i in range(phi.shape[0]):
        rho = phi[i] ** 2
        eps, v = _lsda(rho)
        U.append(0.5 * dV * (rho * V[i]).sum())
        X.append(dV * (rho * eps).sum())
        vs[i] = -(V[i] + v)
        num += rho * vs[i]
    rs = (psi ** 2).sum(0)
    on = rs > 1e-30
    return torch.stack(U), torch.stack(X), torch.where(on, scale * num / torch.where(on, rs, 1.0), 0.0), vs


def _backward(s, blk, lo, psi, phi, vsic, want_dpsi=True):
    """dE_SIC/dpsi [N, G] and dE_SIC/dfod [N, 3] of one spin block."""
    dV = s.h ** 3
    T, Q, U, lam = lo["T"], lo["Q"], lo["U"], lo["lam"]
    bar = 2.0 * dV * vsic * phi                       # dE/dphi
    P = (bar @ psi.T).cpu().numpy()                   # <bar_k | psi_a> on the grid
    Qb = P @ T.T
    a = np.sqrt(lam)
    K = -1.0 / (a[:, None] * a[None, :] * (a[:, None] + a[None, :]))
    Sb = U @ ((U.T @ Qb @ U) * K) @ U.T
    Sb = Sb + Sb.T
    # F-bar = Q^T bar + dV Sb F; psi-bar = T^T F-bar; T-bar = F-bar psi^T
    over = dV * (psi @ psi.T).cpu().numpy()
    Tb = Q.T @ P + Sb @ T @ over
    vals, rho = lo["vals"], lo["rho"]
    sq = np.sqrt(rho)
    vb = Tb / sq[:, None] - vals * ((Tb * vals).sum(1) / (rho * sq))[:, None]
    dfod = torch.tensor(np.einsum("ia,iad->id", vb, lo["grads"]), device="cuda")
    if not want_dpsi:
        return None, dfod
    dpsi = torch.tensor(T.T @ Q.T, device="cuda") @ bar
    dpsi += torch.tensor(dV * T.T @ Sb @ T, device="cuda") @ psi
    (qx, Lx, _), (qy, Ly, _), (qz, Lz, _) = s.nodes(blk)
    nx, ny, _ = s.sides
    for i in range(vb.shape[0]):
        at = (np.maximum(qz[i], 0)[:, None, None] * ny + np.maximum(qy[i], 0)[None, :, None]) * nx \
            + np.maximum(qx[i], 0)[None, None, :]
        w = Lz[i][:, None, None] * Ly[i][None, :, None] * Lx[i][None, None, :]
        dpsi.index_add_(1, torch.tensor(at.reshape(-1), device="cuda"),
                        torch.tensor(vb[i][:, None] * w.reshape(1, -1), device="cuda"))
    return dpsi, dfod


def _hamiltonian(s, psi, v):
    nx, ny, nz = s.sides
    out = torch.empty_like(psi)
    for i in range(psi.shape[0]):
        f = psi[i].reshape(nz, ny, nx)
        lap = 3.0 * _W[0] * f
        for k in range(1, _M + 1):
            for d in range(3):
                m = f.shape[d] - k
                if m > 0:
                    lap.narrow(d, 0, m).add_(f.narrow(d, k, m), alpha=_W[k])
                    lap.narrow(d, k, m).add_(f.narrow(d, 0, m), alpha=_W[k])
        out[i] = (-0.5 / (s.h * s.h) * lap).reshape(-1) + v * psi[i]
    return out


def exact(case, seed):
    systems = _make(case, seed)
    kind = case["kind"]
    if kind == "poisson":
        it = iter(_phi(systems))
        return _cat([_solve(s, next(it)) for s in systems for _ in s.blocks]), None
    if kind == "hamiltonian":
        out = []
        for s, vl, va in _fields(systems, seed):
            for b, v in zip(s.blocks, va):
                out.append(_hamiltonian(s, s.fields(b, b["C"]), vl + v))
        return _cat(out)
    phis, Ss, Qs, E, Us, Xs, Va, dp, df = [], [], [], [], [], [], [], [], []
    for s in systems:
        e = 0.0
        for b in s.blocks:
            lo = s.loewdin(b)
            phi = s.fields(b, lo["Q"] @ lo["T"] @ b["C"])
            if kind == "flos":
                phis.append(phi)
                Ss.append(torch.tensor(lo["S"], device="cuda"))
                Qs.append(torch.tensor(lo["Q"], device="cuda"))
                continue
            psi = s.fields(b, b["C"])
            U, X, v, vs = _energy(s, psi, phi, _solve(s, phi), case["scale"])
            e = e - (U + X).sum()
            Us.append(U)
            Xs.append(X)
            Va.append(v)
            if kind != "energy":
                p, f = _backward(s, b, lo, psi, phi, vs, kind != "fod_step")
                dp.append(p)
                df.append(f)
        E.append(e)
    if kind == "flos":
        return _cat(phis), _cat(Ss), _cat(Qs)
    if kind == "backward":
        return _cat(dp), _cat(df)
    E, Us, Xs = torch.stack(E), _cat(Us), _cat(Xs)
    if kind == "energy":
        return E, _cat(Va), Us, Xs
    if kind == "fod_step":
        return E, Us, Xs, _cat(df)
    return E, _cat(Va), Us, Xs, _cat(dp), _cat(df)


# --------------------------------------------------------------------------
# a case's state and its pass
# --------------------------------------------------------------------------

def _fields(systems, seed):
    """Per system: a smooth local potential (wells at the box centre) and one
    averaged potential per spin block."""
    rng = random.Random(seed + 1)
    for s in systems:
        x = [torch.arange(n, device="cuda", dtype=torch.float64) * s.h - 0.5 * s.h * (n - 1) for n in s.sides]
        r2 = x[2][:, None, None] ** 2 + x[1][None, :, None] ** 2 + x[0][None, None, :] ** 2
        wells = [(-rng.uniform(0.5, 4.0) * torch.exp(-rng.uniform(0.02, 0.3) * r2)).reshape(-1)
                 for _ in range(1 + len(s.blocks))]
        yield s, wells[0], wells[1:]


def prepare(case, seed):
    systems = _make(case, seed)
    kind = case["kind"]
    ctx = F.Context([dict(nx=s.sides[0], ny=s.sides[1], nz=s.sides[2], h=s.h, origin=s.origin, norb=s.norb)
                     for s in systems],
                    precision=_PREC[case["precision"]], solver=_SOLVER[case["solver"]],
                    boundary=_BC[case["boundary"]])
    st = dict(kind=kind, ctx=ctx, scale=case["scale"])
    if kind == "poisson":
        st["phi"] = _cat(_phi(systems))
        return st
    st["psi"] = _psi(systems)
    if kind == "hamiltonian":
        f = list(_fields(systems, seed))
        st["vloc"] = _cat([v for _, v, _ in f])
        st["vavg"] = _cat([v for _, _, va in f for v in va])
        return st
    st["fods"] = _fods(systems)
    if kind in ("energy", "backward"):
        phi = _phi(systems)
        it = iter(phi)
        st["V"] = _cat([_solve(s, next(it)) for s in systems for _ in s.blocks])
        st["phi"] = _cat(phi)
    if kind == "backward":   # the forward step that the reverse mode belongs to
        st["phi"] = ctx.build_flos(st["psi"], st["fods"])[0]
        ctx.sic_energy_potential(st["psi"], st["phi"], st["V"])
        st["gE"] = torch.ones(ctx.nsys, dtype=torch.float64, device="cuda")
    if kind == "fod_step":
        st["gE"] = torch.ones(ctx.nsys, dtype=torch.float64, device="cuda")
    if kind == "step":
        st["psi"].requires_grad_(True)
        st["fods"].requires_grad_(True)
    return st


def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "poisson":
        V, _, conv = ctx.orbital_poisson(st["phi"])
        return V, conv
    if kind == "hamiltonian":
        return ctx.hamiltonian_apply(st["psi"], st["vloc"], st["vavg"])
    if kind == "flos":
        return ctx.build_flos(st["psi"], st["fods"])
    if kind == "energy":
        return ctx.sic_energy_potential(st["psi"], st["phi"], st["V"], st["scale"])
    if kind == "backward":
        return ctx.sic_backward(st["psi"], st["fods"], st["phi"], st["V"], st["gE"])
    if kind == "fod_step":
        out = ctx.forward(st["psi"], st["fods"], scale=st["scale"])
        _, dfod = ctx.sic_backward(st["psi"], st["fods"], out["phi"], out["V"], st["gE"], want_dpsi=False)
        return out["E_sic"], out["U"], out["Exc"], dfod
    E, Vavg, U, Exc = F.FlosicStep.apply(ctx, st["psi"], st["fods"], st["scale"])
    dpsi, dfod = torch.autograd.grad(E.sum(), (st["psi"], st["fods"]))
    return E.detach(), Vavg, U, Exc, dpsi, dfod
