"""The work that is measured: calls of libemd as a user's program makes them.

Each case is one kind of call on one synthetic system (the jittered lattices
of Si-like pseudo-atoms that the tests and the benchmark use, two doubly
occupied orbitals per atom):

  md       n_steps MD steps and the read-out of the state they lead to
  sampled  an MD run that reads energy and forces every few steps
  batch    n_steps MD steps of several replicas of uneven size
  adjoint  the gradient of the final energy with respect to the initial ion
           positions and the field amplitudes of every step
  ground   the Kohn-Sham ground state at fixed ions
  poisson  the Poisson solve on device buffers

``exact`` restates the same results in plain torch, 64 bits, without the
library.
"""
from __future__ import annotations

import ctypes
import dataclasses
import math

import numpy as np
import torch

from paper_0812_2801_gb300 import emd, inputs


def listed():
    si = dict(kind="md", fp64=True, lmax=0, field=False, mu=10.0)
    return [
        # the smallest call: one Poisson solve inside a caller's own loop
        dict(name="poisson_48", kind="poisson", n=48, h=0.3),
        # the BO start of every run of the paper, on a closed-shell dimer
        dict(name="ground_dimer_24", kind="ground", n=24, h=0.4, order=8),
        # vibrations against mu: a long run of a small molecule, sampled
        dict(name="sampled_dimer_48", kind="sampled", n=48, h=0.3, order=8, mu=10.0,
             every=6, samples=4),
        # the FP64 form on the smallest workload (8 atoms, order 4)
        dict(si, name="fp64_tiny_32", n=32, h=0.3, order=4, cells=2, steps=24),
        # a driven FP64 run: field amplitudes per step, order 6, 27 atoms
        dict(si, name="fp64_field_64", n=64, h=0.3, order=6, cells=3, steps=6, field=True),
        # s, p and d projectors on every atom
        dict(si, name="fp64_lmax2_48", n=48, h=0.25, order=8, cells=2, lmax=2, steps=6),
        # the FP64 form of the precision workload: 64 atoms, 128 orbitals, 96^3
        dict(si, name="fp64_c96", n=96, h=0.25, order=8, cells=4, steps=3),
        # the same in complex64 orbitals, the benchmark's headline workload
        dict(si, name="c64_c96", n=96, h=0.25, order=8, cells=4, steps=12, fp64=False),
        # one small complex64 trajectory on its own
        dict(si, name="c64_c48", n=48, h=0.25, order=8, cells=2, steps=12, fp64=False),
        # a cluster in a large box: the grid weighs more, tiles and orbital blocks are ragged
        dict(si, name="c64_c120", n=120, h=0.25, order=8, cells=3, steps=12, fp64=False),
        # ragged replicas advanced together
        dict(name="batch_8", kind="batch", replicas=8, big=4, order=8, mu=10.0, steps=12),
        # field optimisation: the gradient through a trajectory with moving ions
        dict(name="adjoint_64", kind="adjoint", n=64, h=0.3, order=6, cells=2, steps=8, every=4),
    ]


#: grids that the FFT takes, odd and ragged ones among them
SIZES = (16, 18, 20, 21, 22, 24, 26, 27, 28, 30, 32, 33, 35, 36, 39, 40, 42, 44, 45, 48, 49, 50, 52, 54, 55, 56,
         60, 63, 64, 65, 66, 70, 72, 75, 77, 78, 80, 81, 84, 88, 90, 91, 96, 98, 99, 100, 104, 108, 110, 112)


def _log_size(rng, lo, hi):
    """One of SIZES, spread over the logarithm of the number of points."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((n for n in SIZES if lo <= n <= hi), key=lambda n: abs(math.log(n / x)))


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md", "sampled", "batch", "adjoint", "ground", "poisson"])
    if kind == "poisson":
        return dict(kind=kind, n=_log_size(rng, 16, 64), h=round(rng.uniform(0.2, 0.4), 3))
    if kind == "ground":
        n = rng.choice([20, 21, 22, 24, 27, 28])
        return dict(kind=kind, n=n, h=round(9.6 / n, 4), order=rng.choice([4, 6, 8]))
    if kind == "sampled":
        return dict(kind=kind, n=_log_size(rng, 30, 64), h=0.3, order=rng.choice([4, 6, 8]), mu=rng.choice([5.0, 10.0, 20.0]),
                    every=rng.randint(1, 9), samples=rng.randint(2, 4))
    if kind == "batch":
        m = rng.randint(2, 8)
        return dict(kind=kind, replicas=m, big=rng.randint(0, m // 2), order=rng.choice([4, 6, 8]), mu=rng.choice([10.0, 50.0]),
                    steps=rng.randint(6, 13))
    order = rng.choice([2, 4, 6, 8, 8])
    h = rng.uniform(0.25, 0.33)
    if kind == "adjoint":
        n = _log_size(rng, 30, 64)
        h = round(max(h, 9.7 / n), 4)
        return dict(kind=kind, n=n, h=h, order=order, cells=max(2, int(n * h / 5.6)), steps=rng.randint(3, 8), every=rng.randint(2, 4))
    n = _log_size(rng, 30, 100)
    h = round(max(h, 9.7 / n), 4)
    fp64 = rng.random() < 0.5
    field = rng.random() < 0.25
    lmax = rng.choice([0, 0, 1, 2]) if fp64 and n <= 56 else 0
    cells = max(2, int(n * h / rng.uniform(4.9, 10.0)))
    while 2 * cells ** 3 * n ** 3 > 1.2e8:
        cells -= 1
    work = 2 * cells ** 3 * n ** 3                       # orbital points
    steps = max(1, min(rng.randint(6, 24), int((2e8 if fp64 else 1.2e9) / (work * (1 + 2 * lmax)))))
    return dict(kind="md", n=n, h=h, order=order, cells=cells, steps=steps, fp64=fp64, lmax=lmax, field=field, mu=rng.choice([10.0, 10.0, 50.0]))


# ---- inputs ----------------------------------------------------------------

def _species(case):
    if case.get("lmax", 0) == 0:
        return inputs.SI_LIKE
    return dataclasses.replace(inputs.SI_LIKE, lmax=case["lmax"], h_l=(0.6, 0.4))


def _dt(mu):
    return 0.05 * math.sqrt(mu)


def _gauss(coord, c, L, sigma, moment):
    """Image-summed 1-D factors d^moment exp(-d^2 / 2 sigma^2), [atoms, n]."""
    d = coord[None, None, :] - c[:, None, None] - L * torch.tensor([-1.0, 0.0, 1.0], dtype=torch.float64, device="cuda")[None, :, None]
    g = torch.exp(-d * d / (2 * sigma * sigma))
    return (d * g if moment else g).sum(1)


def _orbitals(n, h, R, rng, extra_px=False):
    """Orthonormal s and p_z Gaussians per atom with random phases (as the
    tests start from), [n_orb, n, n, n] on the GPU; extra_px adds a p_x
    function on the first atom."""
    L, sigma = n * h, 1.2
    x = torch.arange(n, dtype=torch.float64, device="cuda") * h
    Rt = torch.from_numpy(R).cuda()
    s = [_gauss(x, Rt[:, a], L, sigma, False) for a in range(3)]
    z1 = _gauss(x, Rt[:, 2], L, sigma, True)
    X, Y = s[0].repeat_interleave(2, 0), s[1].repeat_interleave(2, 0)
    Z = torch.stack([s[2], z1], 1).reshape(-1, n)
    if extra_px:
        X = torch.cat([X, _gauss(x, Rt[:1, 0], L, sigma, True)])
        Y, Z = torch.cat([Y, s[1][:1]]), torch.cat([Z, s[2][:1]])
    m = X.shape[0]
    ph = torch.from_numpy(np.exp(1j * rng.uniform(0, 2 * math.pi, m))).cuda()
    S = h ** 3 * (ph.conj()[:, None] * ph[None]) * (X @ X.T) * (Y @ Y.T) * (Z @ Z.T)
    M = torch.linalg.inv(torch.linalg.cholesky(S).conj()) * ph[None]
    dt = torch.complex64 if m * n ** 3 > 1 << 23 else torch.complex128
    out = torch.empty((m, n, n * n), dtype=dt, device="cuda")
    P = (Y[:, :, None] * X[:, None, :]).reshape(m, n * n).to(dt)
    for z in range(n):
        out[:, z] = (M * Z[None, :, z]).to(dt) @ P
    return out.reshape(m, n, n, n)


def _lattice(case, seed):
    """R, V, orbitals and field of a jittered simple-cubic lattice."""
    rng = np.random.default_rng([seed, case["n"], case["cells"]])
    L = case["n"] * case["h"]
    sites = inputs.lattice_sites("sc", case["cells"], L / case["cells"])
    if "atoms" in case:
        sites = sites[np.sort(rng.choice(len(sites), case["atoms"], replace=False))]
    R = np.ascontiguousarray(sites + rng.uniform(-0.2, 0.2, sites.shape))
    V = rng.normal(0.0, math.sqrt(inputs.KB_HARTREE_PER_K * 300.0 / inputs.SI_LIKE.mass), R.shape)
    V -= V.mean(0)
    field = rng.uniform(-0.01, 0.01, case["steps"]) if case.get("field") else None
    return dict(n=case["n"], h=case["h"], order=case["order"], sp=_species(case), R=R, V=V, field=field,
                psi=_orbitals(case["n"], case["h"], R, rng))


def _dimer(case, seed):
    """Two N-like atoms (10 electrons in 5 orbitals) near their bond length."""
    rng = np.random.default_rng([seed, case["n"]])
    L = case["n"] * case["h"]
    bond = 3.35 + rng.uniform(-0.1, 0.1)
    c = 0.5 * L + rng.uniform(-0.1, 0.1, 3)
    R = np.array([c - [0, 0, 0.5 * bond], c + [0, 0, 0.5 * bond]])
    return dict(n=case["n"], h=case["h"], order=case["order"], sp=inputs.N_LIKE, R=R, V=np.zeros_like(R), field=None,
                psi=_orbitals(case["n"], case["h"], R, rng, extra_px=True))


def _replica_cases(case):
    """Grids and atom counts of the replicas: 48^3 with 8 atoms, and 64^3
    with 9 to 27 atoms."""
    small = dict(n=48, h=0.25, order=case["order"], cells=2, steps=case["steps"])
    out = []
    for r in range(case["replicas"]):
        if r < case["big"]:
            out.append(dict(small, n=64, h=0.28125, cells=3, atoms=9 + (5 * r) % 19))
        else:
            out.append(dict(small))
    return out


_pinned = {}   # read-out buffers, one per shape (and replica)


class _System:
    """A libemd handle, released with the object."""

    def __init__(self, s, fp64):
        sp = s["sp"]
        self.n, self.n_atoms, self.n_orb = s["n"], len(s["R"]), s["psi"].shape[0]
        cfg = emd.emd_config(n=s["n"], h=s["h"], fd_order=s["order"], n_orb=self.n_orb, occ=2.0,
                             precision=emd.EMD_FP64 if fp64 else emd.EMD_FP32_ORBITALS, n_atoms=self.n_atoms,
                             species=emd.emd_species(sp.z, sp.mass, sp.a_loc, sp.r_loc, sp.r_c, sp.h_kb, sp.r_proj, sp.lmax,
                                                     (ctypes.c_double * 2)(*sp.h_l)),
                             cuda_stream=None, block_orbitals=0)
        self.handle = emd.emd_init_system(cfg)
        emd.emd_set_ions(self.handle, s["R"], s["V"])
        if s["psi"].dtype == torch.complex64:
            pin = torch.empty(s["psi"].shape, dtype=torch.complex64, pin_memory=True)
            pin.copy_(s["psi"])
            emd.emd_set_orbitals_c64(self.handle, pin.numpy())
        else:
            emd.emd_set_orbitals(self.handle, s["psi"].cpu().numpy())

    def __del__(self):
        if getattr(self, "handle", None):
            emd.emd_destroy(self.handle)

    def orbitals(self, slot=0):
        """The current orbitals in a page-locked buffer that the program keeps."""
        key = (slot, self.n_orb, self.n)
        if key not in _pinned:
            _pinned[key] = torch.empty((self.n_orb, self.n, self.n, self.n), dtype=torch.complex64, pin_memory=True)
        emd.emd_get_orbitals_c64(self.handle, self.n_orb, self.n, out=_pinned[key].numpy())
        return _pinned[key]

    def ions(self):
        return emd.emd_get_state(self.handle, self.n_atoms, self.n_orb, self.n, want_psi=False, want_rho=False)[:2]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        g = torch.Generator(device="cuda").manual_seed(seed)
        q = torch.randn(case["n"] ** 3, dtype=torch.float64, device="cuda", generator=g)
        return dict(case=case, q=q, v=torch.empty_like(q))
    if kind == "batch":
        sys = [_System(_lattice(c, seed * 100 + i), False) for i, c in enumerate(_replica_cases(case))]
        return dict(case=case, sys=sys, batch=_Batch(sys))
    s = _dimer(case, seed) if kind in ("sampled", "ground") else _lattice(dict(case, field=case.get("field") or kind == "adjoint"), seed)
    st = dict(case=case, sys=_System(s, case.get("fp64", True)), field=s["field"], R=s["R"], V=s["V"])
    if kind == "ground":
        st["psi"] = s["psi"].cpu().numpy()
    return st


class _Batch:
    def __init__(self, systems):
        self.systems = systems
        self.handle = emd.emd_batch_create([s.handle for s in systems])

    def __del__(self):
        if getattr(self, "handle", None):
            emd.emd_batch_destroy(self.handle)


# ---- one pass --------------------------------------------------------------

def _vector(e):
    """The energy components as float64, in the order of the C struct."""
    return np.array([float(e[k]) for k, _ in emd.emd_energy._fields_])


def _readout(s, fp64, slot=0):
    """The state after a run, velocities in the precision of the orbitals
    that drove them.  The FP64 form also returns what its FP64 results are
    read for: density, energies, forces."""
    R, V = s.ions()
    out = dict(R=R, V=V if fp64 else V.astype(np.float32), psi=s.orbitals(slot))
    if fp64:
        out["rho"] = emd.emd_get_state(s.handle, s.n_atoms, s.n_orb, s.n, want_psi=False, want_rho=True)[3]
        out["E"] = _vector(emd.emd_get_energy(s.handle))
        out["F"] = emd.emd_get_forces(s.handle, s.n_atoms)
    return out


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "poisson":
        emd.emd_poisson_static(case["n"], case["h"], st["q"].data_ptr(), st["v"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return st["v"]
    if kind == "batch":
        emd.emd_batch_propagate(st["batch"].handle, case["steps"], _dt(case["mu"]), case["mu"])
        return [_readout(s, False, i) for i, s in enumerate(st["sys"])]
    s = st["sys"]
    if kind == "ground":
        emd.emd_set_ions(s.handle, st["R"], st["V"])
        emd.emd_set_orbitals(s.handle, st["psi"])
        w, _ = emd.emd_ground_state(s.handle, s.n_orb, max_scf=400, tol=1e-10)
        rho = emd.emd_get_state(s.handle, s.n_atoms, s.n_orb, s.n, want_psi=False, want_rho=True)[3]
        return dict(eps=w, rho=rho, E=_vector(emd.emd_get_energy(s.handle)), F=emd.emd_get_forces(s.handle, s.n_atoms))
    if kind == "sampled":
        E, F = [], []
        for _ in range(case["samples"]):
            emd.emd_propagate(s.handle, case["every"], 0.04 * case["mu"], case["mu"])
            E.append(emd.emd_get_energy(s.handle)["total"])
            F.append(emd.emd_get_forces(s.handle, s.n_atoms))
        return dict(_readout(s, True), energies=np.array(E), forces=np.stack(F))
    if kind == "adjoint":
        L, dR, df = emd.emd_propagate_adjoint(s.handle, case["steps"], _dt(10.0), 10.0, st["field"], case["every"],
                                              emd.EMD_OBS_ENERGY, s.n_atoms)
        R, V = s.ions()
        return dict(L=np.float64(L), dR=dR, dfield=df, R=R, V=V, psi=s.orbitals())
    emd.emd_propagate(s.handle, case["steps"], _dt(case["mu"]), case["mu"], st["field"])
    return _readout(s, case["fp64"])


# ---- what one pass cannot do without ----------------------------------------

def _md_work(n, order, orbitals, atoms, h, steps, fp64, nch=1):
    """Per MD step: 8 applications of H (stencil, local term and the
    projector term at the points its spheres cover), the density and three
    FFTs' worth of grid work.  Memory: each step reads and writes the
    orbitals at least once; they come back once as complex64."""
    pts = float(n ** 3) * orbitals
    cover = atoms * nch * (4.0 / 3.0 * math.pi * (5.0 / h) ** 3) / n ** 3
    flops = steps * (8 * pts * (6 * order + 8 + 8 * cover) + 4 * pts)
    size = 16 if fp64 else 8
    return steps * 2 * pts * size + 8 * pts, flops


def work(case):
    kind = case["kind"]
    n3 = float(case.get("n", 0) ** 3)
    if kind == "poisson":
        return dict(bytes=16 * n3, flops=2 * 2.5 * n3 * math.log2(n3))
    if kind == "batch":
        parts = [_md_work(c["n"], c["order"], 2 * c.get("atoms", c["cells"] ** 3), c.get("atoms", c["cells"] ** 3), c["h"],
                          case["steps"], False) for c in _replica_cases(case)]
        return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))
    if kind == "ground":   # about 40 iterations of a degree-16 filter on 9 states
        b, f = _md_work(case["n"], case["order"], 9, 2, case["h"], 80, True)
        return dict(bytes=b, flops=f)
    if kind == "sampled":
        b, f = _md_work(case["n"], case["order"], 5, 2, case["h"], case["every"] * case["samples"], True)
        return dict(bytes=b + 8 * n3, flops=f)
    atoms = case["cells"] ** 3
    if kind == "adjoint":  # forward and reverse: three times the forward applications
        b, f = _md_work(case["n"], case["order"], 2 * atoms, atoms, case["h"], 3 * case["steps"], True)
        return dict(bytes=b, flops=f)
    b, f = _md_work(case["n"], case["order"], 2 * atoms, atoms, case["h"], case["steps"], case["fp64"], (case["lmax"] + 1) ** 2)
    return dict(bytes=b + (8 * n3 if case["fp64"] else 0), flops=f)


# ---- the same in 64 bits -----------------------------------------------------

FD = {2: (-2.0, 1.0), 4: (-5 / 2, 4 / 3, -1 / 12), 6: (-49 / 18, 3 / 2, -3 / 20, 1 / 90),
      8: (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560)}


def _poisson(q, h):
    n = q.shape[0]
    g = 2 * math.pi / (n * h) * torch.fft.fftfreq(n, d=1.0 / n, dtype=torch.float64, device=q.device)
    G2 = g[:, None, None] ** 2 + g[None, :, None] ** 2 + g[None, None, :] ** 2
    G2[0, 0, 0] = 1.0
    k = 4 * math.pi / G2
    k[0, 0, 0] = 0.0
    return torch.fft.ifftn(k * torch.fft.fftn(q)).real


def _lda(rho):
    """Perdew-Zunger exchange-correlation energy per electron and potential,
    the branches joined with continuous value and slope at r_s = 1."""
    gam, b1, b2, A, B = -0.1423, 1.0529, 0.3334, 0.0311, -0.048
    q1 = 1 + b1 + b2
    D = gam / q1 - B
    C = -gam * (0.5 * b1 + b2) / q1 ** 2 - A - D
    r = rho.clamp_min(1e-30)
    ex = -0.75 * (3 * r / math.pi) ** (1 / 3)
    rs = (3 / (4 * math.pi * r)) ** (1 / 3)
    s = rs.sqrt()
    q = 1 + b1 * s + b2 * rs
    lx = rs.log()
    hi = rs >= 1
    ec = torch.where(hi, gam / q, A * lx + B + C * rs * lx + D * rs)
    vc = torch.where(hi, gam * (1 + 7 / 6 * b1 * s + 4 / 3 * b2 * rs) / (q * q),
                     A * lx + (B - A / 3) + 2 / 3 * C * rs * lx + (2 * D - C) / 3 * rs)
    some = rho >= 1e-30
    return torch.where(some, ex + ec, 0.0), torch.where(some, 4 / 3 * ex + vc, 0.0)


class _Exact:
    """The MD step in torch, float64 and complex128; differentiable in R,
    the orbitals and the field when they require a gradient."""

    def __init__(self, s, seed=None):
        self.n, self.h, self.order, self.sp = s["n"], s["h"], s["order"], s["sp"]
        self.L, self.h3 = s["n"] * s["h"], s["h"] ** 3
        self.psi = s["psi"].to(torch.complex64 if s["psi"].dtype == torch.complex64 else torch.complex128).to(torch.complex128)
        self.R, self.V = (torch.from_numpy(s[k]).cuda() for k in "RV")
        z = torch.arange(self.n, dtype=torch.float64, device="cuda") * self.h - 0.5 * self.L
        self.saw = z[:, None, None].expand(self.n, self.n, self.n)

    # supports: every (point, image) pair within r of each atom
    def spheres(self, R, r):
        n, h, L = self.n, self.h, self.L
        ar = torch.arange(n, device="cuda")
        co = ar.double() * h
        Rw = (R - L * torch.floor(R / L)).detach()
        out = []
        for j in range(len(Rw)):
            ax = []
            for a in range(3):
                d = torch.stack([(co - Rw[j, a]) - m * L for m in (-1.0, 0.0, 1.0)])
                keep = d.abs() < r
                ax.append((ar.expand(3, n)[keep], d[keep]))
            (ix, dx), (iy, dy), (iz, dz) = ax
            dx2, dy2, dz2 = (dx * dx)[None, None, :], (dy * dy)[None, :, None], (dz * dz)[:, None, None]
            m = ((dx2 + dy2) + dz2) < r * r
            idx = ((iz[:, None, None] * n + iy[None, :, None]) * n + ix[None, None, :])[m]
            sh = m.shape
            d = torch.stack([dx[None, None, :].expand(sh)[m], dy[None, :, None].expand(sh)[m], dz[:, None, None].expand(sh)[m]])
            if R.requires_grad:
                d = d - (R[j] - R[j].detach())[:, None]
            out.append((idx, d))
        return out

    def tables(self, R):
        sp = self.sp
        t = dict(R=R, proj=[], loc=self.spheres(R, sp.r_loc))
        for idx, d in self.spheres(R, sp.r_proj):
            x, y, z = d
            e = torch.exp(-(d * d).sum(0) / (2 * sp.r_c ** 2))
            o, zero, s3 = torch.ones_like(x), torch.zeros_like(x), math.sqrt(3.0)
            S = [(0, o, (zero, zero, zero))]
            if sp.lmax >= 1:
                S += [(1, x, (o, zero, zero)), (1, y, (zero, o, zero)), (1, z, (zero, zero, o))]
            if sp.lmax >= 2:
                S += [(2, s3 * x * y, (s3 * y, s3 * x, zero)), (2, s3 * y * z, (zero, s3 * z, s3 * y)),
                      (2, s3 * z * x, (s3 * z, zero, s3 * x)), (2, 0.5 * s3 * (x * x - y * y), (s3 * x, -s3 * y, zero)),
                      (2, 0.5 * (2 * z * z - x * x - y * y), (-x, -y, 2 * z))]
            P, G, H = [], [], []
            for l, f, g in S:
                N = (2 * math.pi / (2 * l + 1) * math.gamma(l + 1.5) * sp.r_c ** (2 * l + 3)) ** -0.5
                P.append(N * f * e)
                G.append(torch.stack([N * e * (f * d[a] / sp.r_c ** 2 - g[a]) for a in range(3)]))   # d p / d R
                H.append(sp.h_kb if l == 0 else sp.h_l[l - 1])
            t["proj"].append((idx, torch.stack(P), torch.stack(G), torch.tensor(H, dtype=torch.float64, device="cuda")))
        g = torch.zeros(self.n ** 3, dtype=torch.float64, device="cuda")
        t["g"] = [sp.z * math.pi ** -1.5 * sp.a_loc ** -3 * torch.exp(-(d * d).sum(0) / sp.a_loc ** 2) for _, d in t["loc"]]
        for (idx, _), v in zip(t["loc"], t["g"]):
            g = g.index_add(0, idx, v)
        t["gion"] = g.reshape(self.n, self.n, self.n)
        t["vloc"] = _poisson(-t["gion"], self.h)
        return t

    def kinetic(self, u):
        c = FD[self.order]
        out = (-1.5 * c[0] / self.h ** 2) * u
        for a in (1, 2, 3):
            for k in range(1, len(c)):
                out = out + (-0.5 * c[k] / self.h ** 2) * (torch.roll(u, k, a) + torch.roll(u, -k, a))
        return out

    def H(self, u, v, t):
        out = (self.kinetic(u) + v * u).reshape(len(u), -1)
        flat = u.reshape(len(u), -1)
        for idx, P, _, hP in t["proj"]:
            c = self.h3 * (flat[:, idx] @ P.T.to(u.dtype))
            out = out.index_add(1, idx, (c * hP) @ P.to(u.dtype))
        return out.reshape(u.shape)

    def half(self, psi, tau, v, t):
        def block(p):
            out, term = p, p
            for k in range(1, 5):
                term = (-1j * tau / k) * self.H(term, v, t)
                out = out + term
            return out
        if psi.requires_grad or v.requires_grad:
            return block(psi)
        return torch.cat([block(p) for p in psi.split(max(1, (1 << 25) // self.n ** 3))])

    def density(self, psi):
        return 2.0 * (psi.real ** 2 + psi.imag ** 2).sum(0)

    def electrons(self, psi):
        rho = self.density(psi)
        vh = _poisson(rho, self.h)
        eps, vxc = _lda(rho)
        return rho, vh, eps, vh + vxc

    def short_range(self, R):
        sp, L = self.sp, self.L
        m = int(math.ceil(12.0 / L)) + 1
        a = torch.arange(-m, m + 1, dtype=torch.float64, device="cuda") * L
        img = torch.stack(torch.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3)
        Rw = R - (L * torch.floor(R / L)).detach()
        s = math.sqrt(2.0) * sp.a_loc
        E, F = 0.0, []
        for j in range(len(R)):
            dv = (Rw[j] - Rw[:, None, :] - img[None]).reshape(-1, 3)
            d2 = (dv * dv).sum(1)
            keep = (d2 < 144.0) & (d2 > 0)
            dv, d = dv[keep], d2[keep].sqrt()
            e = torch.erfc(d / s) / d
            E = E + 0.5 * sp.z ** 2 * e.sum()
            F.append((sp.z ** 2 * ((e + 2 / (s * math.sqrt(math.pi)) * torch.exp(-d * d / s ** 2)) / (d * d))[:, None] * dv).sum(0))
        return E, torch.stack(F)

    def forces(self, psi, vh, t):
        ves = (vh + t["vloc"]).reshape(-1)
        flat = psi.reshape(len(psi), -1)
        F = []
        for (idx, d), g, (pi, P, G, hP) in zip(t["loc"], t["g"], t["proj"]):
            f = self.h3 * 2 / self.sp.a_loc ** 2 * (d * (ves[idx] * g)).sum(1)
            u = flat[:, pi]
            c = self.h3 * (u @ P.T.to(u.dtype))                              # [orb, ch]
            dc = self.h3 * torch.einsum("ok,cak->oca", u, G.to(u.dtype))
            f = f - 4.0 * ((c.conj()[:, :, None] * dc).real * hP[None, :, None]).sum((0, 1))
            F.append(f)
        return torch.stack(F) + self.short_range(t["R"])[1]

    def energies(self, psi, V, rho, vh, eps, t):
        sp = self.sp
        kin = 2.0 * self.h3 * sum((p.conj() * self.kinetic(p)).real.sum() for p in psi.split(max(1, (1 << 25) // self.n ** 3)))
        nl = 0.0
        flat = psi.reshape(len(psi), -1)
        for idx, P, _, hP in t["proj"]:
            c = self.h3 * (flat[:, idx] @ P.T.to(psi.dtype))
            nl = nl + 2.0 * ((c.real ** 2 + c.imag ** 2) * hP).sum()
        sr = self.short_range(t["R"])[0]
        es = 0.5 * self.h3 * ((rho - t["gion"]) * (vh + t["vloc"])).sum() - len(V) * sp.z ** 2 / (math.sqrt(2 * math.pi) * sp.a_loc) + sr
        xc = self.h3 * (rho * eps).sum()
        ki = 0.5 * sp.mass * (V * V).sum()
        ks = kin + nl + es + xc
        return dict(kin_e=kin, nl=nl, es=es, xc=xc, sr=sr, kin_ion=ki, ks=ks, total=ks + ki, n_elec=self.h3 * rho.sum())

    def start(self):
        self.t = self.tables(self.R)
        self.rho, self.vh, self.eps, v = self.electrons(self.psi)
        self.hist = [v]
        self.F = self.forces(self.psi, self.vh, self.t)
        return self

    def step(self, dt, mu, e=None):
        tau, M = 0.5 * (dt / mu), self.sp.mass
        ext = 0.0 if e is None else e * self.saw
        R = self.R + self.V * dt + self.F * (dt * dt / (2 * M))
        t = self.tables(R)
        x = self.hist
        v2 = x[0] if len(x) == 1 else 2 * x[0] - x[1] if len(x) == 2 else 3 * x[0] - 3 * x[1] + x[2]
        psi = self.half(self.psi, tau, self.t["vloc"] + x[0] + ext, self.t)
        self.psi = self.half(psi, tau, t["vloc"] + v2 + ext, t)
        self.rho, self.vh, self.eps, v = self.electrons(self.psi)
        self.hist = [v] + x[:2]
        F = self.forces(self.psi, self.vh, t)
        if e is not None:
            F = F + self.sp.z * e * torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda")
        self.V = self.V + (self.F + F) * (dt / (2 * M))
        self.R, self.t, self.F = R, t, F

    def readout(self, fp64):
        out = dict(R=self.R, V=self.V, psi=self.psi)
        if fp64:
            out.update(rho=self.rho, F=self.F, E=_vector(self.energy()))
        return out

    def energy(self):
        return self.energies(self.psi, self.V, self.rho, self.vh, self.eps, self.t)


def exact(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        st = prepare(case, seed)
        n = case["n"]
        return _poisson(st["q"].reshape(n, n, n), case["h"]).reshape(-1)
    if kind == "ground":
        return None      # the fixed point of an iteration of its own
    if kind == "batch":
        out = []
        for i, c in enumerate(_replica_cases(case)):
            x = _Exact(_lattice(c, seed * 100 + i)).start()
            for _ in range(case["steps"]):
                x.step(_dt(case["mu"]), case["mu"])
            out.append(x.readout(False))
        return out
    if kind == "sampled":
        x = _Exact(_dimer(case, seed)).start()
        E, F = [], []
        for _ in range(case["samples"]):
            for _ in range(case["every"]):
                x.step(0.04 * case["mu"], case["mu"])
            E.append(float(x.energy()["total"]))
            F.append(x.F)
        return dict(x.readout(True), energies=np.array(E), forces=torch.stack(F))
    s = _lattice(dict(case, field=case.get("field") or kind == "adjoint"), seed)
    x = _Exact(s)
    if kind == "adjoint":
        x.R.requires_grad_(True)
        e = torch.from_numpy(s["field"]).cuda().requires_grad_(True)
        R0 = x.R
        x.start()
        for k in range(case["steps"]):
            x.step(_dt(10.0), 10.0, e[k])
        en = x.energy()
        L = en["ks"] + en["kin_ion"]
        dR, df = torch.autograd.grad(L, (R0, e))
        return dict(L=np.float64(float(L)), dR=dR, dfield=df, R=x.R.detach(), V=x.V.detach(), psi=x.psi.detach())
    x.start()
    for k in range(case["steps"]):
        x.step(_dt(case["mu"]), case["mu"], None if s["field"] is None else float(s["field"][k]))
    return x.readout(case["fp64"])
