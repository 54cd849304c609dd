"""Timed cases of the coupled Maxwell-Schroedinger step, through the ctypes binding of include/ms.h.

A case is one pass of a user's loop: a handle that already exists takes `steps`
steps and the loop reads back what it looks at (populations, dipoles, norm,
Eq. 8 sums; fields or flux spectra where those are what the run is for).  The
grids, geometries and species are those of workloads/configs.py, with fewer
molecules where three handles would not fit the card together; the smallest and
the ragged ones are those of the tests.

The handle starts from a seeded smooth field of 1e9 V/m order in the whole box
under a continuous-wave source, so that every molecule is driven from the first
step on and the work per step (terms of the coupling series) is that of a pulse
in flight and stays so from pass to pass.  `preroll` steps run in prepare(), as
a run that is under way has them behind it.

Populations, dipoles, norms and Eq. 8 sums are computed from an FP32 state by
FP32 arithmetic and handed out in FP64; they are returned as FP32, and each
quantity by itself (P_e beside P_g, not under it).  The absorbed norm of a species
whose packet has not reached the absorber is the rounding noise of its tail, so
it is returned inside the norm bookkeeping P_g + P_e + absorbed, and by itself
only where the absorber cuts into the packet.
"""
import math
import types

import numpy as np
import torch

from paper_2209_04487_gb300 import binding as B

# CODATA 2018
C0, MU0, EPS0 = 299792458.0, 1.25663706212e-6, 8.8541878128e-12
HBAR_EVS, T_AU, F_AU = 6.582119569e-16, 2.4188843265857e-17, 5.14220674763e11
EA0, HARTREE_EV = 8.4783536255e-30, 27.211386245988
DX = 2e-9
DT = DX / (2.0 * C0)
PML = 10
SRC_K = 18
VACUUM, GLASS, SILVER = 0, 1, 2
MATERIALS = [(1.0, 0.0, 0.0), (2.25, 0.0, 0.0), (3.7, 9.0, 0.02)]


def _case(name, grid, mols, species, steps, *, nsim=1, geometry="vacuum", preroll=8, model="wavepacket",
          state="full", precision="fp32", substeps=1, drive="fdtd", d_of_r=False, absorber=8.5, planes=0,
          nfreq=0, fields=False):
    c = dict(nx=grid[0], ny=grid[1], nz=grid[2], nsim=nsim, geometry=geometry, mols=mols, species=species,
             steps=steps, preroll=preroll, model=model, state=state, precision=precision, substeps=substeps,
             drive=drive, d_of_r=d_of_r, absorber=absorber, planes=planes, nfreq=nfreq, fields=fields)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a loop of the user's own around single steps of the small vacuum workload
        # (1,000 molecules, N_r 64, J <= 1), reading dipoles and populations after each
        _case("single_step", (32, 32, 64), 1000, "64/1", 1, preroll=64),
        # the same workload run by the library for a while, fields read back at the end (snapshots)
        _case("small_run", (32, 32, 64), 1000, "64/1", 128, preroll=64, fields=True),
        # the split-ring array with its 50,000 molecules (N_r 128, J <= 4), the ordinary run
        _case("split_ring", (128, 128, 192), 50000, "128/4", 8, geometry="ring"),
        # the nanohole array at J <= 8 (N_r 128), the largest: its 256^3 grid with 100,000 of its 700,000
        # molecules (33 GB of state and scratch)
        _case("nanohole", (256, 256, 256), 100000, "128/8", 8, geometry="hole", preroll=2),
        # the same species with the reduced state form, on a smaller grid
        _case("nanohole_parity", (160, 160, 160), 60000, "128/8", 8, geometry="hole", state="parity"),
        # three species with uneven radial grids and rotational cutoffs in one step, 0.5/0.3/0.2
        _case("three_species", (192, 192, 192), 50000, "64/4 128/8 256/16", 3, geometry="ring"),
        # a carrier-frequency sweep: sixteen independent cells, 2,000 molecules each, in one handle
        _case("sweep", (64, 64, 128), 2000, "64/8", 16, nsim=16, geometry="hole"),
        # the mixed-precision kinetic pass (split FP16 on tensor cores)
        _case("mixed", (96, 96, 128), 20000, "128/4", 8, geometry="ring", precision="mixed"),
        # the multiscale cadence: molecules every 40th field step
        _case("cadence40", (128, 128, 192), 50000, "128/4", 80, geometry="ring", substeps=40, preroll=40),
        # frozen two-level molecules, a field-bound run on a grid larger than L2
        _case("frozen", (256, 256, 128), 200000, "1/0", 120, geometry="ring", model="bloch"),
        # no molecules: transmission and reflection spectra of the bare structure
        _case("spectra", (128, 128, 192), 0, "64/1", 240, geometry="ring", planes=2, nfreq=48, fields=True),
        # molecules alone under a prescribed field, transition dipole d(R), absorber inside the packet
        _case("prescribed_dr", (16, 16, 64), 20000, "128/3", 8, drive="prescribed", d_of_r=True, absorber=2.5),
    ]


# state elements (rows x radial points) over all molecules that a drawn case holds at most
MAX_ELEMENTS = 1.5e9


def draw(rng):
    def span(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def mols(species, most):
        per = sum((f * 2 * (j + 1) ** 2 * nr) for f, (nr, j) in zip(_fractions(len(species)), species))
        return max(1, min(span(64, most), int(MAX_ELEMENTS / per)))

    kind = rng.choice(["run", "run", "wide", "wide", "wider", "mixture", "parity", "mixed", "cadence", "frozen",
                       "spectra", "prescribed"])
    grid = (span(36, 200), span(36, 200), span(80, 220))
    geometry = rng.choice(["vacuum", "ring", "hole"])
    steps = rng.randint(4, 12)
    if kind in ("run", "wide", "wider", "parity", "mixed", "mixture"):
        n = 1
        while kind == "mixture" and n < 2:
            n = rng.randint(2, 3)
        top = {"run": (1, 4), "wide": (5, 8), "wider": (9, 16), "parity": (1, 12), "mixed": (1, 8), "mixture": (1, 10)}[kind]
        rs = [64, 128] if kind == "mixed" else [64, 128, 256]
        sp = [(rng.choice(rs), rng.randint(*top)) for _ in range(n)]
        nsim = 1 if rng.random() < 0.7 else rng.randint(2, 5)
        if nsim > 1:
            grid = (span(36, 80), span(36, 80), span(80, 128))
        return _case(None, grid, max(1, mols(sp, 100000) // nsim), " ".join("%d/%d" % s for s in sp), steps, nsim=nsim,
                     geometry=geometry, state="parity" if kind == "parity" else "full",
                     precision="mixed" if kind == "mixed" else "fp32")
    if kind == "cadence":
        sub = rng.choice([2, 5, 10, 20, 40])
        sp = [(rng.choice([64, 128]), rng.randint(1, 8))]
        return _case(None, grid, mols(sp, 30000), "%d/%d" % sp[0], 2 * sub, geometry=geometry, substeps=sub, preroll=sub)
    if kind == "frozen":
        return _case(None, grid, span(64, 300000), "1/0", rng.randint(16, 120), geometry=geometry, model="bloch",
                     substeps=rng.choice([1, 1, 4]))
    if kind == "spectra":
        return _case(None, grid, 0, "64/1", rng.randint(40, 240), geometry=geometry, planes=rng.randint(1, 4),
                     nfreq=span(1, 32), fields=rng.random() < 0.5)
    sp = [(rng.choice([64, 128]), rng.randint(1, 4))]
    dr = rng.random() < 0.5
    return _case(None, (16, 16, 64), mols(sp, 40000), "%d/%d" % sp[0], steps, drive="prescribed", d_of_r=dr,
                 absorber=rng.choice([8.5, 2.5]))


def _fractions(n):
    return {1: [1.0], 2: [0.6, 0.4], 3: [0.5, 0.3, 0.2]}[n]


# ---- inputs: what a user's program has in hand -----------------------------------------------------------------

def _species(case):
    out = []
    for i, s in enumerate(case["species"].split()):
        nr, jmax = (int(v) for v in s.split("/"))
        sp = types.SimpleNamespace(nr=nr, jmax=jmax, rmin=1.0, rmax=10.0, mass=918.0, De=0.1, a=1.0, re=2.0, A=0.15,
                                   B=0.1, beta=1.5, rc=2.0, dipole=1.0, absorber_r=case["absorber"],
                                   absorber_power=0.125, dipole_R=None, model=case["model"], w0_ev=0.0, T1=0.0, T2=0.0)
        if len(case["species"].split()) > 1:  # the three-species workload's masses and well depths
            sp.mass, sp.De = ((918.0, 0.05), (8000.0, 0.1), (14000.0, 0.2))[i]
        if case["model"] == "bloch":
            sp.w0_ev, sp.T1, sp.T2 = 1.6, 200e-15, 50e-15
        if case["d_of_r"]:
            r = np.linspace(sp.rmin, sp.rmax, nr)
            sp.dipole_R = tuple(1.2 * np.exp(-0.3 * (r - 2.0) ** 2) + 0.1)
        out.append(sp)
    return out


def _layers(case):
    """(molecular layer, structure planes, glass from): the structure stands right behind the layer."""
    k0 = SRC_K + 10
    k1 = k0 + max(4, min(10, case["nz"] // 12))
    thick = {"ring": 15, "hole": 50}.get(case["geometry"], 0)
    k2 = min(k1 + thick, case["nz"] - PML - 12)
    return (k0, k1), (k1, k2), k2


def _material(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    m = np.zeros((nz, ny, nx), np.uint8)
    if case["geometry"] == "vacuum":
        return np.repeat(m[None], case["nsim"], 0)
    _, (k1, k2), kg = _layers(case)
    x, y = (np.arange(nx) + 0.5 - nx / 2)[None, :], (np.arange(ny) + 0.5 - ny / 2)[:, None]
    if case["geometry"] == "ring":  # outer side 30 cells, arms 10, a 5-cell gap in the -y arm
        cells = (np.abs(x) < 15) & (np.abs(y) < 15) & ~((np.abs(x) < 5) & (np.abs(y) < 5))
        cells &= ~((x >= -2.5) & (x < 2.5) & (y < -5))
    else:  # a film with an equilateral triangular hole of 0.45 of the cell
        side = 0.45 * min(nx, ny)
        y0 = -side * math.sqrt(3.0) / 6.0
        cells = ~((y >= y0) & (y <= y0 + math.sqrt(3.0) * (x + side / 2)) & (y <= y0 + math.sqrt(3.0) * (side / 2 - x)))
    m[kg:] = GLASS
    m[k1:k2][:, cells] = SILVER
    return np.repeat(m[None], case["nsim"], 0)


def _workload(case, seed):
    rng = np.random.default_rng(seed)
    nsim, per = case["nsim"], case["mols"]
    n = nsim * per
    (k0, k1), _, _ = _layers(case)
    pos = rng.random((n, 3)) * np.array([case["nx"], case["ny"], k1 - k0], np.float64)
    pos[:, 2] += k0
    quat = rng.standard_normal((n, 4))
    sp = _species(case)
    sid = rng.choice(len(sp), size=n, p=_fractions(len(sp))).astype(np.int32)
    # one carrier per cell over 1.2-2.4 eV (a single cell: 800 nm), E0, a 1 fs turn-on, a seeded phase
    ev = [1.5498] if nsim == 1 else [1.2 + 1.2 * s / (nsim - 1) for s in range(nsim)]
    src = np.array([[1e9, e, 1e-15, float(rng.uniform(0, 2e-15))] for e in ev])
    return types.SimpleNamespace(
        name="perf", nx=case["nx"], ny=case["ny"], nz=case["nz"], nsim=nsim, dx=DX, dt=DT, pml=PML, bc_z="pml",
        src_k=SRC_K, src=src, src_kind="cw", materials=list(MATERIALS), mat_id=_material(case), species=sp,
        species_id=sid, sim_id=np.repeat(np.arange(nsim, dtype=np.int32), per), pos=pos * DX, quat=quat,
        mol_substeps=case["substeps"], n_molecules=n)


def _field0(case, seed):
    """[nsim] of [3][nz][ny][nx] FP32: a smooth seeded field of 1e9 V/m order, zero in the absorbers."""
    rng = np.random.default_rng(seed + 1)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x = torch.arange(case["nx"], dtype=torch.float64, device=dev) * (2 * math.pi / case["nx"])
    y = torch.arange(case["ny"], dtype=torch.float64, device=dev) * (2 * math.pi / case["ny"])
    z = torch.arange(case["nz"], dtype=torch.float64, device=dev)
    w = torch.clamp((z - PML) * (case["nz"] - 1 - PML - z), min=0.0)
    w = (w / w.max()).sqrt()
    out = []
    for _ in range(case["nsim"]):
        E = torch.zeros((3, case["nz"], case["ny"], case["nx"]), dtype=torch.float32, device=dev)
        for c in range(3):
            for mode in (1, 2):
                a, p, q, r = rng.uniform(0.5, 1.5), *rng.uniform(0, 2 * math.pi, 3)
                zz = w * torch.cos(2 * math.pi * mode * z / case["nz"] + r)
                E[c] += (2e9 * a * zz[:, None, None] * torch.cos(mode * y + q)[None, :, None]
                         * torch.cos(mode * x + p)[None, None, :]).float()
        out.append(E.cpu().numpy())
    return out


# a prescribed run's samples: enough for any number of passes over one handle
WAVE = 1 << 20


def _drive(case, seed):
    rng = np.random.default_rng(seed + 2)
    n = case["nsim"] * case["mols"]
    d = rng.standard_normal((n, 3))
    amp = d / np.linalg.norm(d, axis=1, keepdims=True) * (1e9 * (0.5 + rng.random((n, 1))))
    wave = np.cos(2 * math.pi * np.arange(WAVE) / 800.0 + rng.uniform(0, 0.5))
    return amp.astype(np.float32), wave.astype(np.float32)


def _omega(case):
    return np.linspace(1.2, 2.4, case["nfreq"]) / HBAR_EVS if case["nfreq"] else np.zeros(0)


def _planes(case):
    return [[14, case["nz"] - 16, SRC_K + 4, case["nz"] // 2][p] for p in range(case["planes"])]


def prepare(case, seed):
    wl = _workload(case, seed)
    sim = B.Simulation(wl, drive=B.MS_DRIVE_PRESCRIBED if case["drive"] == "prescribed" else B.MS_DRIVE_FDTD,
                       precision=B.MS_PREC_MIXED_F16X3 if case["precision"] == "mixed" else B.MS_PREC_FP32,
                       state_form=B.MS_STATE_PARITY if case["state"] == "parity" else B.MS_STATE_FULL)
    if case["drive"] == "prescribed":
        sim.set_prescribed(*_drive(case, seed))
    else:
        for s, E in enumerate(_field0(case, seed)):
            sim.write_fields(B.MS_FIELD_E, s, E)
    if case["planes"]:
        sim.set_detectors(_planes(case), _omega(case))
    sim.step(case["preroll"])
    return {"sim": sim, "case": case}


def run(state):
    sim, case = state["sim"], state["case"]
    sim.step(case["steps"])
    out = {}
    if case["mols"]:
        P = sim.populations()
        absorbed, Re = sim.dissociation() if case["steps"] > 1 else (None, None)
        out["P_g"], out["P_e"] = P[:, 0].astype(np.float32), P[:, 1].astype(np.float32)
        out["mu"] = sim.dipoles().astype(np.float32)
        if absorbed is not None:  # a loop over single steps does not look at these
            out["norm"] = (P[:, 0] + P[:, 1] + (absorbed[:, 0] + absorbed[:, 1])).astype(np.float32)
            out["R_e"] = Re.astype(np.float32)
            if case["absorber"] < 8.0:
                out["absorbed"] = absorbed.astype(np.float32)
    if case["fields"]:
        out["E"] = [sim.fields(B.MS_FIELD_E, s) for s in range(case["nsim"])]
        out["H"] = [sim.fields(B.MS_FIELD_H, s) for s in range(case["nsim"])]
    for p in range(case["planes"]):
        out["flux%d" % p] = sim.flux(p).astype(np.float32)
    return out


def work(case):
    """Of one pass.  A wavepacket molecule's state is read and written once per molecular step: the (J + 1)^2 rows
    that its j = 0 start can populate (each coupling changes j by one and swaps the surfaces; the other rows of the
    full state are zeros).  A field step reads and writes E and H and reads the material; metal cells read and
    write their current; a detector adds into one accumulator per (cell, frequency, component) and call, and its
    arithmetic counts per step.  Arithmetic of a molecule: the two transforms of the kinetic pass, the phases and
    two terms of the coupling series, the update and the dipole."""
    cells = case["nx"] * case["ny"] * case["nz"] * case["nsim"] if case["drive"] == "fdtd" else 0
    b = f = 0.0
    if cells:
        metal = float((_material(dict(case, nsim=1)) == SILVER).sum()) * case["nsim"]
        b += case["steps"] * (49.0 * cells + 24.0 * metal)
        f += case["steps"] * (36.0 * cells + 12.0 * metal)
    if case["planes"]:
        acc = case["planes"] * case["nfreq"] * 4 * case["nx"] * case["ny"] * case["nsim"]
        b += 32.0 * acc
        f += case["steps"] * 4.0 * acc
    n = case["nsim"] * case["mols"]
    msteps = case["steps"] / case["substeps"]
    for fr, s in zip(_fractions(len(case["species"].split())), case["species"].split()):
        nr, j = (int(v) for v in s.split("/"))
        if case["model"] == "bloch":
            b += msteps * n * fr * 180.0
            f += msteps * n * fr * 150.0
        else:
            el = n * fr * (j + 1) ** 2 * nr
            b += msteps * (16.0 * el + 168.0 * n * fr)
            f += msteps * el * (10.0 * math.log2(nr) + 110.0)
    b += n * 72.0 + (24.0 * cells if case["fields"] else 0.0)
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits, in plain torch ------------------------------------------------------------------------

# work of an exact pass (molecular element steps) beyond which none is given
EXACT_ELEMENT_STEPS = 1.4e10


class _Fields:
    """Yee grid in FP64: Drude current, CPML in z, TF/SF source with its 1D line, conductors at both ends."""

    def __init__(self, case, wl, seed, dev):
        self.dt, self.n, self.src = DT, 0, wl.src
        shape = (wl.nsim, wl.nz, wl.ny, wl.nx)
        f8 = dict(dtype=torch.float64, device=dev)
        self.E = [torch.zeros(shape, **f8) for _ in range(3)]
        self.H = [torch.zeros(shape, **f8) for _ in range(3)]
        self.J = [torch.zeros(shape, **f8) for _ in range(3)]
        for s, e in enumerate(_field0(case, seed)):
            for c in range(3):
                self.E[c][s] = torch.from_numpy(e[c]).to(dev).double()
        mat = torch.from_numpy(wl.mat_id).to(dev).long()
        self.inv_eps = (1.0 / (EPS0 * torch.tensor([m[0] for m in MATERIALS], **f8)))[mat]
        self.metal = mat == SILVER
        _, wp, ga = MATERIALS[SILVER]
        wp, ga = wp / HBAR_EVS, ga / HBAR_EVS
        self.al = (1 - 0.5 * ga * DT) / (1 + 0.5 * ga * DT)
        self.be = EPS0 * wp * wp * DT / (1 + 0.5 * ga * DT)
        z = np.arange(wl.nz) * DX
        self.cE, self.cH = (self._cpml(zz, wl.nz, f8) for zz in (z, z + 0.5 * DX))
        self.psi = [torch.zeros(shape, **f8) for _ in range(4)]
        L = case["preroll"] + case["steps"] + 16
        self.aE, self.aH = torch.zeros((wl.nsim, L + 1), **f8), torch.zeros((wl.nsim, L), **f8)
        self.aE[:, 0] = self._source(0)

    def _cpml(self, z, nz, f8):
        L, smax = PML * DX, 0.8 * 4 / (math.sqrt(MU0 / EPS0) * DX)
        rho = np.maximum(L - z, 0) + np.maximum(z - (nz * DX - L), 0)
        sg, al = smax * (rho / L) ** 3, 0.05 * (1 - rho / L)
        b = np.where(rho > 0, np.exp(-(sg + al) * DT / EPS0), 1.0)
        a = np.where(rho > 0, sg / np.where(rho > 0, sg + al, 1.0) * (b - 1.0), 0.0)
        return [torch.from_numpy(v).to(f8["device"])[None, :, None, None] for v in (b, a)]

    def _source(self, n):
        t = n * DT
        out = []
        for E0, ev, t_on, t0 in self.src:
            ramp = math.sin(0.5 * math.pi * max(t, 0.0) / t_on) ** 2 if t < t_on else 1.0
            out.append(E0 * ramp * math.cos(ev / HBAR_EVS * (t - t0)))
        return torch.tensor(out, dtype=torch.float64, device=self.aE.device)

    def step_h(self):
        Ex, Ey, Ez = self.E

        def up(F):
            return torch.cat([F[:, 1:], torch.zeros_like(F[:, :1])], 1)

        dyz, dxz = (up(Ey) - Ey) / DX, (up(Ex) - Ex) / DX
        b, a = self.cH
        self.psi[0], self.psi[1] = b * self.psi[0] + a * dyz, b * self.psi[1] + a * dxz
        dyz, dxz = dyz + self.psi[0], dxz + self.psi[1]
        k = DT / MU0
        self.H[0] -= k * ((Ez.roll(-1, 2) - Ez) / DX - dyz)
        self.H[1] -= k * (dxz - (Ez.roll(-1, 3) - Ez) / DX)
        self.H[2] -= k * ((Ey.roll(-1, 3) - Ey) / DX - (Ex.roll(-1, 2) - Ex) / DX)
        self.H[1][:, SRC_K - 1] += (k / DX) * self.aE[:, 2][:, None, None]
        self.aH -= (k / DX) * (self.aE[:, 1:] - self.aE[:, :-1])

    def step_e(self, dP=None):
        Hx, Hy, Hz = self.H

        def down(F):
            return torch.cat([torch.zeros_like(F[:, :1]), F[:, :-1]], 1)

        dyz, dxz = (Hy - down(Hy)) / DX, (Hx - down(Hx)) / DX
        b, a = self.cE
        self.psi[2], self.psi[3] = b * self.psi[2] + a * dyz, b * self.psi[3] + a * dxz
        cx = (Hz - Hz.roll(1, 2)) / DX - dyz - self.psi[2]
        cy = dxz + self.psi[3] - (Hz - Hz.roll(1, 3)) / DX
        cz = (Hy - Hy.roll(1, 3)) / DX - (Hx - Hx.roll(1, 2)) / DX
        cx[:, SRC_K] += self.aH[:, 1][:, None, None] / DX
        for c, curl in enumerate((cx, cy, cz)):
            self.J[c] = torch.where(self.metal, self.al * self.J[c] + self.be * self.E[c], torch.zeros_like(curl))
            self.E[c] += self.inv_eps * DT * (curl - self.J[c])
            if dP is not None:
                self.E[c] -= self.inv_eps * dP[c]
        for c in (0, 1):
            self.E[c][:, 0] = 0.0
        self.aE[:, 1:-1] -= (DT / (EPS0 * DX)) * (self.aH[:, 1:] - self.aH[:, :-1])
        self.aE[:, 0] = self._source(self.n + 1)
        self.n += 1


class _Wavepackets:
    """FP64 split-operator step of one species over the rows its start can populate, (ground, even j) and
    (excited, odd j); every operator as the equations have it, the coupling by its Taylor series."""

    def __init__(self, sp, O, dtau, dev):
        self.sp, self.O, self.dtau = sp, O, dtau
        r = np.linspace(sp.rmin, sp.rmax, sp.nr)
        self.dR = r[1] - r[0]
        k = 2 * math.pi * np.fft.fftfreq(sp.nr, self.dR)
        rows = [[(j, m) for j in range(sp.jmax + 1) for m in range(-j, j + 1) if j % 2 == s] for s in (0, 1)]
        U = [sp.De * (1 - np.exp(-sp.a * (r - sp.re))) ** 2 - sp.De, sp.A + sp.B * np.exp(-sp.beta * (r - sp.rc))]
        t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)  # noqa: E731
        self.vh = [t(np.exp(-0.5j * dtau * np.array([U[s] + j * (j + 1) / (2 * sp.mass * r * r) for j, _ in rows[s]]
                                                   or np.zeros((0, sp.nr))))) for s in (0, 1)]
        self.th = t(np.exp(-0.5j * dtau * k * k / (2 * sp.mass)))
        m = np.ones(sp.nr)
        sel = r > sp.absorber_r
        m[sel] = np.clip(np.cos(0.5 * math.pi * (r[sel] - sp.absorber_r) / (sp.rmax - sp.absorber_r)), 0, None) ** sp.absorber_power
        self.mask, self.r = t(m), t(r)
        self.d = t(np.asarray(sp.dipole_R)) if sp.dipole_R is not None else None
        # ground state of the Fourier-grid Hamiltonian
        diff = r[:, None] - r[None, :]
        T = sum(kk * kk / (2 * sp.mass) * np.cos(kk * diff) for kk in k) / sp.nr
        g = np.linalg.eigh(T + np.diag(U[0]))[1][:, 0]
        g *= np.sign(g[np.argmax(np.abs(g))]) / math.sqrt((g * g).sum() * self.dR)
        n = O.shape[0]
        self.psi = [torch.zeros((n, len(rows[s]), sp.nr), dtype=torch.complex128, device=dev) for s in (0, 1)]
        self.psi[0][:, 0] = t(g).to(torch.complex128)
        self.absorbed = torch.zeros((n, 2), dtype=torch.float64, device=dev)
        self.nbr = [[[t(np.array(v)) for v in self._neighbours(rows[s], rows[1 - s], kind)] for kind in range(6)]
                    for s in (0, 1)]

    @staticmethod
    def _neighbours(to, frm, kind):
        """Row (j, m) of Z (kinds 0, 1), S+ (2, 3), S- (4, 5), from j - 1 and j + 1: (index, coefficient)."""
        at, idx, cf = {c: i for i, c in enumerate(frm)}, [], []
        for j, m in to:
            jn, mn = j + (1 if kind % 2 else -1), m - (0, 1, -1)[kind // 2]
            if (jn, mn) not in at:
                idx.append(0)
                cf.append(0.0)
                continue
            a, b = (jn, mn), (j, m)
            if kind // 2 == 0:
                q = min(j, jn)
                v = math.sqrt(((q + 1) ** 2 - m * m) / ((2 * q + 1) * (2 * q + 3)))
            else:
                if kind // 2 == 2:  # <a|S-|b> = <b|S+|a>
                    a, b = b, a
                jj, mm = a
                if b[0] == jj + 1:
                    v = -math.sqrt((jj + mm + 1) * (jj + mm + 2) / ((2 * jj + 1) * (2 * jj + 3)))
                else:
                    v = math.sqrt((jj - mm) * (jj - mm - 1) / ((2 * jj - 1) * (2 * jj + 1)))
            idx.append(at[a if kind // 2 != 2 else b])
            cf.append(v)
        return idx, cf

    def _apply(self, s, x, kinds):
        """Sum over the kinds of coefficient times neighbour row, into surface s's rows."""
        out = None
        for k in kinds:
            i, c = self.nbr[s][k]
            if x.shape[1] == 0 or c.numel() == 0:
                continue
            v = x.index_select(1, i) * c[None, :, None]
            out = v if out is None else out + v
        if out is None:
            out = torch.zeros((x.shape[0], self.nbr[s][0][1].numel(), x.shape[2]), dtype=x.dtype, device=x.device)
        return out

    def _coupling(self, psi, E):
        ez, em, ep = E[:, 2, None, None], 0.5 * (E[:, 0] - 1j * E[:, 1])[:, None, None], 0.5 * (E[:, 0] + 1j * E[:, 1])[:, None, None]
        d = self.d if self.d is not None else self.sp.dipole
        x = self.dtau * float(E.norm(dim=1).max()) * (float(self.d.abs().max()) if self.d is not None else self.sp.dipole)
        out, term, size, n = [p.clone() for p in psi], psi, 1.0, 0
        while size > 1e-19 and n < 60:
            n += 1
            size *= x / n
            term = [(1j * self.dtau / n) * (d * (ez * self._apply(s, term[1 - s], (0, 1)) + em * self._apply(s, term[1 - s], (2, 3))
                                                 + ep * self._apply(s, term[1 - s], (4, 5)))) for s in (0, 1)]
            out = [a + b for a, b in zip(out, term)]
        return out

    def step(self, E_lab):
        """Advances every molecule; the lab dipoles (a.u.)."""
        mu = torch.empty((E_lab.shape[0], 3), dtype=torch.float64, device=E_lab.device)
        per = max(1, int(4e7 / (self.sp.nr * (self.sp.jmax + 1) ** 2)))
        for a in range(0, E_lab.shape[0], per):
            c = slice(a, a + per)
            O = self.O[c]
            E = torch.einsum("kji,kj->ki", O, E_lab[c]) / F_AU
            psi = [torch.fft.ifft(torch.fft.fft(p[c]) * self.th) * v for p, v in zip(self.psi, self.vh)]
            psi = [p * v for p, v in zip(self._coupling(psi, E), self.vh)]
            for s in (0, 1):
                self.absorbed[c, s] += ((psi[s].abs() ** 2) * (1 - self.mask ** 2)).sum((1, 2)) * self.dR
                psi[s] = torch.fft.ifft(torch.fft.fft(psi[s] * self.mask) * self.th)
                self.psi[s][c] = psi[s]
            g = psi[0].conj() * (self.d if self.d is not None else self.sp.dipole)
            Z, P, M = ((g * self._apply(0, psi[1], k)).sum((1, 2)) for k in ((0, 1), (2, 3), (4, 5)))
            m = torch.stack([(P + M).real, (P - M).imag, 2 * Z.real], 1) * self.dR
            mu[c] = torch.einsum("kij,kj->ki", O, m)
        return mu

    def populations(self):
        return torch.stack([(p.abs() ** 2).sum((1, 2)) * self.dR for p in self.psi], 1)

    def excited_R(self):
        e = self.psi[1].abs() ** 2
        return torch.stack([(e * self.r).sum((1, 2)), e.sum((1, 2))], 1) * self.dR


class _Frozen:
    """FP64 Bloch equations, one classical RK4 step per molecular step with the field held."""

    def __init__(self, sp, O, dtau, dev):
        self.sp, self.h, self.axis = sp, dtau, O[:, :, 2]
        self.w0, self.g1, self.g2 = sp.w0_ev / HARTREE_EV, T_AU / sp.T1, T_AU / sp.T2
        self.y = torch.zeros((O.shape[0], 3), dtype=torch.float64, device=dev)
        self.y[:, 2] = -1.0
        self.absorbed = torch.zeros((O.shape[0], 2), dtype=torch.float64, device=dev)

    def step(self, E):
        om = 2 * self.sp.dipole * (self.axis * E).sum(1) / F_AU

        def rhs(y):
            u, v, w = y.unbind(1)
            return torch.stack([self.w0 * v - self.g2 * u, -self.w0 * u - om * w - self.g2 * v, om * v - self.g1 * (w + 1)], 1)

        k1 = rhs(self.y)
        k2 = rhs(self.y + 0.5 * self.h * k1)
        k3 = rhs(self.y + 0.5 * self.h * k2)
        k4 = rhs(self.y + self.h * k3)
        self.y = self.y + self.h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
        return self.sp.dipole * self.y[:, :1] * self.axis

    def populations(self):
        return torch.stack([0.5 * (1 - self.y[:, 2]), 0.5 * (1 + self.y[:, 2])], 1)

    def excited_R(self):
        pe = 0.5 * (1 + self.y[:, 2])
        return torch.stack([self.sp.re * pe, pe], 1)


def _rotation(q, dev):
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    R = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                  2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                  2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1)
    return torch.from_numpy(R.reshape(-1, 3, 3)).to(dev)


def exact(case, seed):
    steps = case["preroll"] + case["steps"]
    n = case["nsim"] * case["mols"]
    msteps = -(-steps // case["substeps"])
    el = sum(fr * (int(s.split("/")[1]) + 1) ** 2 * int(s.split("/")[0])
             for fr, s in zip(_fractions(len(case["species"].split())), case["species"].split()))
    if case["model"] != "bloch" and n * el * msteps > EXACT_ELEMENT_STEPS:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    wl = _workload(case, seed)
    O = _rotation(wl.quat, dev)
    sid = torch.from_numpy(wl.species_id).to(dev)
    dtau = DT * case["substeps"] / T_AU
    groups = []
    for i, sp in enumerate(wl.species):
        at = torch.nonzero(sid == i)[:, 0]
        if at.numel():
            groups.append((at, (_Frozen if case["model"] == "bloch" else _Wavepackets)(sp, O[at], dtau, dev)))
    mu = torch.zeros((n, 3), dtype=torch.float64, device=dev)
    fld = _Fields(case, wl, seed, dev) if case["drive"] == "fdtd" else None
    if fld is None:
        amp, wave = _drive(case, seed)
        amp = torch.from_numpy(amp).to(dev).double()
    elif n:
        ijk = np.floor(wl.pos / DX).astype(np.int64)
        cell = ((wl.sim_id.astype(np.int64) * wl.nz + ijk[:, 2]) * wl.ny + ijk[:, 1]) * wl.nx + ijk[:, 0]
        cell = torch.from_numpy(cell).to(dev)
    om = torch.from_numpy(_omega(case)).to(dev)
    acc = [[torch.zeros((case["nsim"], case["nfreq"], wl.ny, wl.nx), dtype=torch.complex128, device=dev) for _ in range(4)]
           for _ in range(case["planes"])]
    for q in range(steps):
        molecular = n > 0 and q % case["substeps"] == 0
        if fld is not None:
            fld.step_h()
        dP = None
        if molecular:
            E = amp * float(wave[q]) if fld is None else torch.stack([e.reshape(-1)[cell] for e in fld.E], 1)
            new = torch.empty_like(mu)
            for at, g in groups:
                new[at] = g.step(E[at])
            if fld is not None:
                dP = []
                for c in range(3):
                    p = torch.zeros(fld.E[c].numel(), dtype=torch.float64, device=dev)
                    dP.append((p.index_add_(0, cell, new[:, c] - mu[:, c]) * (EA0 / DX ** 3)).reshape(fld.E[c].shape))
            mu = new
        if fld is not None:
            fld.step_e(dP)
            pe, ph = torch.exp(1j * om * fld.n * DT) * DT, torch.exp(1j * om * (fld.n - 0.5) * DT) * DT
            for k, a in zip(_planes(case), acc):
                v = (fld.E[0][:, k], fld.E[1][:, k], 0.5 * (fld.H[0][:, k - 1] + fld.H[0][:, k]), 0.5 * (fld.H[1][:, k - 1] + fld.H[1][:, k]))
                for c in range(4):
                    a[c] += (pe if c < 2 else ph)[None, :, None, None] * v[c][:, None]
    out = {}
    if n:
        def collect(f, width):
            o = torch.zeros((n, width), dtype=torch.float64, device=dev)
            for at, g in groups:
                o[at] = f(g)
            return o

        P, ab = collect(lambda g: g.populations(), 2), collect(lambda g: g.absorbed, 2)
        out["P_g"], out["P_e"], out["mu"] = P[:, 0], P[:, 1], mu
        if case["steps"] > 1:
            out["norm"] = P.sum(1) + ab.sum(1)
            out["R_e"] = collect(lambda g: g.excited_R(), 2)
            if case["absorber"] < 8.0:
                out["absorbed"] = ab
    if case["fields"]:
        out["E"] = [torch.stack([e[s] for e in fld.E]) for s in range(case["nsim"])]
        out["H"] = [torch.stack([h[s] for h in fld.H]) for s in range(case["nsim"])]
    for p, a in enumerate(acc):
        f = (a[0] * a[3].conj() - a[1] * a[2].conj()).real.sum((2, 3))
        out["flux%d" % p] = f * DX ** 2
    return out
