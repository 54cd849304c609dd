"""The rows a full-form species processes: the point-resident kernels and the
static rule's kernels from J = 5 on work on the rows that the j = 0 start can
populate, plans that name a tiled, pair or chunked kernel on every row, and a
loaded state that populates the other rows makes every kernel process them.
Against the FP64 oracle at the plain FP32 tolerances (populations 1e-5
absolute, dipoles 1e-4 of the largest)."""
import ctypes

import numpy as np
import pytest

import workloads as W
from oracle.coupled import PrescribedOracle
from test_gpu_state import _CkHeader

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2209_04487_gb300 import build
    build.build()
    from paper_2209_04487_gb300 import binding
    return binding


def _workload(nr, jmax, nmol, nsteps, dipole_R=None):
    sp = W.Species(nr=nr, jmax=jmax, A=0.05, dipole_R=dipole_R)
    wl = W.custom("rows", 8, 8, 48, n_per_sim=nmol, species=[sp], layer=(20, 24), seed=nr + jmax, nsteps=nsteps)
    amp, wave = W.prescribed_drive(nmol, nsteps, wl.dt, E0=3e10, carrier_ev=6.0, fwhm=0.5e-15, t0=0.4e-15)
    return wl, amp, wave


def _state(path, nmol, sp):
    raw = bytearray(open(path, "rb").read())
    off = ctypes.sizeof(_CkHeader) + 8
    st = np.frombuffer(raw, np.complex64, nmol * 2 * sp.nrot * sp.nr, off).reshape(nmol, 2, sp.nrot, sp.nr)
    return raw, st


@pytest.mark.parametrize("nr,jmax,nmol,path,prec,dip", [
    (128, 4, 7, "fused", 0, False), (64, 1, 9, "streaming", 0, False), (128, 3, 5, "streaming", 1, False),
    (128, 2, 5, "fused", 0, True), (64, 5, 5, "streaming", 0, False), (128, 8, 3, "streaming", 0, False),
    (64, 8, 3, "streaming", 1, False), (64, 9, 2, "streaming", 0, False)])
def test_loaded_state_with_the_other_rows_populated(B, tmp_path, nr, jmax, nmol, path, prec, dip):
    dR = tuple(np.linspace(1.2, 0.4, nr)) if dip else None
    n = 80
    wl, amp, wave = _workload(nr, jmax, nmol, n, dR)
    sp = wl.species[0]
    kw = dict(drive=B.MS_DRIVE_PRESCRIBED, precision=prec,
              mol_path=B.MS_MOL_FUSED if path == "fused" else B.MS_MOL_STREAMING)
    a = B.Simulation(wl, **kw)
    p = str(tmp_path / "a.ck")
    a.save(p)
    a.close()
    raw, st = _state(p, nmol, sp)
    assert np.count_nonzero(np.abs(st).sum(axis=(0, 3))) == 1
    # half of the amplitude squared into (ground, j = 1, m = 0), the other half stays: both parts run
    row = st[:, 0, 0].copy() * np.float32(np.sqrt(0.5))
    st[:, 0, 0], st[:, 0, 2] = row, row
    open(p, "wb").write(raw)
    b = B.Simulation(wl, **kw)
    b.load(p)
    b.set_prescribed(amp, wave)
    b.step(n)
    P, mu = b.populations(), b.dipoles()
    b.save(p)
    b.close()
    o = PrescribedOracle(wl, amp, wave)
    psi = o.groups[0][1].psi
    psi[:, 0, 0] *= np.sqrt(0.5)
    psi[:, 0, 2] = psi[:, 0, 0]
    o.run(n)
    assert np.abs(P - o.populations()).max() < 1e-5
    assert np.abs(mu - o.mu).max() < 1e-4 * np.abs(o.mu).max()
    _, st = _state(p, nmol, sp)
    pop = (np.abs(st.astype(np.complex128)) ** 2).sum(axis=(0, 3))
    assert (pop[0, 1:4] > 0).all() and (pop[1, 1:4] > 0).all()   # both halves of the j <= 1 rows


@pytest.mark.parametrize("nr,jmax,nmol,plans", [
    (128, 4, 5, [(1, 1, 0), (2, 2, 16), (2, 1, 0), (2, 4, 32), (1, 0, 0)]),
    (64, 7, 4, [(2, 0, 0), (2, 3, 8), (2, 0, 0), (2, 4, 16), (2, 2, 32)]),
    (64, 10, 2, [(2, 0, 0), (2, 4, 8), (2, 0, 0)])])
def test_plans_change_and_checkpoints_move_under_way(B, tmp_path, nr, jmax, nmol, plans):
    """A run that changes its plan (and with it the order of the rows) every 16
    steps, saved and loaded into a handle of another plan at each change."""
    n = 16 * len(plans)
    wl, amp, wave = _workload(nr, jmax, nmol, n)
    o = PrescribedOracle(wl, amp, wave).run(n)
    p = str(tmp_path / "p.ck")
    sim = B.Simulation(wl, drive=B.MS_DRIVE_PRESCRIBED, mol_path=B.MS_MOL_STREAMING)
    sim.set_prescribed(amp, wave)
    for k, plan in enumerate(plans):
        sim.set_plan(0, *plan)
        sim.step(16)
        before = sim.populations()
        sim.save(p)
        assert np.array_equal(before, sim.populations())
        sim.step(0)
        other = B.Simulation(wl, drive=B.MS_DRIVE_PRESCRIBED, mol_path=B.MS_MOL_STREAMING)
        other.set_prescribed(amp, wave)
        other.set_plan(0, *plans[(k + 1) % len(plans)])
        other.load(p)
        sim.close()
        sim = other
    P, mu = sim.populations(), sim.dipoles()
    _, Re = sim.dissociation()
    sim.close()
    assert np.abs(P - o.populations()).max() < 1e-5
    assert np.abs(mu - o.mu).max() < 1e-4 * np.abs(o.mu).max()
    Ro = o.excited_R()
    assert np.abs(Re - Ro).max() < 1e-3 * Ro.max()
