"""Graphs that the caller captures and replays, against the FP64 oracle at the
plain FP32 tolerances: what they captured stays right when the plan or the
loaded state, and with them the order of the stored rows, change under them."""
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


def _capture(sim, n, step=None):
    """A graph of n steps of the handle, and a call that replays it k times."""
    import torch
    sim.populations()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=sim.stream):
        (step or sim.step)(n)

    def replay(k):
        with torch.cuda.stream(sim.stream):
            for _ in range(k):
                g.replay()
    return replay


def _workload(nr, jmax, nmol, nsteps, dipole_R=None):
    sp = W.Species(nr=nr, jmax=jmax, A=0.05, dipole_R=dipole_R)
    wl = W.custom("graphs", 8, 8, 48, n_per_sim=nmol, species=[sp], layer=(20, 24), seed=nr + jmax, nsteps=nsteps)
    amp, wave = W.prescribed_drive(nmol, nsteps, wl.dt, E0=3e10, carrier_ev=6.0, fwhm=0.5e-15, t0=0.4e-15)
    return wl, amp, wave


def _close(sim, o):
    P, mu = sim.populations(), sim.dipoles()
    assert o.populations()[:, 1].max() > 1e-6
    assert np.abs(P - o.populations()).max() < 1e-5
    assert np.abs(mu - o.mu).max() < 1e-4 * np.abs(o.mu).max()


KINDS = [  # nr, jmax, molecules, layout, precision, d(R), the captured plan, another plan
    (128, 4, 5, 1, 0, False, (1, 0, 0), (2, 2, 16)), (64, 2, 7, 2, 0, False, (2, 1, 0), (2, 3, 8)),
    (128, 3, 5, 2, 1, False, (2, 0, 0), (2, 4, 32)), (128, 2, 5, 1, 0, True, None, None),
    (64, 7, 4, 2, 0, False, (2, 0, 0), (2, 2, 16)), (128, 5, 4, 2, 0, False, (2, 4, 8), (2, 0, 0)),
    (64, 10, 2, 2, 0, False, (2, 0, 0), (2, 4, 8)), (64, 6, 3, 1, 0, False, (1, 3, 8), (2, 0, 0))]


@pytest.mark.parametrize("batches", [0, 2])
@pytest.mark.parametrize("nr,jmax,nmol,path,prec,dip,plan,other", [k for k in KINDS if k[6]])
def test_replays_after_plan_changes(B, nr, jmax, nmol, path, prec, dip, plan, other, batches):
    n = 48
    wl, amp, wave = _workload(nr, jmax, nmol, n)
    sim = B.Simulation(wl, drive=B.MS_DRIVE_PRESCRIBED, precision=prec, mol_path=path)
    sim.set_prescribed(amp, wave)
    sim.set_plan(0, *plan)
    sim.set_batches(batches)
    sim.step(5)
    replay = _capture(sim, 4)
    replay(2)                       # 13
    sim.set_plan(0, *other)
    replay(2)                       # 21
    sim.step(3)                     # 24
    replay(1)                       # 28
    sim.set_plan(0, *plan)
    replay(2)                       # 36
    sim.step(4)                     # 40
    sim.populations()
    _close(sim, PrescribedOracle(wl, amp, wave).run(40))
    sim.close()


@pytest.mark.parametrize("nr,jmax,nmol,path,prec,dip,plan,other", KINDS)
def test_replays_after_loads(B, tmp_path, nr, jmax, nmol, path, prec, dip, plan, other):
    """A graph captured on an ordinary state, replayed on a loaded one that populates every row, then on an ordinary
    one again; and one captured while every row was populated, replayed on an ordinary state."""
    n = 40
    wl, amp, wave = _workload(nr, jmax, nmol, n, tuple(np.linspace(1.2, 0.4, nr)) if dip else None)
    sp = wl.species[0]
    kw = dict(drive=B.MS_DRIVE_PRESCRIBED, precision=prec, mol_path=path)
    a = B.Simulation(wl, **kw)
    plain, every = str(tmp_path / "plain.ck"), str(tmp_path / "every.ck")
    a.save(plain)
    a.close()
    raw = bytearray(open(plain, "rb").read())
    st = np.frombuffer(raw, np.complex64, nmol * 2 * sp.nrot * nr, ctypes.sizeof(_CkHeader) + 8)
    st = st.reshape(nmol, 2, sp.nrot, nr)
    row = st[:, 0, 0].copy() * np.float32(np.sqrt(0.5))
    st[:, 0, 0], st[:, 0, 2] = row, row    # half of the population into (ground, j = 1, m = 0)
    open(every, "wb").write(raw)
    oe = PrescribedOracle(wl, amp, wave)
    psi = oe.groups[0][1].psi
    psi[:, 0, 0] *= np.sqrt(0.5)
    psi[:, 0, 2] = psi[:, 0, 0]
    oe.run(n)
    op = PrescribedOracle(wl, amp, wave).run(n)

    sim = B.Simulation(wl, **kw)
    sim.set_prescribed(amp, wave)
    if plan:
        sim.set_plan(0, *plan)
    first = _capture(sim, 4)
    for path_, o, replay in ((every, oe, first), (plain, op, first), (every, oe, None), (plain, op, None)):
        sim.load(path_)
        if replay is None and path_ == every:
            second = _capture(sim, 4)
            sim.load(path_)         # capturing has advanced nothing
        (replay or second)(n // 4)
        _close(sim, o)
    sim.close()


@pytest.mark.parametrize("substeps,captured", [(1, 1), (1, 4), (3, 3), (3, 6)])
def test_replays_count(B, tmp_path, substeps, captured):
    """Capture, replay, save, load, step: the steps, the cadence, the source and the detectors' phases are those of
    plain stepping, bit for bit, in the handle and in one that loads its checkpoint."""
    wl = W.custom("count", 20, 12, 48, src_k=14, pulses=[[1e10, 1.5, 1e-15, 2e-16]], layer=(20, 24), n_per_sim=40,
                  species=[W.species_config0(jmax=1)], seed=3, nsteps=100, mol_substeps=substeps)
    planes, om = [12, 40], np.linspace(1.0, 3.0, 2) / 6.582119569e-16
    lead, reps, tail = 2 * substeps, 5, 7

    def make(graphs):
        s = B.Simulation(wl, step_graphs=graphs)
        s.set_detectors(planes, om)
        return s

    def out(s):
        r = [s.populations(), s.dipoles(), s.fields(B.MS_FIELD_E), s.fields(B.MS_FIELD_H)]
        r += [s.dft(p, 0, c, f) for p in range(2) for c in range(4) for f in range(2)]
        s.close()
        return r

    a = make(B.MS_GRAPHS_OFF)
    a.step(lead + reps * captured + tail)
    b = make(B.MS_GRAPHS_AUTO)
    b.step(lead)
    replay = _capture(b, captured)
    assert b.steps == lead                 # capturing takes no step
    replay(reps)
    p = str(tmp_path / "c.ck")
    b.save(p)
    assert b.steps == lead + reps * captured
    c = make(B.MS_GRAPHS_AUTO)
    c.load(p)
    assert c.steps == lead + reps * captured
    b.step(tail)
    c.step(tail)
    assert a.steps == b.steps == c.steps
    ref = out(a)
    for s in (b, c):
        for x, y in zip(ref, out(s)):
            assert np.array_equal(x, y)
