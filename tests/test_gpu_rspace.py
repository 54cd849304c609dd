"""The R-space passes on the reachable rows over their range of J, radial grids
and coupling-series lengths (no field, one term, two, several), with the
absorber cutting into the packet, against the FP64 oracle at the plain FP32
tolerances."""
import numpy as np
import pytest

import workloads as W
from oracle.coupled import PrescribedOracle

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


def _check(B, nr, jmax, path, E0, state_form=0, nsteps=24, nmol=3):
    sp = W.Species(nr=nr, jmax=jmax, A=0.05, absorber_r=2.4)
    wl = W.custom("rspace", 8, 8, 48, n_per_sim=nmol, species=[sp], layer=(20, 24), seed=nr + jmax, nsteps=nsteps)
    amp, wave = W.prescribed_drive(nmol, nsteps, wl.dt, E0=E0, carrier_ev=6.0, fwhm=0.5e-15, t0=0.05e-15)
    sim = B.Simulation(wl, drive=B.MS_DRIVE_PRESCRIBED, mol_path=path, state_form=state_form)
    sim.set_prescribed(amp, wave)
    sim.step(nsteps)
    P, mu, (ab, Re) = sim.populations(), sim.dipoles(), sim.dissociation()
    sim.close()
    o = PrescribedOracle(wl, amp, wave).run(nsteps)
    Po, Ro = o.populations(), o.excited_R()
    assert np.abs(P - Po).max() < 1e-5
    sel = Po[:, 1] > 1e-10
    if jmax > 0 and E0 >= 1e9:
        assert sel.any()
    if sel.any():
        assert np.max(np.abs(P[sel, 1] - Po[sel, 1]) / Po[sel, 1]) < 1e-3
    assert np.abs(mu - o.mu).max() <= 1e-4 * np.abs(o.mu).max()
    assert np.abs(ab - o.absorbed()).max() < 1e-6
    assert np.abs(Re - Ro).max() <= 1e-3 * Ro.max() + 1e-12
    assert np.abs(P.sum(axis=1) + ab.sum(axis=1) - 1).max() < 1e-6


@pytest.mark.parametrize("E0", [0.0, 1e6, 1e9, 6e10])
@pytest.mark.parametrize("nr,jmax,path", [(64, 0, 2), (128, 0, 1), (128, 1, 1), (256, 1, 2), (64, 2, 2), (128, 3, 1),
                                          (64, 4, 2), (128, 4, 1), (128, 4, 2), (256, 4, 2)])
def test_whole_rotor_kernel(B, nr, jmax, path, E0):
    _check(B, nr, jmax, path, E0)


@pytest.mark.parametrize("E0", [0.0, 1e6, 1e9, 6e10])
@pytest.mark.parametrize("nr,jmax,form", [(64, 5, 0), (128, 6, 1), (64, 7, 1), (256, 8, 0), (128, 8, 1)])
def test_column_kernel(B, nr, jmax, form, E0):
    _check(B, nr, jmax, 2, E0, state_form=form)


@pytest.mark.parametrize("nr,jmax,nmol", [(64, 1, 45), (128, 3, 14), (128, 4, 7), (256, 4, 3), (256, 9, 2)])
def test_dissociation_readout_blocks(B, nr, jmax, nmol):
    """The readout's blocks: several molecules each with a remainder, one
    each, and a molecule over two passes."""
    _check(B, nr, jmax, 2, 6e10, nmol=nmol)


@pytest.mark.parametrize("nfreq,calls", [(1, (1, 15, 16, 17, 3)), (9, (33, 1, 40)), (8, (7,) * 6)])
def test_detector_batches_do_not_depend_on_the_calls(B, nfreq, calls):
    """Detector samples are added up to 16 steps at a time within a call, in
    their order: any division of a run into calls gives the accumulators of
    single steps, bit for bit."""
    def geo(nx, ny, nz):
        m = np.zeros((nz, ny, nx), np.uint8)
        m[24:28, 2:, 3:-4] = W.configs.MAT_SILVER
        return m
    n = sum(calls)
    wl = W.custom("dft", 20, 18, 48, nsim=2, src_k=14, pulses=[[1e9, 1.5, 1e-15, 1e-16]] * 2, geometry=geo,
                  n_per_sim=0, nsteps=n)
    planes, om = [12, 40, 25], np.linspace(1.0, 3.0, nfreq) / 6.582119569e-16
    got = []
    for steps in ((1,) * n, calls):
        sim = B.Simulation(wl, step_graphs=B.MS_GRAPHS_AUTO)
        sim.set_detectors(planes, om)
        for k in steps:
            sim.step(k)
        got.append(np.array([[[sim.dft(p, s, c, f) for f in range(nfreq)] for c in range(4) for s in range(2)]
                             for p in range(3)]))
        sim.close()
    assert (np.abs(got[0]).max(axis=(0, 2, 3, 4)) > 0).all()   # every component of both simulations
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("nx,ny,nsim,nfreq", [(8, 8, 1, 1), (16, 32, 2, 3), (19, 27, 3, 2), (150, 130, 1, 2)])
def test_flux_is_the_sum_over_the_accumulators(B, nx, ny, nsim, nfreq):
    """Flux spectra against FP64 sums of the accumulators that are read back: planes below, of and above a block's
    threads.  A term has three roundings; a sum adds at most one per cell of a thread, five over a warp and 16."""
    wl = W.custom("flux", nx, ny, 48, nsim=nsim, src_k=14, pulses=[[1e9, 1.5, 1e-15, 1e-16]] * nsim, n_per_sim=0,
                  nsteps=40)
    sim = B.Simulation(wl)
    sim.set_detectors([40, 25], np.linspace(1.0, 3.0, nfreq) / 6.582119569e-16)
    sim.step(40)
    tol = (3 + -(-nx * ny // 512) + 5 + 16 + 2) * 2.0 ** -53
    for d in range(2):
        got = sim.flux(d)
        for s in range(nsim):
            for f in range(nfreq):
                ex, ey, hx, hy = (sim.dft(d, s, c, f) for c in range(4))
                a, b = ex * np.conj(hy), ey * np.conj(hx)
                size = (np.abs(ex.real * hy.real) + np.abs(ex.imag * hy.imag) + np.abs(ey.real * hx.real)
                        + np.abs(ey.imag * hx.imag)).sum()
                want = np.sum((a - b).real.astype(np.longdouble))
                assert size > 0 and abs(got[s, f] / wl.dx ** 2 - want) <= 1.5 * tol * size
    sim.close()


@pytest.mark.parametrize("piece", [1, 5000, 16384, 16385])
def test_reads_by_pieces(B, piece):
    """Reads of every size class (staged, or straight to their arrays) give the values of one whole read."""
    n = 16400
    wl = W.custom("reads", 32, 32, 64, src_k=14, pulses=[[1e10, 1.5, 1e-15, 2e-16]], layer=(20, 44), n_per_sim=n,
                  species=[W.species_config0(jmax=1)], seed=3, nsteps=40)
    sim = B.Simulation(wl)
    sim.step(40)
    whole = (sim.populations(), sim.dipoles()) + sim.dissociation()
    for first in ([0, 7, n - 1] if piece == 1 else range(0, n, piece)):
        k = min(piece, n - first)
        part = (sim.populations(first, k), sim.dipoles(first, k)) + sim.dissociation(first, k)
        for a, b in zip(whole, part):
            assert np.array_equal(a[first:first + k], b)
    assert np.abs(whole[1]).max() > 0 and whole[3].min() >= 0
    sim.close()


@pytest.mark.parametrize("captured", [1, 2, 3])
def test_steps_captured_by_the_caller_replay(B, captured):
    """A caller's own graph of a few steps, replayed: the step counter's two
    slots end each replay where it began, so the replays, and steps after
    them, are those of plain stepping bit for bit."""
    import torch
    wl = W.custom("captured", 20, 12, 48, src_k=14, pulses=[[1e10, 1.5, 1e-15, 2e-16]], layer=(20, 24), n_per_sim=40,
                  species=[W.species_config0(jmax=1), W.Species(nr=128, jmax=3)], fractions=[0.5, 0.5], seed=3,
                  nsteps=60)
    def out(sim):
        r = sim.populations(), sim.dipoles(), sim.fields(B.MS_FIELD_E), sim.fields(B.MS_FIELD_H)
        sim.close()
        return r
    a = B.Simulation(wl, step_graphs=B.MS_GRAPHS_OFF)
    a.step(5 + 4 * captured + 16)
    b = B.Simulation(wl)
    b.step(5)
    b.populations()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=b.stream):
        b.step(captured)
    with torch.cuda.stream(b.stream):
        for _ in range(4):
            g.replay()
    b.stream.synchronize()
    b.step(16)
    for x, y in zip(out(a), out(b)):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("captured", [1, 2])
def test_replays_between_other_calls(B, captured):
    """A caller's graph replayed after odd numbers of plain and of recorded
    steps starts from the step that those have reached."""
    import torch
    wl = W.custom("between", 20, 12, 48, src_k=14, pulses=[[1e10, 1.5, 1e-15, 2e-16]], layer=(20, 24), n_per_sim=40,
                  species=[W.species_config0(jmax=1)], seed=3, nsteps=60)

    def out(sim):
        r = sim.populations(), sim.dipoles(), sim.fields(B.MS_FIELD_E), sim.fields(B.MS_FIELD_H)
        sim.close()
        return r

    a = B.Simulation(wl, step_graphs=B.MS_GRAPHS_OFF)
    a.step(5 + 3 * captured + 1 + 3 + 17)
    b = B.Simulation(wl)
    b.step(5)
    b.populations()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=b.stream):
        b.step(captured)

    def replay():
        with torch.cuda.stream(b.stream):
            g.replay()

    replay()
    b.step(1)
    replay()
    b.record_local_fields(np.arange(4), 3)
    replay()
    b.step(17)
    for x, y in zip(out(a), out(b)):
        assert np.array_equal(x, y)
