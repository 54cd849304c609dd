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
