"""A molecule whose local field is not a number: the step latches MS_ENUMERIC and leaves the coupling out."""
import ctypes as C

import numpy as np
import pytest

import workloads as W

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


@pytest.mark.parametrize("nr,jmax,path,form", [(128, 4, 1, 0), (64, 1, 2, 0), (64, 3, 2, 1), (128, 8, 2, 0), (64, 6, 2, 1),
                                               (64, 9, 2, 0)])
def test_a_field_that_is_not_a_number(B, nr, jmax, path, form):
    nmol, n = 3, 4
    wl = W.custom("nan", 8, 8, 48, n_per_sim=nmol, species=[W.Species(nr=nr, jmax=jmax)], layer=(20, 24), seed=nr,
                  nsteps=n)
    amp = np.zeros((nmol, 3), np.float32)
    amp[0], amp[1, 1] = 1e9, np.nan
    sim = B.Simulation(wl, drive=B.MS_DRIVE_PRESCRIBED, mol_path=path, state_form=form)
    sim.set_prescribed(amp, np.ones(n, np.float32))
    sim.step(n)
    Pg, Pe, mu = np.empty(nmol), np.empty(nmol), np.empty((nmol, 3))
    ptr = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))  # noqa: E731
    assert B.LIB.ms_read_populations(sim.h, 0, nmol, ptr(Pg), ptr(Pe)) == B.MS_ENUMERIC
    assert B.LIB.ms_read_dipoles(sim.h, 0, nmol, ptr(mu)) == B.MS_ENUMERIC
    sim.close()
    assert np.isfinite(Pg).all() and np.isfinite(Pe).all() and np.isfinite(mu).all()
    assert Pe[0] > 0 and (Pg[1], Pe[1]) == (Pg[2], Pe[2]) and (mu[1:] == 0).all()   # molecule 2 has no field
