"""Sums over a molecule's state against their FP64 values on that same state
(read from a checkpoint), so that only the summation's rounding is seen."""
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


def _state(path, nmol, sp, parity):
    """[nmol][2][nrot][nr] of the checkpoint's wavepackets; the reduced form has (ground, even j), (excited, odd j)."""
    rows = sp.nrot if parity else 2 * sp.nrot
    st = np.frombuffer(open(path, "rb").read(), np.complex64, nmol * rows * sp.nr, ctypes.sizeof(_CkHeader) + 8)
    st = st.reshape(nmol, rows, sp.nr).astype(np.complex128)
    if not parity:
        return st.reshape(nmol, 2, sp.nrot, sp.nr)
    out = np.zeros((nmol, 2, sp.nrot, sp.nr), np.complex128)
    at = 0
    for s in (0, 1):
        for j in range(s, sp.jmax + 1, 2):
            out[:, s, j * j:(j + 1) ** 2] = st[:, at:at + 2 * j + 1]
            at += 2 * j + 1
    return out


@pytest.mark.parametrize("nr,jmax,form", [(64, 5, 0), (128, 6, 1), (64, 7, 0), (128, 8, 0), (256, 8, 1)])
@pytest.mark.parametrize("steps", [1, 2])
def test_column_kernel_dipole_sums(B, tmp_path, nr, jmax, form, steps):
    """The first steps' excited rows are i E'_x and E'_y times the ground row; the part that is not in the dipole is many
    times the dipole and has opposite signs at m = 1 and m = -1, so a sum that rounds at that part's size is off by as
    many more roundings.  A sum at the dipole's own size has about 16: two products and three additions of a point,
    seven levels of addition over points and warps, five of the rotation, two factors."""
    nmol = 64
    sp = W.Species(nr=nr, jmax=jmax)
    wl = W.custom("sums", 8, 8, 48, n_per_sim=nmol, species=[sp], layer=(20, 24), seed=nr + jmax, nsteps=steps)
    amp = np.random.default_rng(jmax).standard_normal((nmol, 3)).astype(np.float32) * np.float32(1e9)
    wave = np.ones(steps, np.float32)
    sim = B.Simulation(wl, drive=B.MS_DRIVE_PRESCRIBED, state_form=form)
    sim.set_prescribed(amp, wave)
    sim.step(steps)
    mu = sim.dipoles()
    p = str(tmp_path / "s.ck")
    sim.save(p)
    sim.close()
    ens = PrescribedOracle(wl, amp, wave).groups[0][1]
    want = np.einsum("kij,kj->ki", ens.O.astype(np.float32).astype(np.float64),
                     ens.dipole_mol(_state(p, nmol, sp, bool(form))))
    assert np.linalg.norm(mu - want) <= 16 * 2.0 ** -24 * np.linalg.norm(want)
