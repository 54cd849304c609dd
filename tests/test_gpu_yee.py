"""The field kernels with four columns a thread against those with one, which take arrays that are not on 16-byte
boundaries (an allocator of the caller places them): grids whose threads walk one, three and eight planes, with walks
that do not divide the planes, several simulations, both ends in z, and rows of one quad."""
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


class _Offset:
    """Places blocks of one size four bytes past their boundary."""

    def __init__(self, B, size):
        inner = B._TorchAllocator()
        self.inner, self.moved = inner, set()

        def alloc(n, ctx):
            if n != size:
                return inner._alloc(n, ctx)
            p = inner._alloc(n + 16, ctx)
            if p is None:
                return None
            self.moved.add(p + 4)
            return p + 4

        def free(p, ctx):
            inner._free(p - 4 if p in self.moved else p, ctx)
        self.c_alloc, self.c_free = B._ALLOC(alloc), B._FREE(free)


@pytest.mark.parametrize("bc", ["pml", "periodic"])
@pytest.mark.parametrize("nx,ny,nz,nsim,kz", [(40, 9, 47, 2, 1), (4, 11, 33, 1, 1), (64, 64, 230, 4, 3),
                                              (216, 216, 217, 1, 8)])
def test_four_columns_a_thread_match_one(B, nx, ny, nz, nsim, kz, bc):
    """Both kernels round each term alike up to the compiler's choice of fused products, so a step's difference is a
    few roundings of the values it adds: 8 a half step."""
    assert max(1, min(8, nx * ny * nz // 4 * nsim // (152 * 64 * 32))) == kz
    steps = 12

    def geo(nx_, ny_, nz_):
        m = np.zeros((nz_, ny_, nx_), np.uint8)
        m[nz_ // 3: nz_ // 2, 1: ny_ - 1, 1: nx_ - 2] = W.configs.MAT_SILVER
        m[2 * nz_ // 3:] = W.configs.MAT_GLASS
        return m
    src = dict(src_k=14, pulses=[[1e9, 1.5, 1e-15, 1e-16]] * nsim) if bc == "pml" else dict(src_k=-1, pml=0)
    wl = W.custom("quads", nx, ny, nz, nsim=nsim, bc_z=bc, geometry=geo, n_per_sim=0, nsteps=steps, **src)
    rng = np.random.default_rng(nx + nz)
    E0 = (rng.standard_normal((nsim, 3, nz, ny, nx)) * 1e8).astype(np.float32)
    H0 = (rng.standard_normal((nsim, 3, nz, ny, nx)) * 1e5).astype(np.float32)
    got = []
    off = _Offset(B, 4 * nx * ny * nz * nsim)
    for al in (None, off):
        sim = B.Simulation(wl, allocator=al) if al else B.Simulation(wl)
        for s in range(nsim):
            sim.write_fields(B.MS_FIELD_E, s, E0[s])
            sim.write_fields(B.MS_FIELD_H, s, H0[s])
        sim.step(steps)
        got.append([sim.fields(w, s).astype(np.float64) for w in (B.MS_FIELD_E, B.MS_FIELD_H) for s in range(nsim)])
        sim.close()
    assert len(off.moved) == 6   # the fields, and nothing else
    for a, b, first in zip(*got, [*E0, *H0]):
        assert np.linalg.norm(a - first) > 0.1 * np.linalg.norm(first)
        assert np.linalg.norm(a - b) <= 2 * 8 * steps * 2.0 ** -24 * np.linalg.norm(b)
