"""Which calls replay a captured cycle, and that the replays are the steps."""
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
    _graph_launches(lambda: torch.zeros(1, device="cuda"))  # the profiler's first session may miss calls
    return binding


def _graph_launches(fn):
    """cudaGraphLaunch calls that fn makes, or None where the profiler records no runtime calls."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
        fn()
        torch.cuda.synchronize()
    names = [e.name for e in p.events()]
    return names.count("cudaGraphLaunch") if any(n.startswith("cuda") for n in names) else None


def _run(B, substeps, calls, graphs, planes=None):
    wl = W.custom("cycles", 20, 12, 48, src_k=14, pulses=[[1e10, 1.5, 1e-15, 2e-16]], layer=(20, 24), n_per_sim=20,
                  species=[W.species_config0(jmax=1)], seed=3, nsteps=200, mol_substeps=substeps)
    sim = B.Simulation(wl, step_graphs=graphs)
    if planes:
        sim.set_detectors(planes, np.linspace(1.0, 3.0, 5) / 6.582119569e-16)
    launches = []
    for n in calls:
        if graphs == B.MS_GRAPHS_OFF:
            sim.step(n)
        else:
            launches.append(_graph_launches(lambda: sim.step(n)))
    out = [sim.populations(), sim.dipoles(), sim.fields(B.MS_FIELD_E), sim.fields(B.MS_FIELD_H)]
    if planes:
        out += [sim.dft(p, 0, c, f) for p in range(len(planes)) for c in range(4) for f in range(5)]
    sim.close()
    return launches, out


@pytest.mark.parametrize("substeps,calls,want", [
    (1, (7, 8, 17), (0, 1, 2)), (3, (9, 17, 1, 20), (1, 1, 0, 2)), (9, (9, 9, 4, 23), (1, 1, 0, 2)),
    (11, (11, 22, 5, 17), (1, 2, 0, 1)), (40, (39, 1, 40, 80), (0, 0, 1, 2))])
def test_whole_cycles_replay(B, substeps, calls, want):
    """A cycle is the least number of whole molecular cycles with 8 field steps, odd ones too: every call that holds
    one from the start of a molecular cycle on replays it."""
    launches, got = _run(B, substeps, calls, B.MS_GRAPHS_AUTO)
    _, ref = _run(B, substeps, calls, B.MS_GRAPHS_OFF)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)
    if None in launches:
        pytest.skip("the profiler records no runtime calls")
    assert tuple(launches) == want


@pytest.mark.parametrize("substeps,calls,want", [
    (1, (7, 8, 15, 16, 17, 1, 40, 25), (0, 1, 1, 2, 2, 0, 5, 3)), (3, (9, 17, 1, 20, 31), (1, 1, 0, 2, 3)),
    (20, (20, 5, 55, 40), (1, 0, 2, 2))])
def test_cycles_with_detectors(B, substeps, calls, want):
    """Detectors leave the cycle's length as it is, and the accumulators are those of single steps: cycles shorter
    than a batch of kept samples, longer ones, and steps before, between and after them."""
    launches, got = _run(B, substeps, calls, B.MS_GRAPHS_AUTO, planes=[12, 40])
    _, ref = _run(B, substeps, (1,) * sum(calls), B.MS_GRAPHS_OFF, planes=[12, 40])
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)
    if None in launches:
        pytest.skip("the profiler records no runtime calls")
    assert tuple(launches) == want


def test_short_calls_keep_no_samples(B):
    """Calls of up to three steps add their samples from the fields: two half steps and one launch a step."""
    wl = W.custom("single", 20, 18, 48, src_k=14, pulses=[[1e9, 1.5, 1e-15, 1e-16]], n_per_sim=0, nsteps=10)
    sim = B.Simulation(wl)
    sim.set_detectors([12, 40], np.array([2.0, 3.0]) / 6.582119569e-16)
    for n, most in ((1, 3), (2, 6), (3, 9), (4, 13)):
        sim.timing_begin()
        sim.step(n)
        assert sim.timing_end()[2] <= most
    sim.close()


class _NoBlocksOf:
    """An allocator that refuses blocks of one size."""

    def __init__(self, B, size):
        inner = B._TorchAllocator()
        self.inner, self.refused = inner, 0

        def alloc(n, ctx):
            if n == size:
                self.refused += 1
                return None
            return inner._alloc(n, ctx)
        self.c_alloc, self.c_free = B._ALLOC(alloc), B._FREE(inner._free)


def test_detectors_without_memory_for_kept_samples(B):
    """Detectors are set where only the kept samples find no memory, with the same accumulators."""
    nx, ny, planes, om = 20, 18, [12, 40], np.linspace(1.0, 3.0, 2) / 6.582119569e-16
    wl = W.custom("no ring", nx, ny, 48, src_k=14, pulses=[[1e9, 1.5, 1e-15, 1e-16]], n_per_sim=0, nsteps=100)
    got = []
    for al in (None, _NoBlocksOf(B, 384 * len(planes) * nx * ny)):
        sim = B.Simulation(wl, allocator=al) if al else B.Simulation(wl)
        sim.set_detectors(planes, om)
        for n in (1, 5, 24, 13):
            sim.step(n)
        got.append([sim.dft(p, 0, c, f) for p in range(2) for c in range(4) for f in range(2)])
        sim.close()
    assert al.refused == 1
    assert max(np.abs(a).max() for a in got[0]) > 0
    for a, b in zip(*got):
        assert np.array_equal(a, b)
