"""AC_STENCIL_AUTO where the integer form's memory cannot be had: the plain binary64
stencils run in its place, bit for bit, with any spacing.
"""
import numpy as np
import pytest
import torch

from paper_2103_01597_gb300 import ac, build, synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    ac.load_library()
    torch.cuda.init()


def _sim(n, hs, f, mode=ac.AC_STENCIL_AUTO, stream=None):
    sim = ac.Simulation(n, L=tuple(0.25 * h * v for v, h in zip(n, hs)), stream=stream)
    ac.ac_set_stencil_mode(sim.h, mode)
    sim.load(f)
    return sim


def _plain(n, hs, f):
    sim = _sim(n, hs, f, ac.AC_STENCIL_FP64)
    sim.step(1e-3)
    out = sim.store()
    sim.close()
    return out


HS = [(1.0, 1.5, 1.0), (1.0, 1.0, 1.0)]


@pytest.mark.parametrize("hs", HS)
def test_no_memory_left(hs):
    n = (200, 190, 180)  # copies of 470 MB
    f = synthetic.noise_state(n, 3, sigma=1e-2)
    want = _plain(n, hs, f)
    sim = _sim(n, hs, f)
    sim.store()  # the staging buffer
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    filler = torch.empty(free - (300 << 20), dtype=torch.uint8, device="cuda")
    try:
        sim.step(1e-3)
        assert not ac.ac_get_stencil_path(sim.h)
    finally:
        del filler
        torch.cuda.empty_cache()
    assert np.array_equal(sim.store(), want)
    # memory is back: the integer form from the next choice of the mode on
    ac.ac_set_stencil_mode(sim.h, ac.AC_STENCIL_AUTO)
    sim.load(f)
    sim.step(1e-3)
    got = sim.store()
    sim.close()
    assert not np.array_equal(got, want)
    assert np.max(np.abs(got - want)) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("hs", HS)
def test_first_step_under_capture(hs):
    n = (33, 32, 17)
    f = synthetic.noise_state(n, 5, sigma=1e-2)
    want = _plain(n, hs, f)
    stream = torch.cuda.Stream()
    sim = _sim(n, hs, f, stream=stream.cuda_stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        sim.step(1e-3)
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(sim.store(), want)
    sim.load(f)
    sim.step(1e-3)  # outside a capture: the integer form
    assert not np.array_equal(sim.store(), want)
    sim.close()
