"""Bounded waits of the integer-sum substep that run out, without a fault: the limit is set
so low that the kernel gives up on its own copies.  It has to end (after the copies it
asked for have landed), the host has to learn of it, and the next handle has to compute
what it always does.
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


def _sim(n):
    sim = ac.Simulation(n, L=tuple(0.25 * v for v in n), force_amp=0.0, seed=1)
    sim.load(synthetic.smooth_state(n, 3, amp=0.2))
    return sim


def _reference(n):
    sim = _sim(n)
    sim.step(1e-3)
    out = sim.store()
    sim.close()
    return out


# one tile and one plane; ragged tiles; more CTAs than run at once, several planes each
@pytest.mark.parametrize("n", [(16, 16, 1), (40, 24, 20), (128, 128, 96)])
@pytest.mark.parametrize("polls", [0, 1])
def test_substep_gives_up_and_the_next_one_is_sound(n, polls):
    want = _reference(n)
    sim = _sim(n)
    ac.ac_diag_substep_polls(sim.h, polls)
    sim.substep(1e-3, 0)
    if polls == 0:  # (one poll waits microseconds, within which a copy may well land)
        with pytest.raises(ac.AcError) as ei:
            sim.store()
        assert ei.value.code == ac.AC_ERR_TIMEOUT
        sim.store()  # reported once
    sim.close()
    assert np.array_equal(_reference(n), want)


REPORTS = {
    "store_w": lambda sim: sim.store_w(),
    "reduce": lambda sim: sim.reduce(ac.AC_MAX, ac.AC_UX),
    "last_cfl": lambda sim: ac.ac_last_cfl(sim.h),
    "modes": lambda sim: ac.ac_get_stencil_modes(sim.h),
    "next_step": lambda sim: (torch.cuda.synchronize(), sim.step(1e-3)),
}


@pytest.mark.parametrize("call", sorted(REPORTS))
def test_every_call_that_waits_reports_it_once(call):
    """The step's last substep gives up; a program that never stores the state still learns
    of it."""
    sim = _sim((40, 24, 20))
    sim.substep(1e-3, 0)
    sim.substep(1e-3, 1)
    ac.ac_diag_substep_polls(sim.h, 0)
    sim.substep(1e-3, 2)
    ac.ac_diag_substep_polls(sim.h, 1 << 18)
    with pytest.raises(ac.AcError) as ei:
        REPORTS[call](sim)
    assert ei.value.code == ac.AC_ERR_TIMEOUT
    try:
        REPORTS[call](sim)
    except ac.AcError as e:  # (the undefined state may hold anything)
        assert e.code == ac.AC_ERR_NONFINITE
    sim.close()
