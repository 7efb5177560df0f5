"""ac_get_stencil_forms: which arithmetic a substep ran, where ac_get_stencil_modes counts by
the state alone."""
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


PRODUCTS, GROUP, FIELD, PLAIN = range(4)
CUBE, THIN = (24, 24, 24), (130, 4, 66)


def _pinned(n):
    f = synthetic.smooth_state(n, 3, amp=0.02)
    for q in (1, 2, 3, 5, 6, 7):
        f[q].flat[0], f[q].flat[-1] = 0.1, -0.1
    return f


@pytest.mark.parametrize("n,hs,change,form,mode", [
    (CUBE, (1, 1, 1), None, PRODUCTS, 0),
    (CUBE, (1, 1, 1), (3, 2.0 ** -4), PRODUCTS, 1),   # four binades: group products, counted FIELD
    (CUBE, (1, 1, 1), (3, 2.0 ** -9), FIELD, 1),
    (CUBE, (1, 1, 1), "flow", FIELD, 0),              # a mean flow: per-field, counted GROUP
    (CUBE, (1, 1, 1), "nan", PLAIN, 2),
    ((33, 32, 17), (1, 1.5, 0.7), None, PRODUCTS, None),
    ((33, 32, 17), (1, 1.5, 0.7), (3, 2.0 ** -9), PLAIN, None),
    (CUBE, (1, 1.5, 1), None, None, None),            # plain stencils by the box's size
    (THIN, (1, 1, 1), None, GROUP, 0),
    (THIN, (1, 1, 1), (3, 2.0 ** -4), FIELD, 1),
])
def test_forms(n, hs, change, form, mode):
    f = _pinned(n)
    if change == "flow":
        f[1] += 100.0
    elif change == "nan":
        f[2].flat[5] = np.nan
    elif change:
        f[change[0]] *= change[1]
    sim = ac.Simulation(n, L=tuple(0.25 * h * v for v, h in zip(n, hs)))
    sim.load(f)
    assert ac.ac_get_stencil_forms(sim.h) == (0, 0, 0, 0)
    sim.substep(1e-3, 0)
    assert ac.ac_get_stencil_forms(sim.h) == tuple(int(m == form) for m in range(4))
    assert ac.ac_get_stencil_modes(sim.h) == tuple(int(m == mode) for m in range(3))
    sim.close()
