"""The search for the largest CFL speed of binary64 states, where a cell of its first guess
is not finite and where speeds leave binary32's range (1e-12 relative, the bound of
test_gpu_substep.py).
"""
import math

import numpy as np
import pytest
import torch

from paper_2103_01597_gb300 import ac, build, synthetic

pytestmark = pytest.mark.gpu

PHYS = dict(nu=5e-3, eta=5e-3, cs0=1.2, gamma=1.4, cp=1.1, lnrho0=0.1)
LARGE = (48, 40, 36)  # 69120 cells: the search starts from a guess on every 4th, 8th, 8th cell
SMALL = (20, 18, 16)


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    ac.load_library()
    torch.cuda.init()


def _state(n):
    return synthetic.smooth_state(n, seed=31, amp=0.3) + synthetic.noise_state(n, seed=32, sigma=1e-3)


def _sim(n, f, **kw):
    sim = ac.Simulation(n, **kw, **PHYS)
    sim.load(f)
    return sim


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("at", [(0, 0, 0), (8, 8, 8), (8, 8, 4), (32, 32, 44), (9, 8, 4)])
def test_nonfinite_cell_of_the_first_guess_is_reported(bad, at):
    """Cells (z, y, x) that the guess visits, and one beside them."""
    for q in (0, 2, 4, 6):
        f = _state(LARGE)
        f[q][at] = bad
        sim = _sim(LARGE, f)
        if q == 4 and bad == -math.inf:  # c_s = 0 there: a finite speed
            assert math.isfinite(sim.reduce(ac.AC_MAX, ac.AC_Q_CFL))
        else:
            with pytest.raises(ac.AcError) as ei:
                sim.reduce(ac.AC_MAX, ac.AC_Q_CFL)
            assert ei.value.code == ac.AC_ERR_NONFINITE, q
        sim.close()


CELLS = [(0, 0, 0), (1, 2, 3), (8, 8, 8), (9, 7, 5), (15, 17, 19)]


@pytest.mark.parametrize("n", [SMALL, LARGE])
@pytest.mark.parametrize("low", CELLS)
def test_speeds_beyond_binary32(n, low):
    """A speed of 1e40 at one cell, a larger one or an infinity at another."""
    for high in CELLS:
        if high == low:
            continue
        f = _state(n)
        f[1][low], f[2][high] = 1e40, 1e50
        sim = _sim(n, f)
        got = sim.reduce(ac.AC_MAX, ac.AC_Q_CFL)
        assert abs(got - 1e50) <= 1e-12 * 1e50, (high, got)
        f[2][high] = np.inf
        sim.load(f)
        with pytest.raises(ac.AcError) as ei:
            sim.reduce(ac.AC_MAX, ac.AC_Q_CFL)
        assert ei.value.code == ac.AC_ERR_NONFINITE, high
        sim.close()
