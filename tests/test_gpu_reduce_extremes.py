"""The binary64 reductions that search or align: the largest CFL speed where a cell of the
first guess is not finite and where speeds leave binary32's range, and E_M where a part
of A is uniform or one component is far smaller than another.

CFL speeds: 1e-12 relative to the oracle, the bound of test_gpu_substep.py.  E_M: 1e-14
relative to the same stencils in extended precision on the stored values (a cell's |B|^2
carries some eight roundings, its sum over the cells some forty).
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


def _b2(A, h):
    """|curl A|^2 in extended precision, sixth order."""
    A = A.astype(np.longdouble)

    def d1(f, a):
        ax = 2 - a
        s = sum(w * (np.roll(f, -m, ax) - np.roll(f, m, ax)) for m, w in ((1, 45), (2, -9), (3, 1)))
        return s / (60 * np.longdouble(h[a]))

    B = [d1(A[2], 1) - d1(A[1], 2), d1(A[0], 2) - d1(A[2], 0), d1(A[1], 0) - d1(A[0], 1)]
    return B[0] ** 2 + B[1] ** 2 + B[2] ** 2


@pytest.mark.parametrize("offset,amps", [((0, 0, 0), (1, 1, 1)), ((0, 0, 1e4), (1, 1, 1)),
                                         ((0, 0, 1e6), (1, 1, 1)), ((1, 1, 1), (1e-8, 1e-8, 1e-8)),
                                         ((1, 0, 0), (0, 1e-4, 1e-4)), ((1, 0, 0), (0, 1e-8, 1e-8)),
                                         ((0, 0, 0), (1, 1e-8, 1e-8)), ((3, 0, 0), (0, 0, 1e-10))])
@pytest.mark.parametrize("L", [(2 * math.pi,) * 3, (2 * math.pi, 3.0, 11.0), (2.0, 40.0, 3.0)])
def test_magnetic_energy_with_uniform_parts(offset, amps, L):
    """A_x varies along x only where it is the large one, so that it adds nothing to B."""
    n = (32, 30, 28)
    f = np.zeros((8,) + n[::-1])
    z, y, x = np.meshgrid(*[np.arange(m) * 2 * np.pi / m for m in n[::-1]], indexing="ij")
    waves = (np.cos(x + 0.3) if amps[1] < amps[0] else np.sin(y - 2 * z + 0.4) + 0.5 * np.cos(z + 1.0),
             np.sin(z + 2 * x + 0.1) + 0.3 * np.cos(x - 1.2), np.cos(x - y + 0.7) + 0.4 * np.sin(2 * y))
    for q in range(3):
        f[5 + q] = offset[q] + amps[q] * waves[q]
    want = float(0.5 * np.sum(_b2(f[5:8], [L[a] / n[a] for a in range(3)])))
    sim = _sim(n, f, L=L)
    got = sim.reduce(ac.AC_SUM, ac.AC_Q_EMAG)
    sim.close()
    assert want > 0 and abs(got - want) <= 1e-14 * want, (got, want, abs(got - want) / want)
