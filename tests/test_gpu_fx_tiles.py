"""The tiled integer-product substep (binary64) where it can go wrong:
grids against the edges of its 16 x 16 tiles and of its z march, states against the
edges of the ranges its fixed point is sized for.  Each substep runs from the GPU's
own previous state and is compared with the FP64 oracle at 1e-12 relative per field
in the max norm (the bound the method is held to; test_gpu_substep.py); the CFL
speed at 1e-12 relative.
"""
import math

import numpy as np
import pytest
import torch

from oracle import core
from paper_2103_01597_gb300 import ac, build, synthetic

from gpu_util import rel_err

pytestmark = pytest.mark.gpu

PHYS = dict(nu=2e-2, eta=3e-2, cs0=1.1, gamma=1.4, cp=1.3, lnrho0=0.2)


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    ac.load_library()
    torch.cuda.init()


def _state(n, seed, amp=0.2):
    f = synthetic.smooth_state(n, seed, amp=amp) + synthetic.noise_state(n, seed + 1, sigma=1e-3)
    f[0] += 0.1 * synthetic.uniform_state(n, seed + 2)[0]
    return f


def _parity(n, f, force_amp=0.05, phys=PHYS, **terms):
    L = tuple(0.25 * v for v in n)  # spacing 1/4 on every axis, exactly
    sim = ac.Simulation(n, L=L, force_amp=force_amp, seed=3, **phys, **terms)
    assert ac.ac_get_stencil_path(sim.h)
    p = core.Params(n=n, L=L, forcing=core.forcing_draw(3, 0, force_amp), **phys, **terms)
    sim.load(f)
    w = None
    for s in range(3):
        fo, wo = core.substep(f, w, p, 1e-3, s)
        if s == 0:
            cfl = core.reduce(f, p, "max", "cfl")
        sim.substep(1e-3, s)
        if s == 0:
            assert abs(ac.ac_last_cfl(sim.h) - cfl) <= 1e-12 * cfl
        fg, wg = sim.store(), sim.store_w()
        assert np.all(rel_err(fg, fo) <= 1e-12), (s, rel_err(fg, fo))
        assert np.all(rel_err(wg, wo) <= 1e-12), (s, rel_err(wg, wo))
        f, w = fg, wg
    modes = ac.ac_get_stencil_modes(sim.h)
    sim.close()
    return modes


def test_one_cell():
    """On a single cell every derivative vanishes (the oracle's binary64 sums of a
    constant leave rounding noise there, the integer sums exactly zero): ln rho, s and A
    stay as they are, bit for bit, and u gains dt times the forcing."""
    n, L = (1, 1, 1), (0.25,) * 3
    f = _state(n, 5)
    sim = ac.Simulation(n, L=L, force_amp=0.05, seed=3, **PHYS)
    sim.load(f)
    sim.substep(1e-3, 0)
    fg, wg = sim.store(), sim.store_w()
    sim.close()
    frc = core.forcing_draw(3, 0, 0.05)
    want = 1e-3 * 0.05 * np.array(frc.e) * math.cos(frc.phi)
    for q in (0, 4, 5, 6, 7):
        assert np.all(wg[q] == 0.0) and np.array_equal(fg[q], f[q]), q
    assert np.max(np.abs(wg[1:4].ravel() - want)) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("n", [(2, 1, 5), (15, 16, 17), (16, 16, 1), (17, 33, 2),
                               (31, 5, 40), (48, 16, 9)])
@pytest.mark.parametrize("entropy", [False, True])
def test_tile_edges(n, entropy):
    terms = dict(K=1e-2, zeta=2e-2, heat=0.02, cool=0.01) if entropy else {}
    assert sum(_parity(n, _state(n, 5), **terms)) == 3


N = (20, 18, 12)


@pytest.mark.parametrize("binades", [2, 6, 7])
def test_component_disparity(binades):
    """u_z and A_x smaller than their groups' largest by 2^binades: the group scale
    serves six, a seventh goes to per-field scales."""
    f = _state(N, 11)
    f[3] *= 2.0 ** -binades * np.max(np.abs(f[1])) / np.max(np.abs(f[3]))
    f[5] *= 2.0 ** -binades * np.max(np.abs(f[7])) / np.max(np.abs(f[5]))
    _parity(N, f, force_amp=0.0)


@pytest.mark.parametrize("flow", [0.0, 1.0, 15.0, 17.0, 100.0])
def test_mean_flow(flow):
    """A uniform flow added to fluctuations of range about 1: u is taken from F + C up to
    2^4 times its range, beyond that the per-field kernel runs."""
    f = _state(N, 21)
    f[1] += flow
    _parity(N, f, force_amp=0.0)


@pytest.mark.parametrize("ls,cp", [(1e-6, 1.0), (1.0, 1e-3), (1e6, 1.0), (1.0, 1e3), (0.0, 0.7)])
def test_pressure_scales(ls, cp):
    """ln rho's range over that of s / c_p: the ratio of the two scales in
    grad(ln rho + s / c_p), either way, and a constant ln rho."""
    f = _state(N, 31, amp=1e-3)
    f[0] = f[0] * min(ls, 1.0)
    f[4] = f[4] / max(ls, 1.0) * min(cp, 1.0)
    _parity(N, f, phys=dict(PHYS, cp=cp))


@pytest.mark.parametrize("lnrho,ss", [(40.0, -20.0), (-63.0, 10.0), (64.5, -30.0), (3.0, 60.0)])
def test_thermodynamic_range(lnrho, ss):
    """|ln rho| and |xi| up to 64 take the fixed-point exp, beyond that the per-field
    kernel (weak fields: the Lorentz force and the heating carry 1 / rho)."""
    f = _state(N, 41)
    f[5:8] *= math.exp(0.5 * min(lnrho, 0.0))
    f[0] += lnrho
    f[4] += ss
    _parity(N, f, phys=dict(PHYS, cs0=math.exp(-0.5 * (1.4 * ss / 1.3 + 0.4 * lnrho))))


# unequal spacings on grids large enough for the integer form (16384 cells), ragged
# against the tiles; the ratios of the spacings up to 8, either way
UNEQUAL = [((33, 32, 17), (1.0, 1.5, 0.7)), ((17, 31, 33), (8.0, 1.0, 1.0)),
           ((16, 1, 1100), (1.0, 3.0, 2.0)), ((26, 26, 26), (1.0, 1.0, 8.0)),
           ((48, 40, 9), (1.0, 1.0 + 2.0 ** -50, 1.0))]


def _unequal(n, hs, f, mode, **terms):
    L = tuple(0.25 * h * v for v, h in zip(n, hs))
    sim = ac.Simulation(n, L=L, force_amp=0.05, seed=3, **PHYS, **terms)
    ac.ac_set_stencil_mode(sim.h, mode)
    sim.load(f)
    out = []
    for s in range(3):
        sim.substep(1e-3, s)
        out.append((sim.store(), sim.store_w()))
    cfl = ac.ac_last_cfl(sim.h)
    sim.close()
    return L, out, cfl


@pytest.mark.parametrize("n,hs", UNEQUAL)
@pytest.mark.parametrize("entropy", [False, True])
def test_unequal_spacing(n, hs, entropy):
    """The default path scales each axis's integer numerators; every substep against the
    oracle from the path's own previous state, and not the plain stencils' bits."""
    terms = dict(K=1e-2, zeta=2e-2, heat=0.02, cool=0.01) if entropy else {}
    f = _state(n, 51)
    L, out, cfl = _unequal(n, hs, f, ac.AC_STENCIL_AUTO, **terms)
    p = core.Params(n=n, L=L, forcing=core.forcing_draw(3, 0, 0.05), **PHYS, **terms)
    c = core.reduce(f, p, "max", "cfl")
    assert abs(cfl - c) <= 1e-12 * c
    w = None
    for s, (fg, wg) in enumerate(out):
        fo, wo = core.substep(f, w, p, 1e-3, s)
        assert np.all(rel_err(fg, fo) <= 1e-12), (s, rel_err(fg, fo))
        assert np.all(rel_err(wg, wo) <= 1e-12), (s, rel_err(wg, wo))
        f, w = fg, wg
    _, plain, _ = _unequal(n, hs, _state(n, 51), ac.AC_STENCIL_FP64, **terms)
    assert not np.array_equal(plain[-1][1], out[-1][1])


@pytest.mark.parametrize("case", ["small", "ratio", "range", "nan"])
def test_unequal_spacing_left_to_the_plain_stencils(case):
    """Few cells, spacings more than 8 apart, a state outside the ranges the fixed point
    is sized for, a NaN: bit for bit what AC_STENCIL_FP64 computes."""
    n, hs = ((15, 16, 17), (1.0, 1.5, 1.0)) if case == "small" else ((26, 26, 26), (1.0, 1.5, 1.0))
    if case == "ratio":
        hs = (1.0, 9.0, 1.0)
    f = _state(n, 61)
    if case == "range":
        f[3] *= 1e-4
    if case == "nan":
        f[2][3, 4, 5] = np.nan
    L, out, plain = None, [], []
    for mode, dst in ((ac.AC_STENCIL_AUTO, out), (ac.AC_STENCIL_FP64, plain)):
        L = tuple(0.25 * h * v for v, h in zip(n, hs))
        sim = ac.Simulation(n, L=L, force_amp=0.05, seed=3, **PHYS)
        ac.ac_set_stencil_mode(sim.h, mode)
        sim.load(f)
        sim.step(1e-3)
        dst += [sim.store(), sim.store_w()]
        sim.close()
    for a, b in zip(out, plain):
        assert np.array_equal(a, b, equal_nan=True)


def test_small_laplacians():
    """One cell sets the scale and the rest of u and A lies 2^33 below it, so that the
    Laplacians' 96-bit numerators there stay below 2^32 units: taken for zero they would
    be 8e-11 of the largest off."""
    n = (21, 18, 20)
    f = np.zeros((8,) + n[::-1])
    noise = synthetic.noise_state(n, 9, sigma=3.5e-11)
    for q in (1, 2, 3, 5, 6, 7):
        f[q] = noise[q]
        f[q][7, 5, 11] = 0.3 if q % 2 else -0.2
    _parity(n, f, force_amp=0.0)
