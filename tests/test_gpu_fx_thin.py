"""Thin boxes on the integer-sum path: columns over copies without a halo in place of padded
tiles.  Every substep from the GPU's own previous state against the FP64 oracle at 1e-12
relative per field in the max norm, the CFL speed at 1e-12 (the bounds the method is held
to; test_gpu_substep.py).  A derivative along an axis of one or two cells is zero exactly
in integers and the oracle's rounding noise otherwise: fields whose change is nothing but
that are compared with 1e-15 of the state.
"""
import numpy as np
import pytest
import torch

from oracle import core
from paper_2103_01597_gb300 import ac, build, synthetic

pytestmark = pytest.mark.gpu

PHYS = dict(nu=2e-2, eta=3e-2, cs0=1.1, gamma=1.4, cp=1.3, lnrho0=0.2)
H = 0.25
# shapes on the columns' side of the rule, ragged against their (32, 4) CTAs and z chunks
THIN = [(65, 1, 1), (100, 3, 60), (300, 2, 11), (2, 2, 20000), (1, 1, 3001), (130, 4, 66), (700, 5, 20)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    ac.load_library()
    torch.cuda.init()


def _state(n, seed=5):
    f = synthetic.smooth_state(n, seed, amp=0.2) + synthetic.noise_state(n, seed + 1, sigma=1e-3)
    f[0] += 0.1 * synthetic.uniform_state(n, seed + 2)[0]
    return f


def _sim(n, f, force_amp=0.05, **terms):
    sim = ac.Simulation(n, L=tuple(H * v for v in n), force_amp=force_amp, seed=3, **PHYS, **terms)
    sim.load(f)
    return sim


def _close(g, o, f):
    for q in range(8):
        err = np.max(np.abs(g[q] - o[q]))
        assert err <= max(1e-12 * np.max(np.abs(o[q])), 1e-15 * np.max(np.abs(f))), (q, err)


def _parity(n, f, **terms):
    sim = _sim(n, f, **terms)
    p = core.Params(n=n, L=tuple(H * v for v in n), forcing=core.forcing_draw(3, 0, 0.05), **PHYS,
                    **terms)
    w = None
    for s in range(3):
        fo, wo = core.substep(f, w, p, 1e-3, s)
        cfl = core.reduce(f, p, "max", "cfl")
        sim.substep(1e-3, s)
        if s == 0:
            assert abs(ac.ac_last_cfl(sim.h) - cfl) <= 1e-12 * cfl
        fg, wg = sim.store(), sim.store_w()
        _close(fg, fo, f)
        _close(wg, wo, f)
        f, w = fg, wg
    modes = ac.ac_get_stencil_modes(sim.h)
    sim.close()
    return modes


@pytest.mark.parametrize("n", THIN)
@pytest.mark.parametrize("entropy", [False, True])
def test_thin_boxes(n, entropy):
    terms = dict(K=1e-2, zeta=2e-2, heat=0.02, cool=0.01) if entropy else {}
    f = _state(n)
    for q in (1, 2, 3, 5, 6, 7):  # equal ranges: one scale a group
        f[q] *= 0.11 / np.max(np.abs(f[q]))
        f[q].flat[0], f[q].flat[-1] = 0.12, -0.12
    assert _parity(n, f, **terms)[ac.AC_STENCIL_MODE_GROUP] >= 1


@pytest.mark.parametrize("n", [(100, 3, 60), (2, 2, 20000)])
@pytest.mark.parametrize("entropy", [False, True])
def test_scales_of_their_own(n, entropy):
    """A component of u and one of A far below the others, and a mean flow."""
    terms = dict(K=1e-2, zeta=2e-2, heat=0.02, cool=0.01) if entropy else {}
    f = _state(n)
    f[3] *= 1e-4
    f[5] *= 1e-5
    f[1] += 30.0
    assert _parity(n, f, **terms) == (0, 3, 0)


@pytest.mark.parametrize("n", [(100, 3, 60), (65, 1, 1)])
def test_nan_takes_plain_stencils(n):
    f = _state(n)
    f[2].flat[7] = np.nan
    out = []
    for mode in (ac.AC_STENCIL_AUTO, ac.AC_STENCIL_FP64):
        sim = _sim(n, f)
        ac.ac_set_stencil_mode(sim.h, mode)
        sim.step(1e-3)
        out.append((sim.store(), sim.store_w()))
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)


def test_copies_of_a_thin_box_are_not_padded():
    """64 bytes a cell, where a halo would take 49 times as much."""
    n = (1, 1, 1000000)
    sim = ac.Simulation(n, L=tuple(H * v for v in n))
    sim.store()
    before = torch.cuda.mem_get_info()[0]
    sim.substep(1e-3, 0)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    sim.close()
    assert used <= 64 * n[2] + (64 << 20), used
