"""Reductions and the restriction where their integer forms can go wrong: edges of their
tiles, spacings, values beyond the exponents the integers hold, zeros, non-finite cells.

Reductions: 1e-12 relative to the oracle (sums: to the sum of magnitudes), the bound of
test_gpu_substep.py.  Restriction: every cell within one binary32 unit (2^-23) of the
oracle's binary64 value: a rounding to binary32 is half of that, the integer sum at most
2^-30 of the result.
"""
import math

import numpy as np
import pytest
import torch

from oracle import core
from paper_2103_01597_gb300 import ac, build, synthetic

pytestmark = pytest.mark.gpu

PHYS = dict(nu=5e-3, eta=5e-3, cs0=1.2, gamma=1.4, cp=1.1, lnrho0=0.1)
DERIVED = {ac.AC_Q_UMAG: "umag", ac.AC_Q_EKIN: "ekin", ac.AC_Q_EMAG: "emag", ac.AC_Q_CFL: "cfl"}
OPS = {ac.AC_MAX: "max", ac.AC_MIN: "min", ac.AC_SUM: "sum", ac.AC_RMS: "rms"}


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    ac.load_library()
    torch.cuda.init()


def _state(n):
    f = synthetic.smooth_state(n, seed=31, amp=0.3) + synthetic.noise_state(n, seed=32, sigma=1e-3)
    f[0] += 0.05
    return f


def _check(n, L, f, layout=ac.AC_LAYOUT_PERIODIC):
    sim = ac.Simulation(n, L=L, layout=layout, **PHYS)
    p = core.Params(n=n, L=L, **PHYS)
    sim.load(f)
    for q in [0, 4, 6] + list(DERIVED):
        o_all = core.quantity(f, p, DERIVED.get(q, q))
        for op, name in OPS.items():
            g = sim.reduce(op, q)
            o = core.reduce(f, p, name, DERIVED.get(q, q))
            scale = np.sum(np.abs(o_all)) if name == "sum" else abs(o)
            assert abs(g - o) <= 1e-12 * max(scale, 1e-300), (q, name, g, o)
    sim.close()


@pytest.mark.parametrize("n", [(1, 3, 2), (33, 9, 17), (31, 8, 16), (48, 40, 36)])
@pytest.mark.parametrize("layout", [ac.AC_LAYOUT_PERIODIC, ac.AC_LAYOUT_PADDED])
def test_reductions_at_tile_edges(n, layout):
    _check(n, (2 * math.pi, 3.0, 4.5), _state(n), layout)


@pytest.mark.parametrize("case", ["far_spacings", "tiny_a", "huge_a", "mixed_a", "thin_gas"])
def test_reductions_beyond_the_integers(case):
    """Spacings more than 8 apart, |A| outside 2^+-200 or spread over 2^100, |ln rho|
    beyond 64: the general arithmetic, or alignment that drops what binary64 drops."""
    n, L = (20, 12, 10), (2.0, 3.0, 4.0)
    f = _state(n)
    if case == "far_spacings":
        L = (2.0, 30.0, 4.0)
    elif case == "tiny_a":
        f[5:8] *= 1e-80
    elif case == "huge_a":
        f[5:8] *= 1e70
    elif case == "mixed_a":
        f[5:8, :5] *= 2.0 ** -100
    else:
        f[0] += 70.0
    _check(n, L, f)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_nonfinite_cell_is_reported(bad):
    n = (48, 40, 36)
    for q in (0, 2, 6):
        f = _state(n)
        f[q][7, 8, 9] = bad
        sim = ac.Simulation(n, **PHYS)
        sim.load(f)
        for op in OPS:
            for quantity in (q, ac.AC_Q_CFL):
                with pytest.raises(ac.AcError) as ei:
                    sim.reduce(op, quantity)
                assert ei.value.code == ac.AC_ERR_NONFINITE, (q, op, quantity)
            assert math.isfinite(sim.reduce(op, 4))  # another field: unaffected
        sim.close()


@pytest.mark.parametrize("n", [(2, 2, 2), (66, 18, 34), (64, 16, 70), (130, 6, 4)])
@pytest.mark.parametrize("precision", [ac.AC_FP64, ac.AC_FP32])
@pytest.mark.parametrize("shift", [0, 1])
def test_restriction_cells(n, precision, shift):
    """`shift` elements past the allocation's start: rows off the pair-load boundary.  The
    fields cover zeros, a spread over 2^60 within a row, subnormals and a NaN."""
    dt = torch.float64 if precision == ac.AC_FP64 else torch.float32
    f = _state(n) * np.array([1, 1e3, 1e-30, 1, 1, 1, 1, 1]).reshape(8, 1, 1, 1)
    f[3] = 0.0
    f[4][:, :, ::2] *= 2.0 ** -60
    f[5] *= 1e-310 if precision == ac.AC_FP64 else 1e-40
    f[6][0, 0, 0] = np.nan
    f[7][:, : n[1] // 2] = 0.0
    size = n[0] * n[1] * n[2]
    buf = torch.zeros(8, size + shift + 4, dtype=dt, device="cuda")
    buf[:, shift:shift + size] = torch.from_numpy(f.reshape(8, -1)).to(dt)
    f = buf[:, shift:shift + size].double().cpu().numpy().reshape(f.shape)
    out = torch.full((8, size // 8), 7.0, dtype=torch.float32, device="cuda")
    ac.ac_restrict([buf[q, shift:].data_ptr() for q in range(8)], precision, n,
                   [out[q].data_ptr() for q in range(8)], torch.cuda.current_stream().cuda_stream)
    got = out.double().cpu().numpy().reshape(8, n[2] // 2, n[1] // 2, n[0] // 2)
    for q in range(8):
        o = core.restrict(f[q])
        assert np.array_equal(np.isnan(got[q]), np.isnan(o)), q
        ok = ~np.isnan(o)
        # (subnormal binary32 results: half their spacing)
        tol = np.maximum(2.0 ** -23 * np.abs(o[ok]), 2.0 ** -149)
        assert np.all(np.abs(got[q][ok] - o[ok]) <= tol), (q, np.max(np.abs(got[q][ok] - o[ok]) / tol))
