"""Terms of the binary64 substep whose operands have scales far apart: the pressure
gradient where ln rho and s vary along different axes, and advection by a uniform
velocity component far below the others' range.  One substep at 1e-12 relative per field
in the max norm against the FP64 oracle (the bound the method is held to;
test_gpu_substep.py): here only the small operand reaches the component that is looked at.
"""
import numpy as np
import pytest
import torch

from oracle import core
from paper_2103_01597_gb300 import ac, build

from gpu_util import rel_err

pytestmark = pytest.mark.gpu

PHYS = dict(nu=2e-2, eta=3e-2, cs0=1.1, gamma=1.4, lnrho0=0.2)
N = (24, 20, 18)


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    ac.load_library()
    torch.cuda.init()


def _axes(n):
    z, y, x = np.meshgrid(*[np.arange(m) * 2 * np.pi / m for m in n[::-1]], indexing="ij")
    return x, y, z


def _w(n, f, hs=(1.0, 1.0, 1.0), cp=1.3, **terms):
    L = tuple(0.25 * h * v for v, h in zip(n, hs))
    sim = ac.Simulation(n, L=L, cp=cp, **PHYS, **terms)
    sim.load(f)
    sim.substep(1e-3, 0)
    wg = sim.store_w()
    sim.close()
    _, wo = core.substep(f, None, core.Params(n=n, L=L, cp=cp, **PHYS, **terms), 1e-3, 0)
    return rel_err(wg, wo), wo


@pytest.mark.parametrize("eps", [1.0, 1e-2, 1e-5, 1e-8, 1e-10])
@pytest.mark.parametrize("small", [0, 4])
@pytest.mark.parametrize("n,hs", [(N, (1.0, 1.0, 1.0)), ((26, 28, 25), (1.0, 1.5, 0.75))])
@pytest.mark.parametrize("entropy", [False, True])
def test_pressure_of_fields_on_different_axes(eps, small, n, hs, entropy):
    """At rest: u_x feels the one, u_y only the small other."""
    terms = dict(K=1e-2, zeta=2e-2, heat=0.02, cool=0.01) if entropy else {}
    f = np.zeros((8,) + n[::-1])
    x, y, _ = _axes(n)
    f[4 - small], f[small] = np.sin(x), eps * np.sin(y + 0.2)
    err, wo = _w(n, f, hs, **terms)
    assert np.max(np.abs(wo[2])) > 1e-6 * eps * 1e-3
    assert np.all(err[1:3] <= 1e-12), err


@pytest.mark.parametrize("uz", [0.3, 1e-2, 1e-5, 1e-6, 1e-8])
@pytest.mark.parametrize("n,hs", [(N, (1.0, 1.0, 1.0)), ((26, 28, 25), (1.0, 1.5, 0.75))])
def test_advection_by_a_small_uniform_component(uz, n, hs):
    """u = (sin y, sin x, u_z): divergence-free, and only u_z meets the gradients of
    ln rho(z) and (s being at its reference) A(z)."""
    f = np.zeros((8,) + n[::-1])
    x, y, z = _axes(n)
    f[0] = 0.3 * np.sin(z + 0.1)
    f[1], f[2], f[3] = np.sin(y), np.sin(x), uz
    err, wo = _w(n, f, hs)
    assert np.max(np.abs(wo[0])) > 1e-2 * uz * 1e-3
    assert err[0] <= 1e-12, err


@pytest.mark.parametrize("u", [(1.0, 1e-8, 0.0), (1e-9, 0.0, 2.0), (1e-3, 1e-3, 1e-3)])
def test_advection_by_a_uniform_flow(u):
    """Every component constant: ln rho varies along the axis of the smallest."""
    f = np.zeros((8,) + N[::-1])
    axes = _axes(N)
    small = min((abs(v), a) for a, v in enumerate(u) if v)[1]
    f[0] = 0.3 * np.sin(axes[small] + 0.1)
    for a in range(3):
        f[1 + a] = u[a]
    err, _ = _w(N, f)
    assert err[0] <= 1e-12, err
