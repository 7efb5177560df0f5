"""The tcgen05 convolutions where each CTA runs through several column segments: segments
of one tile and up, a last z-chunk shorter than the others, ragged x-tiles.

Against the mma.sync kernels on the same bfloat16 operands: 1e-2 relative in the max norm
for the forward pass (different accumulation order, so now and then another rounding of a
hidden activation: the bound of test_gpu_closure.py), and 4e-2 for the gradients (either
path lies within 2e-2 of the oracle at the kernels' rounding points).  Two calls give the
same bits: an output that depended on what a ring buffer or an accumulator held before
would not.
"""
import numpy as np
import pytest
import torch

from oracle import closure as oc
from paper_2103_01597_gb300 import ac, build, synthetic
from paper_2103_01597_gb300 import closure as cl

pytestmark = pytest.mark.gpu

SIZES = [27 * 8 * 32, 32, 27 * 32 * 32, 32, 27 * 32 * 8, 8]  # weights and biases of the layers


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    ac.load_library()


def _maxrel(g, o):
    return float((g - o).abs().max() / o.abs().max())


def _state(n, seed):
    x = synthetic.noise_state(n, seed, 0.5).astype(np.float32).reshape(8, -1)
    return torch.from_numpy(x).cuda()


# 400 to 1600 columns (times chunks) over at most 152 CTAs (304 in the last layer)
@pytest.mark.parametrize("n", [(9, 700, 1), (9, 700, 2), (130, 400, 3), (9, 700, 4), (9, 700, 7),
                               (257, 150, 10), (9, 500, 15), (9, 500, 16), (9, 500, 17),
                               (130, 200, 18), (9, 300, 35)])
def test_many_segments(n):
    params = oc.Net.init(3).flat().astype(np.float32)
    x, target = _state(n, 4), _state(n, 5)
    got = {}
    for path in (ac.AC_CONV_TCGEN05, ac.AC_CONV_MMA_SYNC):
        c = cl.Closure(n, params=params, conv_path=path)
        y = c.correction(x).clone()
        assert torch.equal(y, c.correction(x))
        c.loss(x, target)
        g = torch.from_numpy(ac.ac_closure_get_grads(c.c).astype(np.float64))
        c.status()
        c.close()
        got[path] = (y.double(), g)
    (y, g), (yo, go) = got[ac.AC_CONV_TCGEN05], got[ac.AC_CONV_MMA_SYNC]
    assert _maxrel(y, yo) <= 1e-2, _maxrel(y, yo)
    for t, to in zip(g.split(SIZES), go.split(SIZES)):
        assert _maxrel(t, to) <= 4e-2, (t.numel(), _maxrel(t, to))
