"""The restriction's integer sums where a warp's scale is set by another cell: each result
is the binary32 rounding of the exact weighted sum, or that of the binary64 sum where the
exact one is too near a midpoint to tell.
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


def _sums(f):
    """Exact weighted sums of one field as integers in units of 2^-200, and in binary64."""
    exact = np.vectorize(lambda v: int(v * 2.0 ** 140) << 56, otypes=[object])(f * 2.0 ** 4)
    out = []
    for a in (exact, f):
        for ax in range(3):
            a = 2 * a + np.roll(a, 1, ax) + np.roll(a, -1, ax)
        out.append(a[::2, ::2, ::2])
    return out[0], (out[1] / 64).astype(np.float32)


def _float32(s):
    """Round-to-nearest-even binary32 of s 2^-206."""
    m = abs(s)
    if m == 0:
        return np.float32(0)
    k = max(m.bit_length() - 24, 0)
    q, r = m >> k, m & ((1 << k) - 1)
    q += (2 * r > 1 << k) or (2 * r == 1 << k and q & 1) if k else 0
    return np.float32(np.ldexp(float(q if s > 0 else -q), k - 206))


@pytest.mark.parametrize("binades", [0, 10, 20, 25, 30, 60])
def test_rounding_of_small_cells_beside_large_ones(binades):
    n = (64, 32, 12)
    f = np.random.Generator(np.random.PCG64(5)).standard_normal((8,) + n[::-1])
    f[:, :, :, 6:] *= 2.0 ** -binades  # one warp's columns: three large, the rest small
    dev = torch.from_numpy(f.reshape(8, -1)).cuda()
    size = n[0] * n[1] * n[2]
    out = torch.empty((8, size // 8), dtype=torch.float32, device="cuda")
    ac.ac_restrict([dev[q].data_ptr() for q in range(8)], ac.AC_FP64, n,
                   [out[q].data_ptr() for q in range(8)], torch.cuda.current_stream().cuda_stream)
    got = out.cpu().numpy().reshape(8, n[2] // 2, n[1] // 2, n[0] // 2)
    for q in range(8):
        exact, plain = _sums(f[q])
        want = np.vectorize(_float32, otypes=[np.float32])(exact)
        off = (got[q] != want) & (got[q] != plain)
        assert not np.any(off), (q, int(np.sum(off)), got[q][off][:3], want[off][:3])
