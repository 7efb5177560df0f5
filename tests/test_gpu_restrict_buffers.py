"""The restriction into buffers that other fields of the call use: fields go in order, so an
output may reuse an input that is done with, and two fields may share an output.
"""
import numpy as np
import pytest
import torch

from paper_2103_01597_gb300 import ac, build

pytestmark = pytest.mark.gpu

N = (96, 64, 48)


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    ac.load_library()
    torch.cuda.init()


def _restrict(fine, coarse, precision):
    ac.ac_restrict([t.data_ptr() for t in fine], precision, N, [t.data_ptr() for t in coarse],
                   torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("precision", [ac.AC_FP64, ac.AC_FP32])
@pytest.mark.parametrize("reuse", ["before", "after", "shared"])
def test_fields_go_in_order(precision, reuse):
    cells = N[0] * N[1] * N[2]
    dt = torch.float64 if precision == ac.AC_FP64 else torch.float32
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    fine = [torch.randn(cells, dtype=dt, device="cuda", generator=g) for _ in range(8)]
    own = [torch.empty(cells // 8, dtype=torch.float32, device="cuda") for _ in range(8)]
    _restrict(fine, own, precision)
    if reuse == "before":    # field 4's output over the input of field 3
        at, want = (4, fine[3]), {q: own[q] for q in range(8)}
    elif reuse == "after":   # field 1's output over the input of field 6: read as it then is
        at = (1, fine[6])
        changed = [t.clone() for t in fine]
        changed[6].view(torch.float32)[:cells // 8] = own[1]
        ref = [torch.empty_like(t) for t in own]
        _restrict(changed, ref, precision)
        want = {q: ref[q] for q in range(8) if q != 1}
    else:                    # fields 2 and 5 share an output: the later one stays
        at, want = None, {q: own[q] for q in range(8) if q != 2}
    out = [torch.empty_like(t) for t in own]
    if at:
        out[at[0]] = at[1].view(torch.float32)[:cells // 8]
    else:
        out[2] = out[5]
    _restrict(fine, out, precision)
    torch.cuda.synchronize()
    for q, w in want.items():
        assert np.array_equal(out[q].cpu().numpy(), w.cpu().numpy(), equal_nan=True), (reuse, q)
