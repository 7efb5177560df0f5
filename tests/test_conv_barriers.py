"""The barrier protocol of the one-CTA tcgen05 convolution, run as a model on the host.

The roles of conv_tc_kernel (two producers that take ring groups in turn, the MMA warp,
two sets of epilogue warps) are stepped against mbarriers that know only the parity of
their current phase.  Each role in turn is held back at each of its steps until no other
role can move, which is the worst that a scheduler may do; the CTA has to get through
its segments all the same.  A phase that completes before every waiter of the one before
has seen it leaves that waiter with a parity that looks like the phase after: it would
wait until its bound ran out.

The arrival counts and constants are read from the kernel's source.
"""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2103_01597_gb300", "csrc", "conv_tc.cuh")


def _constants():
    s = open(SRC).read()
    c = {k: int(v) for k, v in re.findall(r"constexpr int (GROUP|ESETS|PRODS|RBLK) = (\d+);", s)}
    body = s[s.index("conv_tc_kernel(const __grid_constant__"):]
    body = body[:body.index("// ---- paired CTAs")]
    count = eval(re.search(r"mbar_init\(&acce\[b\], ([^)]*)\)", body).group(1), {}, dict(c))
    producers = body[body.index("TMA producers"):body.index("MMA issuer")]
    return c, count, "mbar_arrive(&acce[" in producers


class Bar:
    def __init__(self, count):
        self.count = self.left = count
        self.phase = 0

    def arrive(self, n=1):
        assert self.left >= n, "an arrival of the next phase came early"
        self.left -= n
        if self.left == 0:
            self.phase += 1
            self.left = self.count

    def done(self, parity):
        return (self.phase & 1) != parity


def _roles(lens, ngrp):
    """Generators that yield (barrier, parity) to wait for; each resumes once it is done."""
    c, count, arrives = _constants()
    group, esets, prods, rblk = c["GROUP"], c["ESETS"], c["PRODS"], c["RBLK"]
    full, empty = [Bar(1) for _ in range(ngrp)], [Bar(1) for _ in range(ngrp)]
    accf = [Bar(1) for _ in range(rblk)]
    acce = [Bar(count) for _ in range((rblk + group - 1) // group)]

    def producer(own):
        grp = rnd = 0
        gpar = [0] * len(acce)
        for n in lens:
            for k, j in enumerate(range(0, n + 2, group)):
                if j < n:
                    yield acce[k], gpar[k] ^ 1
                    if arrives:
                        acce[k].arrive()
                if grp % prods == own:
                    if rnd:
                        yield empty[grp], (rnd - 1) & 1
                    full[grp].arrive()
                if j < n:
                    gpar[k] ^= 1
                grp += 1
                if grp == ngrp:
                    grp, rnd = 0, rnd + 1

    def mma():
        grp = fill = 0
        for n in lens:
            for j in range(0, n + 2, group):
                yield full[grp], fill
                for q in range(j, min(j + group, n + 2)):
                    if q >= 2:
                        accf[q - 2].arrive()
                empty[grp].arrive()
                grp += 1
                if grp == ngrp:
                    grp, fill = 0, fill ^ 1

    def epilogue(own):
        par = [0] * rblk
        for n in lens:
            for i in range(own, n, esets):
                yield accf[i], par[i]
                par[i] ^= 1
                acce[i // group].arrive(group - i % group if i == n - 1 else 1)

    return ([producer(p) for p in range(prods)] + [mma()] +
            [epilogue(e) for e in range(esets) for _ in range(4)])


def _run(lens, ngrp, held, at):
    """Step every role as far as it gets, `held` only when nothing else moves once it has
    taken `at` steps; the roles that did not finish."""
    roles = _roles(lens, ngrp)
    waits = [next(r, None) for r in roles]
    taken = 0
    while any(w is not None for w in waits):
        moved = False
        for r, w in enumerate(waits):
            if w is None or not w[0].done(w[1]) or (r == held and taken >= at):
                continue
            waits[r] = next(roles[r], None)
            taken += r == held
            moved = True
        if not moved:
            w = waits[held]
            if w is None or not w[0].done(w[1]):
                return [r for r, x in enumerate(waits) if x is not None]
            waits[held] = next(roles[held], None)
            at = 1 << 30  # let go
    return []


@pytest.mark.parametrize("ngrp", [2, 4])
@pytest.mark.parametrize("lens", [[1] * 9, [2] * 8, [4] * 8, [16] * 5, [7, 7, 7, 1, 7, 1],
                                  [13, 4, 13, 4, 13], list(range(1, 17))])
def test_no_role_is_left_waiting(lens, ngrp):
    steps = 4 * sum(n + 2 for n in lens)
    for held in (0, 1, 2, 3, 7):
        for at in range(steps):
            left = _run(lens, ngrp, held, at)
            assert not left, (held, at, left)
