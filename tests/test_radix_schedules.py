"""Radix schedules of the mixed-radix passes (host side, by the rule of
make_axis): every supported length has one, every radix that the kernels are
compiled for is chosen by some length, and the GPU tests run all of them."""
import os
import re

from test_gpu_mixed_radix import LENGTHS
from test_gpu_radix_lengths import MORE_LENGTHS

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2106_12487_gb300", "csrc")
SHORT = [5, 3, 7]            # the other axes of the GPU tests' grids


def text(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def lists():
    s = text("bloch_ops.cu")
    return [[int(v) for v in re.search(name + r"\[\] = \{([^}]*)\}", s).group(1).split(",")] for name in ("ends", "mids")]


def schedule(N, ff):
    """Fewest stages, then the smallest sum; the first radix no larger than the last."""
    ends, mids = lists()
    best = None
    for r1 in ends:
        for r2 in mids:
            for r3 in ends:
                if r1 * r2 * r3 != N or (r1 > r3 and r3 > 1):
                    continue
                if (r1 in (12, 14) or r3 in (12, 14)) if ff else r2 == 4:
                    continue
                cost = (1000 if r2 > 1 else 0) + r1 + r2 + r3
                if best is None or cost < best[0]:
                    best = (cost, r1, r2, r3)
    return best[1:]


def supported():
    out = []
    for n in range(1, 513):
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def used(lengths, ff):
    s = [schedule(n, ff) for n in lengths]
    return [{v[i] for v in s} for i in range(3)]


def test_every_compiled_radix_is_chosen():
    """The kernels hold no radix that no length reaches."""
    s = text("passes.cuh")
    body = s[s.index("void with_mid_radix"):]
    body = body[:body.index("using real_t")]
    common, ff_only = body.split("if constexpr")
    mids = {int(v) for v in re.findall(r"BLOCH_RADIX\((\d+)\)", common)}
    extra = {int(v) for v in re.findall(r"BLOCH_RADIX\((\d+)\)", ff_only)}
    assert used(supported(), False)[1] == mids | {1}
    assert used(supported(), True)[1] == mids | extra | {1}
    ends, _ = lists()
    assert set(ends) == used(supported(), False)[0] | used(supported(), False)[2]


def test_gpu_lengths_cover_every_radix():
    for ff in (False, True):
        tested = used(LENGTHS + MORE_LENGTHS + SHORT, ff)
        for stage, want in zip(tested, used(supported(), ff)):
            assert stage == want, (ff, sorted(want - stage))
